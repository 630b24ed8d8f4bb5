"""Writes qs_op_loop.inc: the op loop of the wide fused pass (complex64, 64
amplitudes, 6 register bits per thread) as inline PTX with one indexed branch
per op.

A thread's amplitudes are 32 units of two (16 in the five-bit loops of small
states, which know no code of register bit 5): the amplitudes that differ in
register bit 0 (always tile bit 0, qubit 0).  A unit is two 64-bit registers,
the two real parts and the two imaginary parts, so every gate on register
bits 1..5 is packed FP32x2 arithmetic throughout -- with (re, im) in one
register X^1/2 and T mix the halves and take twice the instructions.  Gates
on register bit 0 work on the halves with scalar instructions.

Every op is one byte code (the host lowers a plan to them, lower_wide in
qs_host.cpp) and a 16-byte record: the selection outside the register set
(8 bytes, tested as (idx & sel) == sel) and two FP32 parameters.

    W_H  + j   H on register bit j (the 1/sqrt2 deferred to the pass end)
    W_XH + j   X^1/2 on register bit j (deferred)
    W_YH + j   Y^1/2 on register bit j (deferred)
    W_T  + j   T phase on the amplitudes with bit j set
    W_CZ + p   sign on the amplitudes with both bits of pair p set
    W_CZO + j  sign on the amplitudes with bit j set where the selection holds
               (an empty selection always holds: Z)
  and, in the loop of passes with parameterised gates (FULL):
    W_RY + j   R_Y on register bit j as three shears x += a y, y += b x,
               x += a y with (a, b) = (-tan(phi/2), sin(phi)), phi = theta/2
    W_RX + j   R_X on register bit j: the same shears between x and i y
    W_PH + j   amplitudes with bit j set times a + i b where the selection holds
    W_PP + p   amplitudes with both bits of pair p set times a + i b
  and, in the loop of the adjoint sweep (ADJ), where register bit 5 selects
  psi (0) or lambda (1), so that every gate runs on both, the derivative terms
  of a thread, sums over its amplitudes:
    W_DX + j   Im <lambda| X_j |psi>          W_DY + j   Im <lambda| Y_j |psi>
    W_DZ + j   Im <lambda| Z_j |psi>
    W_DP + j   Im <lambda| psi> over the amplitudes with bit j set where the
               selection holds, else 0
    W_DPP + p  the same over the amplitudes with both bits of pair p set
    W_DW       w = Im <lambda| psi> (kept for the next two)
    W_DTZ      -w where the selection holds, else w
    W_DTP      w where the selection holds, else 0
    W_RED      the last (1 to 4) terms, widened to FP64 and summed over the
               warp, are added to the warp's partials of their parameters

Every case ends with its own indexed branch to the next op's case (threaded
code); the code is known when the case starts, and the end of a phase is a
code like any other.

The build writes the file into its object directory (build.py).
"""
RB = 6           # register bits of the loop being written (see emit)
NS = 1 << RB     # amplitudes per thread
NU = NS // 2     # units: two amplitudes that differ in register bit 0
CRB = 6          # register bits the codes are numbered for
NPAIR = CRB * (CRB - 1) // 2
W_H, W_XH, W_YH, W_T = 0, CRB, 2 * CRB, 3 * CRB
W_CZ = 4 * CRB
W_CZO = W_CZ + NPAIR
W_CT = W_CZO + CRB            # codes of the Clifford+T loop
W_RY = W_CT
W_RX = W_RY + CRB
W_PH = W_RX + CRB
W_PP = W_PH + CRB
W_ALL = W_PP + NPAIR         # codes of the full loop
AB = CRB - 1                  # register bits of the adjoint sweep (the last selects the state)
W_DX = W_ALL
W_DY, W_DZ, W_DP, W_DPP = W_DX + AB, W_DX + 2 * AB, W_DX + 3 * AB, W_DX + 4 * AB
W_DW = W_DPP + AB * (AB - 1) // 2
W_DTZ, W_DTP, W_RED, W_ADJ = W_DW + 1, W_DW + 2, W_DW + 3, W_DW + 4

F_C = "0f3F3504F3"       # 1/sqrt2 rounded to FP32
F_2C = "0f3FB504F3"      # 2 * that (exact)
F_NC = "0fBF3504F3"      # -(1/sqrt2)
F_2 = "0f40000000"
F_M1 = "0fBF800000"
F_M2 = "0fC0000000"
F_P1 = "0f3F800000"
F_0 = "0f00000000"
# operands: offset of the thread's unit 0 in the tile, shared address of the
# tile, shared address of the staged pass, offset of the phase record in it,
# first op, index, factor (re, im), flags (bits 0..1 the factor's
# mode, then the F_ bits below), swizzled offset of the thread's copies,
# source of the next tile's copies, barrier and its threads, then immediate
# offsets in the staged pass: codes, records (less one), unit table, state
# offsets of the last phase's register bits, threads' state addresses, the
# partials' address and stride
(ADDR, TILE, BASE, PHASE, BEGIN, IDX, FR, FI, FLAGS, SWT, NSRC, BARID, NTHR,
 O_CODES, O_RECS, O_UNIT, O_DREG, O_DST, O_PART) = ("%%%d" % k for k in range(19))
F_DIRECT, F_MORE, F_CANON = 4, 8, 16    # store to the state; copy the next tile in; canonical order


def pair_index(j, k):
    """Pairs (j, k), j < k < CRB, numbered (0,1) (0,2) ... (1,2) (1,3) ..."""
    return j * (CRB - 1) - (j * (j - 1)) // 2 + (k - j - 1)


def adj_pair_index(j, k):
    """Pairs of the adjoint sweep's register bits."""
    return j * (AB - 1) - (j * (j - 1)) // 2 + (k - j - 1)


def re(k):
    return "u%d" % (2 * k)


def im(k):
    return "u%d" % (2 * k + 1)


def units(j):
    """Unit pairs (bit clear, bit set) of register bit j >= 1."""
    b = 1 << (j - 1)
    return [(k, k | b) for k in range(NU) if not k & b]


def const(name, value):
    return "mov.b64 %s, {%s, %s};" % (name, value, value)


TEMPS = 4      # units whose scalar instructions are interleaved


def unpack(k):
    """The unit's components: element 0 (xr, xi), element 1 (yr, yi)."""
    return ["mov.b64 {xr, yr}, %s;" % re(k), "mov.b64 {xi, yi}, %s;" % im(k)]


def pack(k):
    return ["mov.b64 %s, {xr, yr};" % re(k), "mov.b64 %s, {xi, yi};" % im(k)]


def scalar_units(ks, body):
    """`body` on the halves of the units ks, TEMPS units step by step (their
    scalar registers are numbered apart)."""
    out = []
    for g in range(0, len(ks), TEMPS):
        chains = []
        for n, k in enumerate(ks[g:g + TEMPS]):
            c = unpack(k) + body + pack(k)
            for t in ("xr", "xi", "yr", "yi", "na", "xx"):
                c = [x.replace(t, t + str(n)) for x in c]
            chains.append(c)
        for step in range(len(chains[0])):
            out += [c[step] for c in chains]
    return out


def on_bit0(body):
    return scalar_units(list(range(NU)), body)


def case_h(j):
    if j == 0:
        # x' = x + y; y' = x' - 2 y
        return on_bit0(["add.rn.f32 xr, xr, yr;", "fma.rn.f32 yr, yr, %s, xr;" % F_M2,
                        "add.rn.f32 xi, xi, yi;", "fma.rn.f32 yi, yi, %s, xi;" % F_M2])
    return [const("qS", F_M2)] + interleave([["add.rn.f32x2 %s, %s, %s;" % (c(x), c(x), c(y)),
                                              "fma.rn.f32x2 %s, %s, qS, %s;" % (c(y), c(y), c(x))]
                                             for x, y in units(j) for c in (re, im)])


def case_yh(j):
    # x' = x - y; y' = x' + 2 y
    if j == 0:
        return on_bit0(["sub.rn.f32 xr, xr, yr;", "fma.rn.f32 yr, yr, %s, xr;" % F_2,
                        "sub.rn.f32 xi, xi, yi;", "fma.rn.f32 yi, yi, %s, xi;" % F_2])
    return interleave([["fma.rn.f32x2 %s, %s, qM1, %s;" % (c(x), c(y), c(x)),
                        "fma.rn.f32x2 %s, %s, qP2, %s;" % (c(y), c(y), c(x))]
                       for x, y in units(j) for c in (re, im)])


def case_xh(j):
    # x' = x - i y, y' = y - i x: y'.im = y.im - x.re, x'.re = y'.im + 2 x.re;
    # x'.im = x.im - y.re, y'.re = x'.im + 2 y.re
    if j == 0:
        return on_bit0(["sub.rn.f32 yi, yi, xr;", "fma.rn.f32 xr, xr, %s, yi;" % F_2,
                        "sub.rn.f32 xi, xi, yr;", "fma.rn.f32 yr, yr, %s, xi;" % F_2])
    chains = []
    for x, y in units(j):
        chains += [["fma.rn.f32x2 %s, %s, qM1, %s;" % (im(y), re(x), im(y)),
                    "fma.rn.f32x2 %s, %s, qP2, %s;" % (re(x), re(x), im(y))],
                   ["fma.rn.f32x2 %s, %s, qM1, %s;" % (im(x), re(y), im(x)),
                    "fma.rn.f32x2 %s, %s, qP2, %s;" % (re(y), re(y), im(x))]]
    return interleave(chains)


def case_t(j):
    # re' = c re - c im; im' = re' + 2 c im
    if j == 0:
        return on_bit0(["mul.rn.f32 yr, yr, %s;" % F_C, "fma.rn.f32 yr, yi, %s, yr;" % F_NC,
                        "fma.rn.f32 yi, yi, %s, yr;" % F_2C])
    return [const("qS", F_C), const("qt", F_NC), const("qm", F_2C)] + interleave([
        ["mul.rn.f32x2 %s, %s, qS;" % (re(y), re(y)),
         "fma.rn.f32x2 %s, %s, qt, %s;" % (re(y), im(y), re(y)),
         "fma.rn.f32x2 %s, %s, qm, %s;" % (im(y), im(y), re(y))] for _, y in units(j)])


def element1(body, mask=0):
    """`body` on element 1 (yr, yi) of the units whose bits include mask."""
    return scalar_units([k for k in range(NU) if (k & mask) == mask], body)


def sign_units(mask, factor):
    return ["mul.rn.f32x2 %s, %s, %s;" % (c(k), c(k), factor) for k in range(NU) if (k & mask) == mask
            for c in (re, im)]


def case_cz(j, k):
    if j == 0:
        return element1(["neg.f32 yr, yr;", "neg.f32 yi, yi;"], 1 << (k - 1))
    return sign_units((1 << (j - 1)) | (1 << (k - 1)), "qM1")


# The record of the op that runs is op qo - 1 (the head has advanced qo).
RECORD = ["mad.lo.u32 qa, qo, 16, %s;" % BASE]
SELECTED = ["ld.shared.u64 qm, [qa+%s];" % O_RECS,
            "and.b64 qt, %s, qm;" % IDX,
            "setp.eq.u64 qp, qt, qm;"]
PARAMS = ["add.u32 qa, qa, %s;" % O_RECS, "ld.shared.v2.f32 {pa, pb}, [qa+8];"]


def case_czo(j):
    out = RECORD + SELECTED + ["selp.f32 pa, %s, %s, qp;" % (F_M1, F_P1)]
    if j == 0:
        return out + element1(["mul.rn.f32 yr, yr, pa;", "mul.rn.f32 yi, yi, pa;"])
    return out + ["mov.b64 qS, {pa, pa};"] + sign_units(1 << (j - 1), "qS")


def case_ry(j):
    # x += a y, y += b x, x += a y
    if j == 0:
        return RECORD + PARAMS + on_bit0([
            "fma.rn.f32 xr, yr, pa, xr;", "fma.rn.f32 yr, xr, pb, yr;", "fma.rn.f32 xr, yr, pa, xr;",
            "fma.rn.f32 xi, yi, pa, xi;", "fma.rn.f32 yi, xi, pb, yi;", "fma.rn.f32 xi, yi, pa, xi;"])
    return RECORD + PARAMS + ["mov.b64 qS, {pa, pa};", "mov.b64 qt, {pb, pb};"] + interleave([
        ["fma.rn.f32x2 %s, %s, qS, %s;" % (c(x), c(y), c(x)),
         "fma.rn.f32x2 %s, %s, qt, %s;" % (c(y), c(x), c(y)),
         "fma.rn.f32x2 %s, %s, qS, %s;" % (c(x), c(y), c(x))] for x, y in units(j) for c in (re, im)])


def case_rx(j):
    # with w = i y (w.re = -y.im, w.im = y.re): x += a w, w += b x, x += a w
    out = RECORD + PARAMS + ["neg.f32 nc, pa;", "neg.f32 nb, pb;"]
    if j == 0:
        return out + on_bit0([
            "fma.rn.f32 xr, yi, nc, xr;", "fma.rn.f32 xi, yr, pa, xi;",
            "fma.rn.f32 yi, xr, nb, yi;", "fma.rn.f32 yr, xi, pb, yr;",
            "fma.rn.f32 xr, yi, nc, xr;", "fma.rn.f32 xi, yr, pa, xi;"])
    out += ["mov.b64 qS, {pa, pa};", "mov.b64 qt, {nc, nc};", "mov.b64 qm, {pb, pb};", "mov.b64 qv, {nb, nb};"]
    chains = []
    for x, y in units(j):
        chains += [["fma.rn.f32x2 %s, %s, qt, %s;" % (re(x), im(y), re(x)),
                    "fma.rn.f32x2 %s, %s, qv, %s;" % (im(y), re(x), im(y)),
                    "fma.rn.f32x2 %s, %s, qt, %s;" % (re(x), im(y), re(x))],
                   ["fma.rn.f32x2 %s, %s, qS, %s;" % (im(x), re(y), im(x)),
                    "fma.rn.f32x2 %s, %s, qm, %s;" % (re(y), im(x), re(y)),
                    "fma.rn.f32x2 %s, %s, qS, %s;" % (im(x), re(y), im(x))]]
    return out + interleave(chains)


def phase_units(mask):
    # re' = re a - im b; im' = re b + im a
    out = ["neg.f32 nb, pb;", "mov.b64 qS, {pa, pa};", "mov.b64 qt, {pb, pb};", "mov.b64 qm, {nb, nb};"]
    for k in range(NU):
        if (k & mask) == mask:
            out += ["mul.rn.f32x2 qv, %s, qm;" % im(k),
                    "mul.rn.f32x2 qu, %s, qt;" % re(k),
                    "fma.rn.f32x2 %s, %s, qS, qv;" % (re(k), re(k)),
                    "fma.rn.f32x2 %s, %s, qS, qu;" % (im(k), im(k))]
    return out


PHASE1 = ["neg.f32 nb, pb;"]
PHASE1_BODY = ["mul.rn.f32 na, yi, nb;", "mul.rn.f32 xx, yr, pb;", "fma.rn.f32 yr, yr, pa, na;",
               "fma.rn.f32 yi, yi, pa, xx;"]


def case_ph(j):
    out = RECORD + SELECTED + PARAMS + ["selp.f32 pa, pa, %s, qp;" % F_P1, "selp.f32 pb, pb, %s, qp;" % F_0]
    return out + (PHASE1 + element1(PHASE1_BODY) if j == 0 else phase_units(1 << (j - 1)))


def case_pp(j, k):
    out = RECORD + PARAMS
    return out + (PHASE1 + element1(PHASE1_BODY, 1 << (k - 1)) if j == 0
                  else phase_units((1 << (j - 1)) | (1 << (k - 1))))


HALF = NU // 2     # adjoint: unit k of psi, unit k + HALF of lambda


def push(value):
    return ["mov.f32 da3, da2;", "mov.f32 da2, da1;", "mov.f32 da1, da0;"] + value


def packed_sum(terms):
    """Two packed sums each of the positive and the negative products (qS, qu
    and qt, qm): terms (sign, a, b) -> +- a b."""
    acc = {1: ["qS", "qu"], -1: ["qt", "qm"]}
    seen, n, out = set(), {1: 0, -1: 0}, []
    for sign, a, b in terms:
        r = acc[sign][n[sign] & 1]
        n[sign] += 1
        out.append("mul.rn.f32x2 %s, %s, %s;" % (r, a, b) if r not in seen
                   else "fma.rn.f32x2 %s, %s, %s, %s;" % (r, a, b, r))
        seen.add(r)
    for sign, r in ((1, "qS"), (-1, "qt")):
        other = {"qS": "qu", "qt": "qm"}[r]
        if other in seen:
            out.append("add.rn.f32x2 %s, %s, %s;" % (r, r, other))
    return out + ["mov.b64 {pa, nb}, qS;", "mov.b64 {pb, nc}, qt;", "sub.rn.f32 pa, pa, pb;", "sub.rn.f32 nb, nb, nc;"]


def inner(k, sign=1):
    """Im conj(lambda) psi of unit k."""
    return [(sign, re(k + HALF), im(k)), (-sign, im(k + HALF), re(k))]


def case_dx(j, which):
    """X (which 0): (l0r p1i - l0i p1r) + (l1r p0i - l1i p0r);
    Y (which 1): (l1r p0r + l1i p0i) - (l0r p1r + l0i p1i)."""
    if j == 0:
        out = []
        for k in range(HALF):
            regs = (re(k), im(k), re(k + HALF), im(k + HALF))
            u = ["mov.b64 {xr0, yr0}, %s;" % regs[0], "mov.b64 {xi0, yi0}, %s;" % regs[1],
                 "mov.b64 {xr1, yr1}, %s;" % regs[2], "mov.b64 {xi1, yi1}, %s;" % regs[3]]
            terms = ([("pa", "xr1", "yi0"), ("pb", "xi1", "yr0"), ("nb", "yr1", "xi0"), ("nc", "yi1", "xr0")]
                     if which == 0 else
                     [("pa", "yr1", "xr0"), ("nb", "yi1", "xi0"), ("pb", "xr1", "yr0"), ("nc", "xi1", "yi0")])
            out += u + [("mul.rn.f32 %s, %s, %s;" % t) if k == 0 else "fma.rn.f32 %s, %s, %s, %s;" % (t + (t[0],))
                        for t in terms]
        return out + ["add.rn.f32 pa, pa, nb;", "add.rn.f32 pb, pb, nc;"] + push(["sub.rn.f32 da0, pa, pb;"])
    terms = []
    b = 1 << (j - 1)
    for x in range(HALF):
        if x & b:
            continue
        y = x | b
        if which == 0:
            terms += [(1, re(x + HALF), im(y)), (-1, im(x + HALF), re(y)), (1, re(y + HALF), im(x)), (-1, im(y + HALF), re(x))]
        else:
            terms += [(1, re(y + HALF), re(x)), (-1, re(x + HALF), re(y)), (1, im(y + HALF), im(x)), (-1, im(x + HALF), im(y))]
    return packed_sum(terms) + push(["add.rn.f32 da0, pa, nb;"])


def case_dz(j):
    if j == 0:
        return packed_sum([t for k in range(HALF) for t in inner(k)]) + push(["sub.rn.f32 da0, pa, nb;"])
    b = 1 << (j - 1)
    return packed_sum([t for k in range(HALF) for t in inner(k, -1 if k & b else 1)]) + push(["add.rn.f32 da0, pa, nb;"])


def subset_sum(mask, hi):
    """w over the units whose bits include mask (hi: their element 1 only)."""
    out = packed_sum([t for k in range(HALF) if (k & mask) == mask for t in inner(k)])
    return out + (["mov.f32 pa, nb;"] if hi else ["add.rn.f32 pa, pa, nb;"])


def case_dp(j):
    return subset_sum(0 if j == 0 else 1 << (j - 1), j == 0) + RECORD + SELECTED + push(
        ["selp.f32 da0, pa, %s, qp;" % F_0])


def case_dpp(j, k):
    return subset_sum((0 if j == 0 else 1 << (j - 1)) | 1 << (k - 1), j == 0) + push(["mov.f32 da0, pa;"])


def case_red():
    out = RECORD + ["add.u32 qa, qa, %s;" % O_RECS, "ld.shared.v2.u32 {a0, a1}, [qa+8];", "mov.u32 b0, %laneid;"]
    out += ["cvt.f64.f32 e%d, da%d;" % (k, k) for k in range(4)]

    def swap(dst, a, o):                       # dst = a of lane ^ o
        return ["mov.b64 {b2, b3}, %s;" % a, "shfl.sync.bfly.b32 b2, b2, %d, 31, -1;" % o,
                "shfl.sync.bfly.b32 b3, b3, %d, 31, -1;" % o, "mov.b64 %s, {b2, b3};" % dst]
    # recursive halving: lane bit 1 keeps terms 2 and 3, lane bit 0 the odd one
    out += ["and.b32 b1, b0, 2;", "setp.ne.u32 qp, b1, 0;"]
    for k in (0, 1):
        out += ["selp.f64 e4, e%d, e%d, qp;" % (k, k + 2), "selp.f64 e%d, e%d, e%d, qp;" % (k, k + 2, k)]
        out += swap("e4", "e4", 2) + ["add.rn.f64 e%d, e%d, e4;" % (k, k)]
    out += ["and.b32 b1, b0, 1;", "setp.ne.u32 qp, b1, 0;",
            "selp.f64 e4, e0, e1, qp;", "selp.f64 e0, e1, e0, qp;"]
    out += swap("e4", "e4", 1) + ["add.rn.f64 e0, e0, e4;"]
    for o in (4, 8, 16):
        out += swap("e4", "e0", o) + ["add.rn.f64 e0, e0, e4;"]
    # lane i < count holds term i, the (count - 1 - i)-th parameter from a0
    out += ["sub.u32 b1, a1, b0;", "add.u32 b1, b1, a0;", "sub.u32 b1, b1, 1;",
            "ld.shared.v2.u64 {qt, qm}, [%s+%s];" % (BASE, O_PART),
            "cvt.u64.u32 qS, b1;", "mul.lo.u64 qS, qS, qm;", "add.u64 qt, qt, qS;",
            "mov.u32 b1, %tid.x;", "shr.u32 b1, b1, 5;", "mul.wide.u32 qS, b1, 8;", "add.u64 qt, qt, qS;",
            "setp.lt.u32 qp, b0, a1;", "@qp red.global.add.f64 [qt], e0;"]
    return out


GROUP = 8     # independent chains interleaved


def interleave(chains):
    """The instructions of independent chains, GROUP chains at a time step by
    step: a dependent instruction follows its source at a distance that covers
    the FMA latency."""
    out = []
    for g in range(0, len(chains), GROUP):
        grp = chains[g:g + GROUP]
        for step in range(max(len(c) for c in grp)):
            out += [c[step] for c in grp if step < len(c)]
    return out


def cases(full, adj=False):
    """Case bodies by code; None: a code this loop does not hold."""
    body = [None] * (W_ADJ if adj else W_ALL if full else W_CT)
    for j in range(AB if adj else RB):
        body[W_H + j] = case_h(j)
        body[W_XH + j] = case_xh(j)
        body[W_YH + j] = case_yh(j)
        body[W_T + j] = case_t(j)
        body[W_CZO + j] = case_czo(j)
        if full:
            body[W_RY + j] = case_ry(j)
            body[W_RX + j] = case_rx(j)
            body[W_PH + j] = case_ph(j)
        if adj:
            body[W_DX + j] = case_dx(j, 0)
            body[W_DY + j] = case_dx(j, 1)
            body[W_DZ + j] = case_dz(j)
            body[W_DP + j] = case_dp(j)
            for k in range(j + 1, AB):
                body[W_DPP + adj_pair_index(j, k)] = case_dpp(j, k)
        for k in range(j + 1, AB if adj else RB):
            body[W_CZ + pair_index(j, k)] = case_cz(j, k)
            if full:
                body[W_PP + pair_index(j, k)] = case_pp(j, k)
    if adj:
        body[W_DW] = subset_sum(0, False) + ["mov.f32 dw, pa;"]
        body[W_DTZ] = RECORD + SELECTED + ["neg.f32 pb, dw;"] + push(["selp.f32 da0, pb, dw, qp;"])
        body[W_DTP] = RECORD + SELECTED + push(["selp.f32 da0, dw, %s, qp;" % F_0])
        body[W_RED] = case_red()
    assert adj or RB < CRB or all(b is not None for b in body)
    return body


def head(ncodes):
    """Start of every case (op qo, the next op's code in qn): advances qo, takes
    the next op's code for the branch at the case's end and loads the one
    after it.  No test separates the head from the branch -- a phase's codes
    end with the end code -- so the table look-up of the branch target runs
    under the case's arithmetic.  A code outside the table ends the phase (the
    lowering never makes one)."""
    return ["min.u32 qc, qn, %d;" % ncodes,
            "add.u32 qo, qo, 1;",
            "add.u32 qa, %s, qo;" % BASE,
            "ld.shared.u8 qn, [qa+%s+1];" % O_CODES]


def branch(L):
    return ["brx.idx.uni qc, " + L("TBL") + ";"]


def slots(store):
    """All units from / to the tile, in Gray-code order (one XOR with a
    register bit's offset per address), the two halves of the units as two
    chains."""
    out = ["ld.shared.v4.u32 {b0, b1, b2, b3}, [qh];", "ld.shared.v2.u32 {b4, b5}, [qh+16];",
           "mov.u32 a0, %s;" % ADDR, "xor.b32 a1, %s, b%d;" % (ADDR, RB - 1)]
    for i in range(NU // 2):
        if i:
            bit = (i & -i).bit_length()          # register bit 1 + trailing zeros
            out += ["xor.b32 a0, a0, b%d;" % bit, "xor.b32 a1, a1, b%d;" % bit]
        for a, k in (("a0", i ^ (i >> 1)), ("a1", (i ^ (i >> 1)) + NU // 2)):
            # the XORs act on offsets in the tile (its address is not a
            # multiple of its size)
            out.append("add.u32 qa, %s, %s;" % (a, TILE))
            out.append("st.shared.v2.b64 [qa], {%s, %s};" % (re(k), im(k)) if store
                       else "ld.shared.v2.b64 {%s, %s}, [qa];" % (re(k), im(k)))
    return out


def factor(L):
    """The thread's factor: mode 0 none, 1 real, 2 complex."""
    out = ["and.b32 qc, %s, 3;" % FLAGS,
           "setp.eq.u32 qp, qc, 0;",
           "@qp bra.uni " + L("STORE") + ";",
           "mov.b64 qS, {%s, %s};" % (FR, FR),
           "setp.eq.u32 qp, qc, 1;",
           "@qp bra.uni " + L("REAL") + ";",
           "neg.f32 nb, %s;" % FI,
           "mov.b64 qt, {%s, %s};" % (FI, FI),
           "mov.b64 qm, {nb, nb};"]
    for k in range(NU):
        out += ["mul.rn.f32x2 qv, %s, qm;" % im(k),
                "mul.rn.f32x2 qu, %s, qt;" % re(k),
                "fma.rn.f32x2 %s, %s, qS, qv;" % (re(k), re(k)),
                "fma.rn.f32x2 %s, %s, qS, qu;" % (im(k), im(k))]
    out += ["bra.uni " + L("STORE") + ";", L("REAL") + ":"]
    out += sign_units(0, "qS")
    return out


def flag(bit):
    return ["and.b32 qc, %s, %d;" % (FLAGS, bit), "setp.eq.u32 qp, qc, 0;"]


def next_tile(L):
    """Last phase of a direct pass: once every thread has loaded its units the
    tile's buffer is free, and the next tile is copied in while the ops run."""
    out = flag(F_DIRECT) + ["@qp bra.uni " + L("OPS") + ";", "bar.sync %s, %s;" % (BARID, NTHR)]
    out += flag(F_MORE) + ["@qp bra.uni " + L("OPS") + ";"]
    for it in range(NU):
        out += ["ld.shared.v2.u64 {qt, qm}, [%s+%s];" % (BASE, "%s+%d" % (O_UNIT, 16 * it)),
                "cvt.u32.u64 qc, qm;",
                "xor.b32 qc, qc, %s;" % SWT,
                "add.u32 qc, qc, %s;" % TILE,
                "add.u64 qt, qt, %s;" % NSRC,
                "cp.async.cg.shared.global [qc], [qt], 16;"]
    return out + [L("OPS") + ":"]


def state_stores(canon):
    """All units to the state, Gray-code order: from one unit to the next one
    register bit's offset is added or subtracted."""
    out, prev = [], 0
    for i in range(NU):
        k = i ^ (i >> 1)
        if i:
            bit = (k ^ prev).bit_length()       # register bit of the unit bit that changed
            out.append("%s.s64 qt, qt, d%d;" % ("add" if k > prev else "sub", bit))
        prev = k
        if canon:
            out += unpack(k) + ["st.global.v4.f32 [qt], {xr, xi, yr, yi};"]
        else:
            out.append("st.global.v2.b64 [qt], {%s, %s};" % (re(k), im(k)))
    return out


def direct_store(L):
    out = flag(F_DIRECT) + ["@qp bra.uni " + L("TILE") + ";",
                            "mov.u32 qa, %tid.x;",
                            "mad.lo.u32 qa, qa, 8, %s;" % BASE,
                            "ld.shared.u64 qt, [qa+%s];" % O_DST]
    for j in range(1, RB):
        out.append("ld.shared.u64 d%d, [%s+%s];" % (j, BASE, "%s+%d" % (O_DREG, 8 * j)))
    out += flag(F_CANON) + ["@qp bra.uni " + L("RAW") + ";"]
    out += state_stores(True) + ["bra.uni " + L("END") + ";", L("RAW") + ":"]
    out += state_stores(False) + ["bra.uni " + L("END") + ";", L("TILE") + ":"]
    return out


def asm_text(prefix, full, adj=False):
    """PTX of one phase: loads the thread's units, runs the ops from `begin` to the
    end code, applies the factor, stores the units to the tile or (direct) to the
    state.  The units live in registers of the block's own, so nothing has to
    be moved at its boundary."""
    def L(name):
        return "%s_%s" % (prefix, name)
    body = cases(full, adj)
    n = len(body)
    lines = ["{",
             ".reg .pred qp;",
             ".reg .u32 qo, qc, qn, qa, qh, a0, a1, b<%d>;" % CRB,
             ".reg .b64 qm, qt, qS, qv, qu, qM1, qP2, d<%d>;" % RB,
             ".reg .f32 xr, xi, yr, yi, pa, pb, nb, nc;",
             ".reg .f32 " + ", ".join(t + str(n) for n in range(TEMPS) for t in ("xr", "xi", "yr", "yi", "na", "xx")) + ";",
             ".reg .b64 u<%d>;" % NS] + ([".reg .f32 da0, da1, da2, da3, dw;", ".reg .f64 e<5>;"] if adj else []) + [
             "add.u32 qh, %s, %s;" % (BASE, PHASE)]
    lines += slots(False)
    lines += next_tile(L)
    lines += ["mov.b64 qM1, {%s, %s};" % (F_M1, F_M1),
              "mov.b64 qP2, {%s, %s};" % (F_2, F_2),
              "mov.u32 qo, %s;" % BEGIN,
              "add.u32 qa, %s, qo;" % BASE,
              "ld.shared.u8 qc, [qa+%s];" % O_CODES,
              "ld.shared.u8 qn, [qa+%s+1];" % O_CODES,
              L("TBL") + ": .branchtargets " + ", ".join([L("C%d" % c if body[c] else "DONE") for c in range(n)]
                                                              + [L("DONE")]) + ";",
              "min.u32 qc, qc, %d;" % n]
    lines += branch(L)
    for c, b in enumerate(body):
        if b:
            lines.append(L("C%d" % c) + ":")
            lines += head(n) + b + branch(L)
    lines.append(L("DONE") + ":")
    lines += factor(L)
    lines.append(L("STORE") + ":")
    lines += direct_store(L)
    lines.append("add.u32 qh, %s, %s;" % (BASE, PHASE))
    lines += slots(True)
    lines += [L("END") + ":", "}"]
    return lines


def set_register_bits(rb):
    global RB, NS, NU
    RB, NS, NU = rb, 1 << rb, 1 << (rb - 1)


def emit():
    out = ["// qs_op_loop.inc -- generated by gen_op_loop.py; do not edit.",
           "//",
           "// The op loop of the wide fused pass (complex64, 2^RB slots, RB register",
           "// bits) as inline PTX: one byte-code load and one indexed branch per op.",
           "// OpLoop<0, RB>: the Clifford+T gates; OpLoop<1, RB>: also the",
           "// parameterised gates; OpLoop<2, 6>: the adjoint sweep.",
           "",
           "template <int KIND, int RB> struct OpLoop;"]
    for kind, rb, prefix in ((0, 6, "QSWCT"), (1, 6, "QSWFL"), (2, 6, "QSWAD"), (0, 5, "QSVCT"), (1, 5, "QSVFL")):
        set_register_bits(rb)
        out.append("template <> struct OpLoop<%d, %d> {" % (kind, rb))
        out.append("    template <int O_CODES, int O_RECS, int O_UNIT, int O_DREG, int O_DST, int O_PART>")
        out.append("    static __device__ __forceinline__ void run(uint32_t addr, uint32_t tile, uint32_t base,")
        out.append("                                               uint32_t phase, int ob,")
        out.append("                                               unsigned long long idx, float fr, float fi,")
        out.append("                                               uint32_t flags, uint32_t swt, const void *nsrc,")
        out.append("                                               uint32_t barid, uint32_t nthr)")
        out.append("    {")
        out.append("        asm volatile(")
        for line in asm_text(prefix, kind > 0, kind == 2):
            out.append('            "%s\\n"' % line.replace("%tid", "%%tid").replace("%laneid", "%%laneid"))
        out.append('            : : "r"(addr), "r"(tile), "r"(base), "r"(phase), "r"(ob), "l"(idx), "f"(fr), "f"(fi),')
        out.append('                "r"(flags), "r"(swt), "l"(nsrc), "r"(barid), "r"(nthr), "n"(O_CODES), "n"(O_RECS), "n"(O_UNIT),')
        out.append('                "n"(O_DREG), "n"(O_DST), "n"(O_PART)')
        out.append('            : "memory");')
        out.append("    }")
        out.append("};")
    set_register_bits(CRB)
    return "\n".join(out) + "\n"

