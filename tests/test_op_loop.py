"""The wide pass's phase in inline PTX (csrc/gen_op_loop.py), run on the CPU by
an interpreter of the instruction forms it uses: one thread loads its 64
amplitudes from a tile in shared memory through swizzled addresses, runs a
list of ops, applies its factor and stores them back, to the tile or (direct)
to the state while it copies the next tile in.  Every shared access must fall
inside the tile or the staged pass and be aligned to its width; the tile
starts at an address that is no multiple of its size.  Checked against the
gates' definitions in FP64 for every byte code, with several register sets.

Tolerance: an op is at most six FP32 roundings of values of size <= 2 (its
shears' coefficients are below 1.1 here), the phase at most 12 ops and a
factor of three more: 75 * 2^-24 * 2 = 9e-6 absolute."""
import importlib.util
import math
import os
import struct

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1608_00263_gb300", "csrc")
f32 = np.float32


def _gen():
    spec = importlib.util.spec_from_file_location("gen_op_loop", os.path.join(CSRC, "gen_op_loop.py"))
    g = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(g)
    return g


G = _gen()
SMEM_STATIC, TILE = 1024, 1024 + 10608       # staged pass; the tile follows it
O_PHASE, O_DREG, O_OPS, O_CODES, O_UNIT, O_DST = 144, 96, 528, 4624, 5008, 6000
STATE, NEXT = 1 << 40, 3 << 40                # addresses in the state


def swizzle(e):
    u = e >> 1
    return e ^ ((((u >> 3) ^ (u >> 6) ^ (u >> 9) ^ (u >> 12)) & 7) << 1)


class Thread:
    def __init__(self, lines, mem, lo, hi, operands):
        self.mem, self.lo, self.hi = mem, lo, hi
        self.r = dict(operands)
        self.stores, self.copies = {}, []
        self.labels, self.code, self.table = {}, [], None
        for line in lines:
            line = line.strip().rstrip(";").strip()
            if ".branchtargets" in line:
                self.table = [x.strip() for x in line.split(".branchtargets")[1].split(",")]
            elif line.endswith(":"):
                self.labels[line[:-1]] = len(self.code)
            elif line and line not in "{}" and not line.startswith(".reg"):
                self.code.append(line)

    def val(self, t):
        if t.startswith("0f"):
            return np.frombuffer(struct.pack("<I", int(t[2:], 16)), dtype=f32)[0]
        return int(t) if t.lstrip("-").isdigit() else self.r[t]

    def addr(self, t, width):
        a = 0
        for part in t.strip("[]").split("+"):
            a += int(self.val(part))
        assert a % width == 0, ("misaligned", t, a, width)
        assert self.lo <= a and a + width <= self.hi, ("outside shared memory", t, a)
        return a

    def run(self):
        r, pc, steps = self.r, 0, 0
        while pc < len(self.code):
            steps += 1
            assert steps < 200000
            op, rest = self.code[pc].split(None, 1)
            pc += 1
            if op.startswith("@"):
                if not r[op[1:]]:
                    continue
                op, rest = rest.split(None, 1)
            a = [x.strip() for x in rest.replace("{", "").replace("}", "").split(",")]
            if op == "bar.sync":
                continue
            if op == "bra.uni":
                pc = self.labels[a[0]]
            elif op == "brx.idx.uni":
                pc = self.labels[self.table[int(r[a[0]])]]
            elif op in ("add.rn.f32x2", "mul.rn.f32x2", "fma.rn.f32x2"):
                x, y = r[a[1]], r[a[2]]
                if op[0] == "a":
                    r[a[0]] = [f32(x[0] + y[0]), f32(x[1] + y[1])]
                elif op[0] == "m":
                    r[a[0]] = [f32(x[0] * y[0]), f32(x[1] * y[1])]
                else:
                    z = r[a[3]]
                    r[a[0]] = [f32(np.float64(x[i]) * np.float64(y[i]) + np.float64(z[i])) for i in (0, 1)]
            elif op == "mov.b64":
                if rest.startswith("{"):
                    r[a[0]], r[a[1]] = r[a[2]]
                else:
                    r[a[0]] = [self.val(a[1]), self.val(a[2])]
            elif op == "mov.f32":
                r[a[0]] = self.val(a[1])
            elif op == "mov.u32":
                r[a[0]] = int(self.val(a[1]))
            elif op == "add.rn.f32":
                r[a[0]] = f32(self.val(a[1]) + self.val(a[2]))
            elif op == "sub.rn.f32":
                r[a[0]] = f32(self.val(a[1]) - self.val(a[2]))
            elif op == "mul.rn.f32":
                r[a[0]] = f32(self.val(a[1]) * self.val(a[2]))
            elif op == "fma.rn.f32":
                r[a[0]] = f32(np.float64(self.val(a[1])) * np.float64(self.val(a[2])) + np.float64(self.val(a[3])))
            elif op == "neg.f32":
                r[a[0]] = f32(-self.val(a[1]))
            elif op in ("add.u32", "add.u64", "add.s64"):
                r[a[0]] = int(self.val(a[1])) + int(self.val(a[2]))
            elif op == "xor.b32":
                r[a[0]] = int(self.val(a[1])) ^ int(self.val(a[2]))
            elif op == "min.u32":
                r[a[0]] = min(int(self.val(a[1])), int(self.val(a[2])))
            elif op == "mad.lo.u32":
                r[a[0]] = int(self.val(a[1])) * int(a[2]) + int(self.val(a[3]))
            elif op == "setp.ge.s32":
                r[a[0]] = self.val(a[1]) >= self.val(a[2])
            elif op in ("setp.eq.u32", "setp.eq.u64"):
                r[a[0]] = self.val(a[1]) == self.val(a[2])
            elif op == "sub.s64":
                r[a[0]] = int(self.val(a[1])) - int(self.val(a[2]))
            elif op == "cvt.u32.u64":
                r[a[0]] = r[a[1]] & 0xFFFFFFFF
            elif op == "and.b32":
                r[a[0]] = int(self.val(a[1])) & int(a[2])
            elif op == "cp.async.cg.shared.global":
                self.copies.append((self.addr(a[0], 16), int(r[a[1].strip("[]")])))
            elif op in ("st.global.v2.b64", "st.global.v4.f32"):
                at = int(r[a[0].strip("[]")])
                assert at % 16 == 0 and at not in self.stores
                self.stores[at] = r[a[1]] + r[a[2]] if "b64" in op else [r[x] for x in a[1:5]]
            elif op == "ld.shared.v2.u64":
                r[a[0]], r[a[1]] = struct.unpack_from("<2Q", self.mem, self.addr(a[2], 16))
            elif op == "and.b64":
                r[a[0]] = r[a[1]] & r[a[2]]
            elif op == "selp.f32":
                r[a[0]] = self.val(a[1]) if r[a[3]] else self.val(a[2])
            elif op == "ld.shared.u8":
                r[a[0]] = self.mem[self.addr(a[1], 1)]
            elif op == "ld.shared.u64":
                r[a[0]] = struct.unpack_from("<Q", self.mem, self.addr(a[1], 8))[0]
            elif op in ("ld.shared.v4.u32", "ld.shared.v2.u32"):
                n = 4 if "v4" in op else 2
                for k, v in enumerate(struct.unpack_from("<%dI" % n, self.mem, self.addr(a[n], 4 * n))):
                    r[a[k]] = v
            elif op == "ld.shared.v2.f32":
                v = np.frombuffer(self.mem, f32, 2, self.addr(a[2], 8))
                r[a[0]], r[a[1]] = f32(v[0]), f32(v[1])
            elif op == "ld.shared.v2.b64":
                v = np.frombuffer(self.mem, f32, 4, self.addr(a[2], 16)).copy()
                r[a[0]], r[a[1]] = [v[0], v[1]], [v[2], v[3]]
            elif op == "st.shared.v2.b64":
                struct.pack_into("<4f", self.mem, self.addr(a[0], 16), *(r[a[1]] + r[a[2]]))
            else:
                raise AssertionError("instruction form not interpreted: " + self.code[pc - 1])


def op_matrix(code, p0, p1):
    """(register bits, matrix or (mask bits, factor)) of a byte code."""
    s = 1.0
    if code < G.W_T:
        j = code % G.RB
        m = {0: [[s, s], [s, -s]], 1: [[s, -1j], [-1j, s]], 2: [[s, -s], [s, s]]}[code // G.RB]
        return j, np.array(m, dtype=complex)
    if G.W_RY <= code < G.W_PH and code >= G.W_CT:
        j = (code - G.W_RY) % G.RB
        sx = np.array([[1, p0], [0, 1]], dtype=complex)
        sy = np.array([[1, 0], [p1, 1]], dtype=complex)
        m = sx @ sy @ sx
        if code >= G.W_RX:                       # between x and w = i y
            d = np.diag([1, 1j])
            m = np.linalg.inv(d) @ m @ d
        return j, m
    raise AssertionError(code)


def expected(v, t, ops, selected):
    """v: amplitudes of the thread by register index (bit j = register bit j)."""
    idx = np.arange(64)
    for code, p0, p1, sel in ops:
        p0, p1 = float(f32(p0)), float(f32(p1))
        if code < G.W_T or G.W_RY <= code < G.W_PH:
            j, m = op_matrix(code, p0, p1)
            x, y = v[(idx >> j) & 1 == 0], v[(idx >> j) & 1 == 1]
            nx, ny = m[0, 0] * x + m[0, 1] * y, m[1, 0] * x + m[1, 1] * y
            v = v.copy()
            v[(idx >> j) & 1 == 0], v[(idx >> j) & 1 == 1] = nx, ny
            continue
        pairs = [(j, k) for j in range(G.RB) for k in range(j + 1, G.RB)]
        if code < G.W_CZ:
            mask, f = 1 << (code - G.W_T), np.exp(1j * math.pi / 4)
        elif code < G.W_CZO:
            j, k = pairs[code - G.W_CZ]
            mask, f = 1 << j | 1 << k, -1.0
        elif code < G.W_CT:
            mask, f = 1 << (code - G.W_CZO), -1.0 if sel else 1.0
        elif code < G.W_PP:
            mask, f = 1 << (code - G.W_PH), (p0 + 1j * p1) if sel else 1.0
        else:
            j, k = pairs[code - G.W_PP]
            mask, f = 1 << j | 1 << k, p0 + 1j * p1
        v = np.where((idx & mask) == mask, v * f, v)
    return v


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("t,regs", [(13, (0, 1, 2, 3, 4, 5)), (13, (0, 7, 8, 10, 11, 12)), (11, (0, 2, 4, 6, 8, 10)),
                                    (12, (0, 3, 5, 9, 10, 11))])
def test_phase_on_one_thread(full, t, regs):
    rng = np.random.default_rng(7 + t + 100 * full)
    ncodes = G.W_ALL if full else G.W_CT
    lines = G.asm_text("X", full)
    others = [b for b in range(t) if b not in regs]
    # every byte code once, in lists of up to 12 ops
    order = rng.permutation(ncodes)
    for start in range(0, ncodes, 12):
        codes = [int(c) for c in order[start:start + 12]]
        tid = int(rng.integers(0, 1 << len(others)))
        e0 = sum(((tid >> k) & 1) << b for k, b in enumerate(others))
        mem = bytearray(TILE + (8 << t))
        tile = rng.uniform(-1, 1, (1 << t, 2)).astype(f32)
        for u in range(1 << (t - 1)):       # unit: two real parts, two imaginary parts
            a = TILE + swizzle(2 * u) * 8
            struct.pack_into("<4f", mem, a, tile[2 * u, 0], tile[2 * u + 1, 0], tile[2 * u, 1], tile[2 * u + 1, 1])
        struct.pack_into("<6I", mem, SMEM_STATIC + O_PHASE, *[swizzle(1 << b) * 8 for b in regs])
        tau, ops, first = 37, [], 3
        for k, c in enumerate(codes):
            sel = bool(rng.integers(0, 2))
            # a selection on tile bits of the thread and tile-number bits
            want = (37 << 32 | e0) if sel else 1 << 34 | (37 << 32)
            want &= ~((1 << 32) | 1)
            sel = ((tau << 32 | e0) & want) == want
            p = (math.cos(0.7 + k), math.sin(0.7 + k))
            struct.pack_into("<Q2f", mem, SMEM_STATIC + O_OPS + 16 * (first + k), want, *p)
            mem[SMEM_STATIC + O_CODES + first + k] = c
            ops.append((c, p[0], p[1], sel))
        mem[SMEM_STATIC + O_CODES + first + len(codes)] = 255      # the end code
        # the state: tile bit b is qubit 2 b; the thread's copies and slot 0
        qbit = [8 << (2 * b) for b in range(t)]
        deposit = lambda e: sum(qbit[b] for b in range(t) if (e >> b) & 1)
        units = [(deposit(2 * (1 << len(others)) * k), swizzle(2 * (1 << len(others)) * k) * 8) for k in range(32)]
        for k, (goff, soff) in enumerate(units):
            struct.pack_into("<2Q", mem, SMEM_STATIC + O_UNIT + 16 * k, goff, soff)
        struct.pack_into("<6Q", mem, SMEM_STATIC + O_DREG, *[qbit[b] for b in regs])
        struct.pack_into("<Q", mem, SMEM_STATIC + O_DST + 8 * tid, STATE + deposit(e0))
        swt = swizzle(2 * tid) * 8
        for mode, fac in ((0, 1.0), (1, -0.25), (2, 0.6 + 0.8j), (1 | G.F_DIRECT, 0.5), (2 | G.F_DIRECT | G.F_MORE, 1j),
                          (1 | G.F_DIRECT | G.F_CANON, 2.0)):
            m2 = bytearray(mem)
            fac = complex(fac)
            operands = dict(zip(["%%%d" % k for k in range(18)] + ["%tid.x"],
                                [swizzle(e0) * 8, TILE, SMEM_STATIC, O_PHASE, first, tau << 32 | e0,
                                 f32(fac.real), f32(fac.imag), mode, swt, NEXT, 0, 128, O_CODES, O_OPS - 16, O_UNIT,
                                 O_DREG, O_DST, tid]))
            th = Thread(lines, m2, SMEM_STATIC, TILE + (8 << t), operands)
            th.run()
            assert th.copies == ([(TILE + (soff ^ swt), NEXT + goff) for goff, soff in units] if mode & G.F_MORE else [])
            elems = [e0 | sum(((s >> j) & 1) << b for j, b in enumerate(regs)) for s in range(64)]
            v = expected(tile[elems, 0].astype(complex) + 1j * tile[elems, 1], t, ops, None) * fac
            got = np.empty(64, complex)
            if mode & G.F_DIRECT:
                for s, e in enumerate(elems):
                    q = th.stores[STATE + deposit(e & ~1)]
                    got[s] = complex(*(q[2 * (e & 1):][:2] if mode & G.F_CANON else (q[e & 1], q[2 + (e & 1)])))
                assert len(th.stores) == 32 and m2 == mem
            for s, e in enumerate(elems if not mode & G.F_DIRECT else []):
                q = struct.unpack_from("<4f", m2, TILE + swizzle(e & ~1) * 8)
                got[s] = complex(q[e & 1], q[2 + (e & 1)])
            scale = np.max(np.abs(v)) + 1.0     # butterflies grow by sqrt(2) each
            assert np.max(np.abs(got - v)) < 9e-6 * scale, (full, t, regs, codes, mode)
            if mode & G.F_DIRECT:
                continue
            # nothing else in the tile moved
            assert not th.stores
            mine = {TILE + swizzle(e & ~1) * 8 for e in elems}
            for u in range(1 << (t - 1)):
                a = TILE + swizzle(2 * u) * 8
                if a not in mine:
                    assert m2[a:a + 16] == mem[a:a + 16]


@pytest.mark.parametrize("code", [c for c in range(G.W_DX, G.W_RED) if c != G.W_DW])
@pytest.mark.parametrize("sel", [False, True])
def test_derivative_terms(code, sel):
    """The adjoint loop's terms of one thread against their definitions; the
    selector of psi and lambda is register bit 5.  64 products of values <= 1
    in FP32: 64 * 2^-23 absolute at most."""
    t, regs, e0 = 13, (0, 3, 4, 7, 9, 12), (1 << 5) | (1 << 8)
    rng = np.random.default_rng(code)
    mem = bytearray(TILE + (8 << t))
    elems = [e0 | sum(((s >> j) & 1) << b for j, b in enumerate(regs)) for s in range(64)]
    v = rng.uniform(-1, 1, 64).astype(f32) + 1j * rng.uniform(-1, 1, 64).astype(f32)
    for s, e in enumerate(elems):
        a = TILE + swizzle(e & ~1) * 8
        struct.pack_into("<f", mem, a + 4 * (e & 1), v[s].real)
        struct.pack_into("<f", mem, a + 8 + 4 * (e & 1), v[s].imag)
    struct.pack_into("<6I", mem, SMEM_STATIC + O_PHASE, *[swizzle(1 << b) * 8 for b in regs])
    for k, c in enumerate([G.W_DW, code, 255]):
        struct.pack_into("<Q2f", mem, SMEM_STATIC + O_OPS + 16 * k, (1 << 5) if sel else (1 << 6), 1.0, 0.0)
        mem[SMEM_STATIC + O_CODES + k] = c
    operands = dict(zip(["%%%d" % k for k in range(19)] + ["%tid.x"],
                        [swizzle(e0) * 8, TILE, SMEM_STATIC, O_PHASE, 0, e0, f32(1), f32(0), 0, 0, NEXT, 0, 128,
                         O_CODES, O_OPS - 16, O_UNIT, O_DREG, O_DST, 0, 0]))
    operands.update({"da0": f32(0), "da1": f32(0), "da2": f32(0)})
    th = Thread(G.asm_text("A", True, True), mem, SMEM_STATIC, TILE + (8 << t), operands)
    th.run()
    psi, lam = v[:32].astype(complex), v[32:].astype(complex)
    idx = np.arange(32)
    if code < G.W_DZ:
        j = (code - G.W_DX) % G.AB
        p = psi[idx ^ (1 << j)] * (1 if code < G.W_DY else np.where((idx >> j) & 1, 1j, -1j))
        want = np.vdot(lam, p).imag
    else:
        w = (np.conj(lam) * psi).imag
        if code < G.W_DP:
            want = np.sum(w * np.where((idx >> (code - G.W_DZ)) & 1, -1, 1))
        elif code < G.W_DPP:
            want = np.sum(w[(idx >> (code - G.W_DP)) & 1 == 1]) if sel else 0.0
        elif code < G.W_DW:
            j, k = [(j, k) for j in range(G.AB) for k in range(j + 1, G.AB)][code - G.W_DPP]
            want = np.sum(w[((idx >> j) & (idx >> k) & 1) == 1])
        elif code == G.W_DTZ:
            want = np.sum(w) * (-1 if sel else 1)
        else:
            want = np.sum(w) if sel else 0.0
    assert abs(float(th.r["da0"]) - want) < 64 * 2.0 ** -23 * 2
