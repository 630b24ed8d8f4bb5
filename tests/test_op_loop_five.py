"""The wide pass's phase with five register bits (states of few tiles run it),
by the interpreter and with the definitions of test_op_loop.py: 32 amplitudes
per thread, every byte code of the loop, stores to the tile and to the state.

Tolerance as there: at most 12 ops of six FP32 roundings each and a factor,
9e-6 absolute on values that butterflies have grown."""
import math
import struct

import numpy as np
import pytest

from test_op_loop import (G, NEXT, O_CODES, O_DREG, O_DST, O_OPS, O_PHASE, O_UNIT, SMEM_STATIC, STATE, TILE, Thread,
                          expected, f32, swizzle)

NS, NU = 32, 16


def loop(full):
    """The five-bit loop's text and the codes it holds."""
    G.set_register_bits(5)
    try:
        return G.asm_text("V", full), [c for c, b in enumerate(G.cases(full)) if b]
    finally:
        G.set_register_bits(G.CRB)


@pytest.mark.parametrize("full", [False, True])
def test_codes(full):
    """Every code that does not name register bit 5."""
    five = [c for k in range(4) for c in range(k * G.CRB, k * G.CRB + 5)]
    pairs = [G.pair_index(j, k) for j in range(5) for k in range(j + 1, 5)]
    five += [G.W_CZ + p for p in pairs] + [G.W_CZO + j for j in range(5)]
    if full:
        five += [base + j for base in (G.W_RY, G.W_RX, G.W_PH) for j in range(5)] + [G.W_PP + p for p in pairs]
    assert sorted(loop(full)[1]) == sorted(five)


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("t,regs", [(13, (0, 1, 2, 3, 4)), (13, (0, 8, 9, 11, 12)), (11, (0, 3, 5, 7, 10)),
                                    (12, (0, 6, 7, 8, 11))])
def test_phase_on_one_thread(full, t, regs):
    rng = np.random.default_rng(50 + t + 100 * full)
    lines, codes_held = loop(full)
    others = [b for b in range(t) if b not in regs]
    order = rng.permutation(codes_held)
    qbit = [8 << (2 * b) for b in range(t)]         # tile bit b is qubit 2 b
    deposit = lambda e: sum(qbit[b] for b in range(t) if (e >> b) & 1)
    for start in range(0, len(order), 12):
        codes = [int(c) for c in order[start:start + 12]]
        tid = int(rng.integers(0, 1 << len(others)))
        e0 = sum(((tid >> k) & 1) << b for k, b in enumerate(others))
        mem = bytearray(TILE + (8 << t))
        tile = rng.uniform(-1, 1, (1 << t, 2)).astype(f32)
        for u in range(1 << (t - 1)):
            struct.pack_into("<4f", mem, TILE + swizzle(2 * u) * 8, tile[2 * u, 0], tile[2 * u + 1, 0],
                             tile[2 * u, 1], tile[2 * u + 1, 1])
        struct.pack_into("<5I", mem, SMEM_STATIC + O_PHASE, *[swizzle(1 << b) * 8 for b in regs])
        tau, ops, first = 21, [], 5
        for k, c in enumerate(codes):
            want = (tau << 32 | e0) & ~1 if rng.integers(0, 2) else 1 << 33 | (tau << 32)
            sel = ((tau << 32 | e0) & want) == want
            p = (math.cos(0.3 + k), math.sin(0.3 + k))
            struct.pack_into("<Q2f", mem, SMEM_STATIC + O_OPS + 16 * (first + k), want, *p)
            mem[SMEM_STATIC + O_CODES + first + k] = c
            ops.append((c, p[0], p[1], sel))
        mem[SMEM_STATIC + O_CODES + first + len(codes)] = 255
        nthr = 1 << len(others)
        units = [(deposit(2 * nthr * k), swizzle(2 * nthr * k) * 8) for k in range(NU)]
        for k, (goff, soff) in enumerate(units):
            struct.pack_into("<2Q", mem, SMEM_STATIC + O_UNIT + 16 * k, goff, soff)
        struct.pack_into("<5Q", mem, SMEM_STATIC + O_DREG, *[qbit[b] for b in regs])
        struct.pack_into("<Q", mem, SMEM_STATIC + O_DST + 8 * tid, STATE + deposit(e0))
        swt = swizzle(2 * tid) * 8
        elems = [e0 | sum(((s >> j) & 1) << b for j, b in enumerate(regs)) for s in range(NS)]
        # (the definitions hold 64 amplitudes; no op here names bit 5)
        v64 = np.zeros(64, complex)
        v64[:NS] = tile[elems, 0].astype(complex) + 1j * tile[elems, 1]
        v32 = expected(v64, t, ops, None)[:NS]
        for mode, fac in ((0, 1.0), (1, -0.25), (2, 0.6 + 0.8j), (1 | G.F_DIRECT, 0.5), (2 | G.F_DIRECT | G.F_MORE, 1j),
                          (1 | G.F_DIRECT | G.F_CANON, 2.0)):
            m2, fac = bytearray(mem), complex(fac)
            operands = dict(zip(["%%%d" % k for k in range(18)] + ["%tid.x"],
                                [swizzle(e0) * 8, TILE, SMEM_STATIC, O_PHASE, first, tau << 32 | e0,
                                 f32(fac.real), f32(fac.imag), mode, swt, NEXT, 0, nthr, O_CODES, O_OPS - 16, O_UNIT,
                                 O_DREG, O_DST, tid]))
            th = Thread(lines, m2, SMEM_STATIC, TILE + (8 << t), operands)
            th.run()
            assert th.copies == ([(TILE + (soff ^ swt), NEXT + goff) for goff, soff in units] if mode & G.F_MORE else [])
            v, got = v32 * fac, np.empty(NS, complex)
            for s, e in enumerate(elems):
                if mode & G.F_DIRECT:
                    q = th.stores[STATE + deposit(e & ~1)]
                    got[s] = complex(*(q[2 * (e & 1):][:2] if mode & G.F_CANON else (q[e & 1], q[2 + (e & 1)])))
                else:
                    q = struct.unpack_from("<4f", m2, TILE + swizzle(e & ~1) * 8)
                    got[s] = complex(q[e & 1], q[2 + (e & 1)])
            assert np.max(np.abs(got - v)) < 9e-6 * (np.max(np.abs(v)) + 1.0), (full, t, regs, codes, mode)
            if mode & G.F_DIRECT:
                assert len(th.stores) == NU and m2 == mem
                continue
            assert not th.stores
            mine = {TILE + swizzle(e & ~1) * 8 for e in elems}
            for u in range(1 << (t - 1)):
                a = TILE + swizzle(2 * u) * 8
                if a not in mine:
                    assert m2[a:a + 16] == mem[a:a + 16]
