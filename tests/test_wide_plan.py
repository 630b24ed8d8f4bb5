"""Which plans the wide pass runs: those the planner made for it, and no
others, whatever register sets they happen to have.  Its shared memory holds
216 records a pass (kMaxWideOps), end codes included; a plan made for the
(re, im) form holds up to 256 ops."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np
import pytest

import paper_1608_00263_gb300 as qs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAX_WIDE_OPS = 216


@pytest.fixture(scope="module")
def probe():
    so = os.path.join(tempfile.mkdtemp(prefix="qs_wide_"), "libprobe.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "wide_plan_probe.cpp"),
                    os.path.join(ROOT, "paper_1608_00263_gb300", "csrc", "qs_host.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.probe_state.argtypes = [ctypes.c_int] * 5 + [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
    lib.probe_batch.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    lib.probe_held.argtypes = [ctypes.c_int] * 4 + [ctypes.c_void_p, ctypes.c_size_t, ctypes.POINTER(ctypes.c_int)]
    lib.probe_oversize.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_size_t]
    lib.probe_sweep.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_size_t]
    return lib


def low_qubit_gates(count, kinds, seed=0, qubits=5):
    """Gates on the lowest qubits only: one pass, every register set with
    qubit 0."""
    rng = np.random.default_rng(seed)
    g = np.zeros(count, dtype=qs.GATE_DTYPE)
    g["kind"] = rng.choice(kinds, size=count)
    for x in g:
        x["q0"], x["q1"] = rng.choice(qubits, size=2, replace=False)
    g["theta"] = rng.uniform(-3, 3, size=count)
    return g


CT = [qs.QS_H, qs.QS_X_HALF, qs.QS_Y_HALF, qs.QS_T, qs.QS_CZ]
DIAG = [qs.QS_T, qs.QS_CZ, qs.QS_RZ, qs.QS_CPHASE]


@pytest.mark.parametrize("kinds", [CT, DIAG, CT + DIAG], ids=["clifford_t", "diagonal", "both"])
@pytest.mark.parametrize("n", [11, 12, 13, 14, 20])
def test_one_state(probe, n, kinds):
    g = low_qubit_gates(250, kinds)
    out = (ctypes.c_int * 5)()
    for mode, tile, narrow in [(qs.QS_MODE_FUSED, 0, 0), (qs.QS_MODE_FUSED, 11, 0), (qs.QS_MODE_FUSED, 0, 1),
                               (qs.QS_MODE_FUSED, 12 if n > 11 else 11, 1), (qs.QS_MODE_FUSED_TC, 0, 0)]:
        assert probe.probe_state(n, qs.QS_C64, mode, tile, narrow, g.ctypes.data, g.size, out) == 0
        regs, wide, passes, records, ops = out
        if mode == qs.QS_MODE_FUSED and not narrow:
            assert wide == regs and passes >= 1 and records <= MAX_WIDE_OPS
        else:
            # the list that must not be lowered: one pass of more ops than
            # the wide pass holds (or tensor-core phases)
            assert regs == 5 and wide == 0 and passes == 0
            assert mode == qs.QS_MODE_FUSED_TC or ops > MAX_WIDE_OPS


@pytest.mark.parametrize("count", [1, 5, 10, 20, 40])
def test_batch(probe, count):
    """An instance without passes (no gates) does not decide for the others:
    plans of five register bits stay in their form, wide ones have six."""
    rng = np.random.default_rng(count)
    sizes = np.array([8, 12], dtype=np.int32)
    regs = ctypes.c_int(0)
    for _ in range(60):
        g = np.zeros(count, dtype=qs.GATE_DTYPE)
        g["kind"] = rng.choice(CT + DIAG + [qs.QS_RX, qs.QS_RY], size=count)
        for x in g:
            x["q0"], x["q1"] = rng.choice(12, size=2, replace=False)
        g["theta"] = rng.uniform(-3, 3, size=count)
        offsets = np.array([0, 0, count], dtype=np.uint64)
        args = (2, sizes.ctypes.data, g.ctypes.data, offsets.ctypes.data)
        assert probe.probe_batch(*args, 0, ctypes.byref(regs)) == 0
    big = np.array([12, 12], dtype=np.int32)
    assert probe.probe_batch(2, big.ctypes.data, g.ctypes.data, offsets.ctypes.data, 1, ctypes.byref(regs)) >= 1
    assert regs.value == 6


@pytest.mark.parametrize("count,status", [(215, 0), (216, 5), (250, 5)])
def test_a_pass_with_too_many_records_is_an_error(probe, count, status):
    """215 ops and the end code are 216 records; more is QS_ERR_UNSUPPORTED
    (status 5), not a write past the table."""
    g = low_qubit_gates(count, [qs.QS_H, qs.QS_X_HALF, qs.QS_Y_HALF])
    assert probe.probe_oversize(12, g.ctypes.data, g.size) == status


ANY = CT + DIAG + [qs.QS_RX, qs.QS_RY]


@pytest.mark.parametrize("kinds", [DIAG, [qs.QS_RZ, qs.QS_CPHASE], [qs.QS_RY, qs.QS_CZ], [qs.QS_RX, qs.QS_RZ], CT, ANY],
                         ids=["diagonal", "phases", "ry_cz", "rx_rz", "clifford_t", "all"])
@pytest.mark.parametrize("n", [10, 12, 13, 20])
def test_records_of_a_reverse_sweep(probe, n, kinds):
    """The planner's count bounds the records of the sweep's passes, which hold
    derivative terms and their sums besides the gates."""
    for count in (1, 60, 400, 900):
        for qubits in (2, 5, n):
            g = low_qubit_gates(count, kinds, seed=count + qubits, qubits=qubits)
            assert 0 < probe.probe_sweep(n, g.ctypes.data, g.size) <= MAX_WIDE_OPS


@pytest.mark.parametrize("n", [12, 20, 21, 22, 23, 24, 25, 26, 27, 28, 30])
def test_short_lists_on_a_state_in_memory(probe, n):
    """A few gates that one pass applies run the (re, im) form at 21 to 25
    qubits, with a parameterised one among them at 26 and 27; everything else is
    planned as before."""
    most = {21: 5, 22: 16, 23: 16, 24: 12, 25: 12, 26: 8, 27: 8}.get(n, 0)
    passes = ctypes.c_int(0)
    wide = 5 if n <= 21 else 6

    def form(g, mode=qs.QS_MODE_FUSED, tile=0, dt=qs.QS_C64):
        return probe.probe_held(n, dt, mode, tile, g.ctypes.data, g.size, ctypes.byref(passes))

    for count in (1, 5, 6, 8, 9, 12, 13, 16, 17, 40):
        for kinds in (CT, DIAG, [qs.QS_RX, qs.QS_RY], [qs.QS_T, qs.QS_CZ]):
            for qubits in (2, n):
                g = low_qubit_gates(count, kinds, seed=count, qubits=qubits)
                low = {0, 1, 2, 3, 4} | {int(x["q0"]) for x in g if x["kind"] not in DIAG}
                param = bool(np.any(g["kind"] >= qs.QS_RX))
                short = len(low) <= 13 and count <= most and (n <= 25 or param)
                assert form(g) == (0 if short else wide), (count, kinds, qubits)
                assert not short or passes.value == 1
                assert form(g, qs.QS_MODE_FUSED_TC) == 0 and form(g, dt=qs.QS_C128) == 0
                assert form(g, tile=12) == (wide if n <= 12 else 5 if n <= 20 else 6)
    # non-diagonal gates on more qubits than a tile: two passes, the wide form
    g = np.zeros(12, dtype=qs.GATE_DTYPE)
    g["kind"], g["q0"] = qs.QS_X_HALF, n - 1 - np.arange(12)
    assert form(g) == wide
