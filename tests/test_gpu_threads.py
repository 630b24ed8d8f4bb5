"""States of different tile sizes in host threads of their own: a launch must
not depend on the shared memory that another thread's launch asked for.  Every
call has to succeed, and every state to end as it does alone."""
import threading

import numpy as np
import pytest

import oracle as O
import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def circuit(n):
    return np.concatenate([O.generate_circuit(1, n, 0, 0)[:n], O.generate_circuit(1, n, 12, 1)[n:]]).astype(qs.GATE_DTYPE)


def evolve(h, n, out):
    g = circuit(n)
    for _ in range(3000):
        qs.qs_state_reset(h)
        qs.qs_apply_circuit(h, g)
    out.append(qs.qs_state_copy_out(h, n, out[0]))


def gradient(h, n, out):
    g = circuit(n)
    g["kind"][-3:], g["theta"][-3:] = qs.QS_RX, 0.3
    x = np.arange(64, dtype=np.uint64)
    for _ in range(400):
        out.append(qs.qs_adjoint_gradient(h, g, x)[1])
    del out[1:-1]


@pytest.mark.parametrize("work,sizes,dt", [(evolve, (11, 12, 13), qs.QS_C64), (evolve, (8, 9, 10), qs.QS_C64),
                                           (evolve, (10, 11, 12), qs.QS_C128), (gradient, (10, 11, 12), qs.QS_C64),
                                           (gradient, (8, 9, 11), qs.QS_C128)],
                         ids=["wide", "narrow", "c128", "gradient", "gradient_c128"])
def test_states_of_several_sizes(work, sizes, dt):
    import torch
    alone, together, failed = {}, {}, []

    def run(n, results):
        try:
            stream = torch.cuda.Stream()
            h = qs.qs_state_create(n, dt, stream=stream.cuda_stream)
            try:
                out = [dt]
                work(h, n, out)
                results[n] = out[1]
            finally:
                qs.qs_state_destroy(h)
        except Exception as e:      # (a thread's exception does not reach the test)
            failed.append((n, e))

    for n in sizes:
        run(n, alone)
    threads = [threading.Thread(target=run, args=(n, together)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for n in sizes:
        assert np.array_equal(alone[n], together[n]), n
