"""Recorded runs (lwacm_forward_record) beside plain steps of the same context: they run kernels
of their own (the half-row kernel, the 2D tiles, the gather) and keep graphs of their own."""
import ctypes

import numpy as np
import pytest

from paper_1111_2142_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def builds(sim):
    n = ctypes.c_longlong()
    assert sim._lib.lwacm_selftest_graph_builds(sim._h, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("Q,shape", [(9, (200, 300)), (19, (6, 10, 12)), (19, (4, 16, 256))])
def test_graphs_of_plain_and_recorded_steps_live_side_by_side(lw, Q, shape):
    """Segments as long as a graph: an optimisation loop that alternates recorded runs and plain
    steps captures each graph once, and both give what they give alone."""
    import torch
    nz = shape[0] if Q == 19 else 1
    f = inputs.smooth_random(shape, seed=91, u_amp=0.03, d_amp=0.005)
    lam = [torch.from_numpy(a).cuda() for a in inputs.smooth_random(shape, seed=92, u_amp=1.0, d_amp=1.0)]

    def new():
        sim = lw.Lwacm(Q, shape[-1], shape[-2], nz, 0.02, graph_chunk=8)
        sim.set_fields(*f)
        return sim

    sim = new()
    sim.prepare(16)
    assert builds(sim) == 1
    seen = []
    for _ in range(3):
        sim.set_fields(*f)
        sim.forward_record(32, 16)
        recorded = sim.get_fields()
        g, gnu = sim.backward(lam)
        sim.set_fields(*f)
        sim.step(16)
        seen.append((builds(sim), recorded, [t.cpu().numpy() for t in g], gnu, sim.get_fields()))
    assert [s[0] for s in seen] == [2, 2, 2]
    alone, plain = new(), new()
    alone.forward_record(32, 16)
    recorded = alone.get_fields()
    g, gnu = alone.backward(lam)
    for _ in range(16):
        plain.step(1)
    for s in seen:
        assert all(np.array_equal(a, b) for a, b in zip(s[1], recorded))
        assert all(np.array_equal(a, b.cpu().numpy()) for a, b in zip(s[2], g)) and s[3] == gnu
        assert all(np.array_equal(a, b) for a, b in zip(s[4], plain.get_fields()))
    for s in (sim, alone, plain):
        s.close()
