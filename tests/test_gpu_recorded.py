"""Recorded runs (lwacm_forward_record) beside plain steps of the same context: they run kernels
of their own (the half-row kernel, the 2D tiles, the gather) and keep graphs of their own."""
import ctypes

import numpy as np
import pytest

import oracle
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


# (lattice, shape, boundary, force, option that selects the same kernel for plain steps: None where
# there is none, the gather)
RUNS = [(19, (9, 11, 13), 0, False, None), (19, (5, 7, 33), 1, False, None), (19, (6, 9, 31), 2, True, None),
        (19, (24, 20, 4), 0, True, None), (19, (3, 3, 40), 0, False, ("KERNEL", 1)), (19, (4, 16, 256), 0, False, ("KERNEL", 5)),
        (19, (5, 12, 200), 0, True, ("KERNEL", 5)), (19, (6, 16, 128), 1, False, ("KERNEL", 5)),
        (19, (4, 9, 128), 2, True, ("KERNEL", 5)), (9, (37, 41), 0, True, ("BATCH_TILE", 2)),
        (9, (64, 64), 1, False, ("BATCH_TILE", 2)), (9, (33, 70), 2, True, ("BATCH_TILE", 2))]


@pytest.mark.parametrize("Q,shape,bc,forced,option", RUNS)
def test_fields_of_a_recorded_run(lw, Q, shape, bc, forced, option):
    """The state after a recorded run against the oracle, against plain steps of the same kernel bit
    for bit, and against plain steps of the automatic choice, whose order of additions may differ:
    both within rounding of the oracle (1e-5 of the velocity, 1e-4 of the density deviation)."""
    T, nz = 21, shape[0] if Q == 19 else 1
    f = inputs.smooth_random(shape, seed=93, u_amp=0.04, d_amp=0.01)
    force = ((1e-4, -2e-5, 3e-5) if Q == 19 else (1e-4, -2e-5)) if forced else None
    lid = ((0.03, 0.02, 0.0) if Q == 19 else (0.03, 0.0)) if bc else None

    def new():
        sim = lw.Lwacm(Q, shape[-1], shape[-2], nz, 0.02, bc, force=force, lid=lid)
        sim.set_fields(*f)
        return sim

    three = lambda v: None if v is None else tuple(v) + (0.0,) * (3 - len(v))  # noqa: E731
    ref = oracle.step(Q, *f, nu=0.02, bc=bc, nsteps=T, force=three(force), lid=three(lid))
    fields = []
    for how in ("recorded", "plain", "pinned"):
        sim = new()
        if how == "recorded":
            sim.forward_record(T, 4)
        elif how == "pinned" and option is None:
            continue
        else:
            if how == "pinned":
                sim.set_option(getattr(lw, "OPT_" + option[0]), option[1])
            sim.step(T)
        assert sim.step_count() == T
        got = sim.get_fields()
        fields.append(got)
        eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[1:], ref[1:])) / 0.04
        ed = float(np.max(np.abs(got[0] - ref[0]))) / max(float(np.max(np.abs(ref[0]))), 3 * 0.04 ** 2)
        assert eu < 1e-5 and ed < 1e-4, how
        sim.close()
    if option is not None:
        assert all(np.array_equal(a, b) for a, b in zip(fields[0], fields[2]))
