"""Batched independent domains (lwacm_batch_create): per-step launches and the
persistent cooperative launch against the FP64 oracle run domain by domain, and
the bounded grid barrier's timeout path."""
import numpy as np
import pytest

import oracle
from paper_1111_2142_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lw():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def small_ensemble(Q, n, seed):
    rng = np.random.default_rng(seed)
    dims, nus, fields = [], [], []
    for b in range(n):
        if Q == 9:
            d = (int(rng.integers(3, 48)), int(rng.integers(3, 40)))
            shape = (d[1], d[0])
        else:
            d = (int(rng.integers(3, 14)), int(rng.integers(3, 12)), int(rng.integers(2, 10)))
            shape = (d[2], d[1], d[0])
        dims.append(d)
        nus.append(float(rng.uniform(0.002, 0.05)))
        fields.append(inputs.smooth_random(shape, seed=seed * 1000 + b, u_amp=0.04, d_amp=0.01))
    return dims, nus, fields


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("Q", [9, 19])
def test_batch_matches_oracle(lw, Q, mode):
    dims, nus, fields = small_ensemble(Q, 13, seed=61 + Q)
    sim = lw.LwacmBatch(Q, dims, nus, mode=mode)
    sim.set_domains(fields)
    T = 70
    sim.step(T)
    sim.sync()
    got = sim.get_domains()
    worst = 0.0
    for b in range(len(dims)):
        ref = oracle.step(Q, *fields[b], nu=nus[b], nsteps=T)
        eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[b][1:], ref[1:])) / 0.04
        ed = float(np.max(np.abs(got[b][0] - ref[0]))) / max(float(np.max(np.abs(ref[0]))), 3 * 0.04 ** 2)
        worst = max(worst, eu)
        assert eu < 1e-5 and ed < 1e-4, (b, dims[b], eu, ed)
    print(f"[{sim.kernel_name}] Q{Q} 13 domains x{T}: worst du/U = {worst:.2e}")
    sim.close()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("tile", [1, 2, 3, 4, 5, 6])
def test_batch_2d_tiles_match_oracle(lw, tile, mode):
    """D2Q9 ensembles on the 2D-tile kernel (every shape, both launch forms):
    domains smaller and larger than a tile, ragged edges, against the oracle."""
    dims, nus, fields = small_ensemble(9, 11, seed=80 + tile)
    dims[0] = (1, 1)      # one node: every neighbour is itself
    dims[1] = (131, 3)    # wider than every tile, three rows
    fields[0] = inputs.smooth_random((1, 1), seed=5, u_amp=0.04, d_amp=0.01)
    fields[1] = inputs.smooth_random((3, 131), seed=6, u_amp=0.04, d_amp=0.01)
    sim = lw.LwacmBatch(9, dims, nus, mode=mode, tile=tile)
    assert "tiles" in sim.kernel_name
    sim.set_domains(fields)
    T = 40
    sim.step(T)
    got = sim.get_domains()
    for b in range(len(dims)):
        ref = oracle.step(9, *fields[b], nu=nus[b], nsteps=T)
        eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[b][1:], ref[1:])) / 0.04
        ed = float(np.max(np.abs(got[b][0] - ref[0]))) / max(float(np.max(np.abs(ref[0]))), 3 * 0.04 ** 2)
        assert eu < 1e-5 and ed < 1e-4, (tile, mode, b, dims[b], eu, ed)
    sim.close()


def test_tile_shape_switch_mid_run(lw):
    """Changing the tile shape between steps keeps the state and the results."""
    dims, nus, fields = small_ensemble(9, 7, seed=90)
    ref_sim = lw.LwacmBatch(9, dims, nus)
    ref_sim.set_domains(fields)
    sim = lw.LwacmBatch(9, dims, nus, tile=2)
    sim.set_domains(fields)
    for k, shape in enumerate((2, 0, 5, 1)):
        sim.set_option(lw.OPT_BATCH_TILE, shape)
        sim.step(9)
        ref_sim.step(9)
    a, b = sim.get_fields(), ref_sim.get_fields()
    for x, y in zip(a, b):
        assert float(np.max(np.abs(x - y))) < 1e-6
    sim.close()
    ref_sim.close()


def test_persistent_equals_per_step(lw):
    dims, nus, fields = small_ensemble(9, 9, seed=70)
    out = []
    for mode in (0, 1):
        sim = lw.LwacmBatch(9, dims, nus, mode=mode)
        sim.set_domains(fields)
        sim.step(33)
        sim.step(4)
        out.append(sim.get_fields())
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_barrier_timeout_is_reported(lw):
    """A CTA that never arrives (test hook) makes the others' bounded waits run out:
    the launch ends, the error word is set and lwacm_sync reports LWACM_E_TIMEOUT."""
    import time
    dims, nus, fields = small_ensemble(9, 40, seed=71)
    dims = [(max(d[0], 40), max(d[1], 40)) for d in dims]  # enough tiles for several CTAs
    fields = [inputs.smooth_random((d[1], d[0]), seed=k) for k, d in enumerate(dims)]
    sim = lw.LwacmBatch(9, dims, nus, mode=1)
    sim.set_domains(fields)
    sim.set_option(lw.OPT_TEST_WITHHOLD, 3)
    t0 = time.time()
    sim.step(10)
    with pytest.raises(lw.LwacmError) as ei:
        sim.sync()
    assert ei.value.status == lw.E_TIMEOUT
    assert time.time() - t0 < 30
    sim.close()
    # the device is still usable afterwards
    ok = lw.LwacmBatch(9, dims[:3], nus[:3], mode=1)
    ok.set_domains(fields[:3])
    ok.step(5)
    ok.sync()
    ok.close()


def test_ensemble_256(lw):
    """The batched workload: 256 periodic D2Q9 domains, sides log-uniform on
    [32, 512] (seed 1), nu uniform on [0.002, 0.05], band-limited divergence-free
    initial velocity (wave numbers 1-4, rms U = 0.02), 2000 steps in one
    persistent launch.

    * after 2000 steps: every one of the 256 domains, stepped once more from the
      GPU's state by GPU and oracle, agrees to 1e-6 U (one step of FP32 rounding);
    * the runs themselves drift apart: the per-step FP32 rounding is carried
      forward by the nonlinear flow (domain Reynolds numbers up to ~500), about
      linearly in T: measured on the worst of six sampled domains (the five
      smallest and a mid-size one) 1.04e-5 U at 200, 4.6e-5 U at 1000 and
      1.1e-4 U at 2000 steps, i.e. ~5.5e-8 U per step. Bound: 1.25e-7 U per step
      (2.5e-5 U at 200 steps, 2.5e-4 U at 2000).
    """
    U = 0.02
    drift_per_step = 1.25e-7
    doms = inputs.ensemble_2d(256, seed=1)
    dims = [(d["nx"], d["ny"]) for d in doms]
    nus = [d["nu"] for d in doms]
    fields = [(d["d"], d["ux"], d["uy"]) for d in doms]
    sizes = [d[0] * d[1] for d in dims]
    order = np.argsort(sizes)
    check = [int(b) for b in order[:5]] + [int(order[len(order) // 2])]
    sim = lw.LwacmBatch(9, dims, nus, mode=1)
    sim.set_domains(fields)
    sim.step(200)
    got = sim.get_domains()
    for b in check:
        ref = oracle.step(9, *fields[b], nu=nus[b], nsteps=200)
        eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[b][1:], ref[1:])) / U
        assert eu < drift_per_step * 200, (b, dims[b], eu)
    sim.step(1800)
    sim.sync()
    assert sim.diagnostics()["finite"]
    got = sim.get_domains()
    long_err = 0.0
    for b in check:
        ref = oracle.step(9, *fields[b], nu=nus[b], nsteps=2000)
        long_err = max(long_err, max(float(np.max(np.abs(g - r))) for g, r in zip(got[b][1:], ref[1:])) / U)
    sim.step(1)
    one = sim.get_domains()
    worst1 = 0.0
    for b in range(256):
        ref1 = oracle.step(9, *got[b], nu=nus[b], nsteps=1)
        worst1 = max(worst1, max(float(np.max(np.abs(g - r))) for g, r in zip(one[b][1:], ref1[1:])) / U)
    print(f"ensemble: {sim.n_nodes} nodes in 256 domains; 2000 steps: sampled drift {long_err:.2e} U; "
          f"one step from the GPU state, all domains: {worst1:.2e} U")
    assert worst1 < 1e-6
    assert long_err < drift_per_step * 2000
    sim.close()


# ensembles each side of the line between strips and 1D runs (10 nodes a strip's row, small ones
# on strips): narrow and wide domains, mixtures
@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("dims,rows", [([(1, 3000), (2, 2300), (3, 7)], False), ([(7, 4000)] * 6, False), ([(9, 1950), (8, 1721)], True),
                                       ([(22, 64), (31, 9)], True), ([(1, 40), (2, 90), (3, 33)], True),
                                       ([(60, 41), (2, 90), (90, 33)], True), ([(60, 200)] + [(3, 800)] * 9, False)])
def test_narrow_ensembles(lw, dims, rows, storage):
    """The kernel by name in both launch forms of one context, and every domain's fields (FP32
    against the oracle; BF16 one step, within half a storage ulp and FP32 rounding)."""
    nus = [0.01 + 0.002 * b for b in range(len(dims))]
    fields = [inputs.smooth_random((h, w), seed=900 + b, u_amp=0.04, d_amp=0.01) for b, (w, h) in enumerate(dims)]
    sim = lw.LwacmBatch(9, dims, nus, storage=storage)
    if storage:  # the state as stored
        sim.set_domains(fields)
        fields = [tuple(np.asarray(a, dtype=np.float64) for a in d) for d in sim.get_domains()]
    T = 1 if storage else 7
    last = None
    for mode in (0, 1, 0):
        sim.set_option(lw.OPT_BATCH_MODE, mode)
        name = ("batch_rows_" if rows else "batch_") + ("persistent" if mode else "step")
        assert sim.kernel_name == name
        sim.set_domains(fields)
        sim.step(T)
        all_ = sim.get_domains()
        assert last is None or all(np.array_equal(a, b) for x, y in zip(all_, last) for a, b in zip(x, y))
        last = all_  # both launch forms, bit for bit
        for f, nu, got in zip(fields, nus, all_):
            ref = oracle.step(9, *f, nu=nu, nsteps=T)
            for g, r in zip(got, ref):
                tol = 1.05 * 2.0 ** -8 * np.abs(r) + 8 * 2.0 ** -24 * 0.04 if storage else 4e-7
                assert np.all(np.abs(g - r) <= tol)
    sim.close()


def test_a_graph_of_one_launch_form_outlives_a_change_to_the_other(lw):
    """Steps captured with a launch a step replay the same after the context has run the one-launch
    form, whose strips are cut otherwise."""
    import torch
    dims, nus = [(10, 200)] * 20 + [(70, 31)], [0.01 + 0.001 * b for b in range(21)]
    fields = [inputs.smooth_random((h, w), seed=950 + b, u_amp=0.04, d_amp=0.01) for b, (w, h) in enumerate(dims)]
    sim = lw.LwacmBatch(9, dims, nus, graph_chunk=0, stream=torch.cuda.Stream())
    assert sim.kernel_name == "batch_rows_step"
    sim.set_domains(fields)
    sim.step(2)
    want = sim.get_domains()
    sim.set_domains(fields)
    sim.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=sim.stream):
        sim.step(2)
    sim.set_option(lw.OPT_BATCH_MODE, 1)
    sim.set_domains(fields)
    sim.step(2)
    assert all(np.array_equal(a, b) for x, y in zip(sim.get_domains(), want) for a, b in zip(x, y))
    sim.set_domains(fields)
    with torch.cuda.stream(sim.stream):
        g.replay()
    sim.sync()
    assert all(np.array_equal(a, b) for x, y in zip(sim.get_domains(), want) for a, b in zip(x, y))
    sim.close()
