"""The D2Q9 kernel of warps that march along y (kernels_rows2.cu, the automatic choice for
one domain): edges of its 30-column strips, of its runs of rows and of both its forms (one
and two strips a warp), every variant, against the FP64 oracle and the 2D-tile kernel."""
import numpy as np
import pytest

import oracle
from paper_1111_2142_gb300 import inputs

pytestmark = pytest.mark.gpu

# one strip a warp: 1 .. 3 columns, a strip's edges, ragged; the last two take two strips a
# warp (more than five rows an item)
SHAPES = [(1, 1), (5, 1), (1, 9), (2, 2), (3, 29), (4, 30), (5, 31), (7, 59), (6, 60), (9, 61), (40, 91), (1210, 839),
          (2051, 602)]


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def run(lw, shape, f, T, bc=0, tile=0, nu_p=None, g=None, **kw):
    ny, nx = shape
    sim = lw.Lwacm(9, nx, ny, 1, 0.02, bc, force_field=g is not None, **kw)
    if nu_p:
        sim.set_option(lw.OPT_NU_P, nu_p)
    sim.set_option(lw.OPT_BATCH_TILE, tile)
    assert sim.kernel_name.startswith("tiles2d_d2q9_rows" if tile == 0 else "tiles2d_d2q9_30x14")
    sim.set_fields(*f)
    if g is not None:
        sim.set_force_field(*g)
    sim.step(T)
    got = list(sim.get_fields())
    if kw.get("bulk_gamma"):
        got.append(sim.get_trace())
    sim.close()
    return got


def within(got, ref, U=0.05):
    eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[1:3], ref[1:3])) / U
    ed = float(np.max(np.abs(got[0] - ref[0]))) / max(float(np.max(np.abs(ref[0]))), 3 * U * U)
    assert eu < 1e-5 and ed < 1e-4, (eu, ed)


@pytest.mark.parametrize("bc", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_rows_kernel_matches_oracle(lw, shape, bc):
    """Plain scheme, periodic, cavity and channel with a moving wall, the channel forced."""
    if (bc == 1 and min(shape) < 2) or (bc == 2 and shape[0] < 2):
        pytest.skip("walled axes need two nodes")
    f = inputs.smooth_random(shape, seed=21, u_amp=0.05, d_amp=0.01)
    lid = (0.05, 0.01) if bc else None
    force = (1e-4, -2e-5) if bc == 2 else None
    T = 15 if shape[0] < 1000 else 3
    got = run(lw, shape, f, T, bc, lid=lid, force=force)
    ref = oracle.step(9, *f, nu=0.02, bc=bc, nsteps=T, lid=None if lid is None else lid + (0.0,),
                      force=None if force is None else force + (0.0,))
    within(got, ref)


@pytest.mark.parametrize("shape", [(1, 1), (4, 30), (9, 61), (2051, 602)])
def test_rows_kernel_variants(lw, shape):
    """A per-node force field and omega_p against the oracle."""
    f = inputs.smooth_random(shape, seed=22, u_amp=0.05, d_amp=0.01)
    g = [1e-4 * c for c in inputs.smooth_random(shape, seed=23, u_amp=1.0, d_amp=1.0)[1:3]]
    within(run(lw, shape, f, 4, g=g), oracle.step_force_field(9, *f, nu=0.02, g=g, nsteps=4))
    within(run(lw, shape, f, 4, nu_p=0.1), oracle.step_nu_p(9, *f, nu=0.02, nu_p=0.1, nsteps=4))


@pytest.mark.parametrize("nu_p", [None, 0.1])
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 1), (3, 29), (5, 31), (40, 91), (2051, 602)])
def test_bulk_variant_equals_the_tile_kernel(lw, shape, storage, nu_p):
    """The bulk-viscosity variant adds a node's values in the tile kernel's order: the same
    fields and trace bit for bit."""
    f = inputs.smooth_random(shape, seed=24, u_amp=0.05, d_amp=0.01)
    a, b = (run(lw, shape, f, 4, tile=t, nu_p=nu_p, storage=storage, bulk_gamma=0.4) for t in (0, 2))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("bad", [np.inf, np.nan, 3e38, -1.0])
@pytest.mark.parametrize("field", [0, 1])
def test_rows_kernel_carries_extreme_values(lw, field, bad):
    """A node that has blown up (or whose density is zero) spreads as in the tile kernel:
    the same infinities and NaNs."""
    f = [a.astype(np.float32) for a in inputs.smooth_random((40, 91), seed=25, u_amp=0.05, d_amp=0.01)]
    f[field][17, 30] = bad
    import torch
    t = [torch.from_numpy(a).cuda() for a in f]
    a, b = (run(lw, (40, 91), t, 2, tile=k) for k in (0, 2))
    for x, y in zip(a, b):
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.array_equal(np.isinf(x), np.isinf(y))
        ok = np.isfinite(y) & (np.abs(y) < 1e3)
        assert np.allclose(x[ok], y[ok], rtol=0, atol=1e-3)


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("scale", [1, 12])
def test_ensemble_strips_equal_single_domains(lw, storage, scale):
    """An ensemble's strips give each domain the fields it has alone, bit for bit, in both
    launch forms: a node's sums do not depend on how its domain is cut (scale 12: two strips
    a warp)."""
    dims = [(1, 1), (29, 3), (31, 7), (60, 5), (61, 2), (120, 40), (3, 90), (97, 61)]
    dims = [(w * (scale if w > 60 else 1), h * (scale if w > 60 else 1)) for w, h in dims]
    nus = [0.01 + 0.01 * b for b in range(len(dims))]
    fields = [inputs.smooth_random((h, w), seed=30 + b, u_amp=0.04, d_amp=0.01) for b, (w, h) in enumerate(dims)]
    for mode in (0, 1):
        sim = lw.LwacmBatch(9, dims, nus, mode=mode, storage=storage)
        sim.set_domains(fields)
        sim.step(7)
        got = sim.get_domains()
        sim.close()
        for (w, h), nu, f, g in zip(dims, nus, fields, got):
            one = lw.Lwacm(9, w, h, 1, nu, storage=storage)
            one.set_fields(*f)
            one.step(7)
            for x, y in zip(g, one.get_fields()):
                assert np.array_equal(x, y), (mode, w, h)
            one.close()


# more rows than the GPU holds warps at once, five and more rows an item: up to 30 columns on one
# strip a warp, up to 60 on two; both edges
@pytest.mark.parametrize("shape", [(30011, 1), (30011, 29), (26003, 30), (30011, 31), (25013, 60), (25013, 61)])
def test_tall_narrow_domains(lw, shape):
    """The plain scheme and a cavity against the oracle, the bulk variant against the tile kernel."""
    f = inputs.smooth_random(shape, seed=26, u_amp=0.05, d_amp=0.01)
    within(run(lw, shape, f, 3), oracle.step(9, *f, nu=0.02, nsteps=3))
    if shape[1] > 1:
        within(run(lw, shape, f, 3, 1, lid=(0.05, 0.01)),
               oracle.step(9, *f, nu=0.02, bc=1, nsteps=3, lid=(0.05, 0.01, 0.0)))
    a, b = (run(lw, shape, f, 3, tile=t, bulk_gamma=0.4) for t in (0, 2))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
