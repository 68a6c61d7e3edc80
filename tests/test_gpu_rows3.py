"""The D3Q19 kernel of warps that march along z (kernels_rows3.cu): edges of its 30-column
strips, four-row tiles and runs of planes, and forcing, against the FP64 oracle and the
gather kernel (the 16-bit storage types run on it in test_gpu_parity.py)."""
import numpy as np
import pytest

import oracle
from paper_1111_2142_gb300 import inputs

pytestmark = pytest.mark.gpu

# (nz, ny, nx): one plane, one column, the edges of a strip, a tile and a CTA's four tiles,
# tiles that overlap (ny % 4 != 0), runs of several planes
SHAPES = [(1, 4, 1), (2, 5, 29), (3, 6, 30), (1, 7, 31), (4, 4, 59), (3, 16, 60), (2, 17, 61), (5, 15, 33), (40, 9, 7),
          (3, 130, 91), (61, 66, 70)]


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def run(lw, shape, f, T, g=None, nu_p=None, bc=0, **kw):
    nz, ny, nx = shape
    sim = lw.Lwacm(19, nx, ny, nz, 0.02, bc, force_field=g is not None, kernel=1, **kw)
    if nu_p:
        sim.set_option(lw.OPT_NU_P, nu_p)
    sim.set_fields(*f)
    if g is not None:
        sim.set_force_field(*g)
    sim.step(T)
    got = sim.get_fields()
    sim.close()
    return got


def within(got, ref, U=0.05):
    eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[1:], ref[1:])) / U
    ed = float(np.max(np.abs(got[0] - ref[0]))) / max(float(np.max(np.abs(ref[0]))), 3 * U * U)
    assert eu < 1e-5 and ed < 1e-4, (eu, ed)


@pytest.mark.parametrize("shape", SHAPES)
def test_march_matches_oracle(lw, shape):
    f = inputs.smooth_random(shape, seed=51, u_amp=0.05, d_amp=0.01)
    within(run(lw, shape, f, 9), oracle.step(19, *f, nu=0.02, nsteps=9))


# walls in the kernel: two nodes an axis, strips and tiles that are at both walls, at one, at
# none, tiles that overlap at the wall, several runs of planes
@pytest.mark.parametrize("bc", [1, 2])
@pytest.mark.parametrize("shape", [(2, 4, 2), (2, 5, 3), (3, 6, 29), (4, 7, 30), (5, 9, 31), (3, 8, 61), (6, 33, 95), (61, 66, 70)])
def test_march_with_walls(lw, shape, bc):
    """A cavity whose lid moves along all three axes' directions in the top z plane, and a
    forced channel with a moving wall."""
    f = inputs.smooth_random(shape, seed=56, u_amp=0.05, d_amp=0.01)
    lid, force = (0.05, -0.03, 0.01), (1e-5, 0.0, 2e-5) if bc == 2 else None
    got = run(lw, shape, f, 12, bc=bc, lid=lid, force=force)
    within(got, oracle.step(19, *f, nu=0.02, nsteps=12, bc=bc, lid=lid, force=force))


@pytest.mark.parametrize("shape", [(1, 4, 1), (2, 17, 61), (5, 15, 33)])
def test_march_with_forcing(lw, shape):
    """A constant acceleration, and a per-node field on top of it."""
    f = inputs.smooth_random(shape, seed=52, u_amp=0.05, d_amp=0.01)
    g0 = (1e-4, -2e-5, 3e-5)
    g = [1e-4 * c for c in inputs.smooth_random(shape, seed=53, u_amp=1.0, d_amp=1.0)[1:4]]
    within(run(lw, shape, f, 4, force=g0), oracle.step(19, *f, nu=0.02, nsteps=4, force=g0))
    both = [a + b for a, b in zip(g, g0)]
    within(run(lw, shape, f, 4, force=g0, g=g), oracle.step_force_field(19, *f, nu=0.02, g=both, nsteps=4))


@pytest.mark.parametrize("bad", [np.inf, np.nan, 3e38, -1.0])
@pytest.mark.parametrize("field", [0, 3])
def test_march_carries_extreme_values(lw, field, bad):
    """A node that has blown up (or whose density is zero) spreads as in the gather kernel
    (which an omega_p a part in 10^12 from omega selects): the same infinities and NaNs."""
    import torch
    f = [a.astype(np.float32) for a in inputs.smooth_random((9, 11, 40), seed=55, u_amp=0.05, d_amp=0.01)]
    f[field][4, 5, 30] = bad
    t = [torch.from_numpy(a).cuda() for a in f]
    a, b = run(lw, (9, 11, 40), t, 2), run(lw, (9, 11, 40), t, 2, nu_p=0.02 * (1 + 1e-12))
    for x, y in zip(a, b):
        assert np.array_equal(np.isfinite(x), np.isfinite(y))
        ok = np.isfinite(y) & (np.abs(y) < 1e3)
        assert np.allclose(x[ok], y[ok], rtol=0, atol=1e-3)


# narrow domains of many nodes, each side of the line between the gather and the march (with the
# scalar, in a channel, a force field): the kernel and its fields
@pytest.mark.parametrize("shape,kw,name", [
    ((256, 256, 2), {}, "generic_d3q19"), ((256, 256, 4), {}, "generic_d3q19"), ((256, 256, 6), {}, "generic_d3q19_march"),
    ((10000, 6, 6), {}, "generic_d3q19"), ((10000, 6, 15), {}, "generic_d3q19_march"),
    ((64, 64, 1), {}, "generic_d3q19_march"), ((256, 256, 3), dict(bc=2), "generic_d3q19"),
    ((256, 256, 5), dict(bc=2), "generic_d3q19_march"), ((256, 256, 3), dict(bc=1), "generic_d3q19"),
    ((1000, 6, 6), dict(bc=1), "generic_d3q19_march"),
    ((256, 256, 4), dict(g=True), "generic_d3q19"), ((256, 256, 5), dict(scalar=True), "generic_d3q19"),
    ((256, 256, 10), dict(scalar=True), "generic_d3q19_march+scalar_march"),
    ((1000, 16, 4), dict(scalar=True), "generic_d3q19"), ((24, 24, 4), dict(scalar=True), "generic_d3q19_march+scalar_march")])
def test_narrow_domains(lw, shape, kw, name):
    nz, ny, nx = shape
    f = inputs.smooth_random(shape, seed=57, u_amp=0.05, d_amp=0.01)
    bc, lid = kw.get("bc", 0), (0.05, -0.03, 0.01) if kw.get("bc") else None
    g = [1e-4 * c for c in inputs.smooth_random(shape, seed=58, u_amp=1.0, d_amp=1.0)[1:4]] if kw.get("g") else None
    sim = lw.Lwacm(19, nx, ny, nz, 0.02, bc, lid=lid, force_field=g is not None, scalar_alpha=0.03 if kw.get("scalar") else None)
    sim.set_fields(*f)
    if g is not None:
        sim.set_force_field(*g)
    T0 = 1.0 + 0.2 * f[0] / float(np.max(np.abs(f[0])))
    if kw.get("scalar"):
        sim.set_scalar(T0)
    assert sim.kernel_name == name
    sim.step(3)
    got = sim.get_fields()
    if kw.get("scalar"):
        ref = oracle.step_scalar(19, *f, T=T0, nu=0.02, alpha=0.03, nsteps=3)
        assert float(np.max(np.abs(sim.get_scalar() - ref[-1]))) < 2e-6
        ref = ref[:-1]
    elif g is not None:
        ref = oracle.step_force_field(19, *f, nu=0.02, g=g, nsteps=3)
    else:
        ref = oracle.step(19, *f, nu=0.02, nsteps=3, bc=bc, lid=lid)
    within(got, ref)
    sim.close()
