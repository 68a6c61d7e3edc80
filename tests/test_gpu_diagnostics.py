"""lwacm_diagnostics on both of its paths (FP64 node by node below 2^18 nodes, exact FP32
expansions from there) against extended-precision sums."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# 2^18 - 1 nodes (the FP64 path), 2^18 and just above (the expansions; node counts that are
# and are not multiples of four, two and three dimensions)
SHAPES = [(63, 73, 57), (64, 64, 64), (61, 71, 67), (513, 515)]


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def diagnose(lw, f, storage=0):
    shape = f[0].shape
    Q = 9 if len(shape) == 2 else 19
    sim = lw.Lwacm(Q, shape[-1], shape[-2], shape[0] if Q == 19 else 1, 0.02, storage=storage)
    sim.set_fields(*f)
    got = sim.diagnostics()
    stored = sim.get_fields()  # FP64 copies of what is stored
    sim.close()
    return got, stored


def sums(f):
    """The same quantities with every product and sum in extended precision (63 bits here
    and more elsewhere), and the sum of magnitudes each is measured against."""
    L = np.longdouble
    d, u, v = [a.astype(L) for a in f[:3]]
    w = f[3].astype(L) if len(f) > 3 else 0 * u
    rho, uu = 1 + d, u * u + v * v + w * w
    z = len(f) > 3
    terms = dict(mass=d, jx=rho * u, jy=rho * v, jz=rho * w, ke=rho * uu / 2,
                 mpar=(u + v) ** 2 / 2 if z else 0 * u, mperp=(u - v) ** 2 / 2 if z else 0 * u)
    ref = {k: (t.sum(), np.abs(t).sum()) for k, t in terms.items()}
    ref["umax"] = (np.sqrt(uu.max()), np.sqrt(uu.max()))
    return ref


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("scale", [1.0, 1e-13])
@pytest.mark.parametrize("shape", SHAPES)
def test_diagnostics_to_fp64_rounding(lw, shape, scale, storage):
    """Every quantity within 64 FP64 roundings of its terms' magnitude (each of some 300
    blocks' sums of 256 threads' sums is a chain of at most 8 + 8 additions after a thread's
    own, and FP64 throughout adds 4); velocities of 1e-13 take the FP64 path of a thread."""
    rng = np.random.default_rng(61)
    s = scale if storage != 2 else 1.0  # FP16 has no 1e-13
    f = [(rng.normal(size=shape) * a * b).astype(np.float32) for a, b in zip((1e-2, 3e-2, 3e-2, 3e-2), (1, s, s, s))]
    f = f[:len(shape) + 1]
    got, stored = diagnose(lw, [a.astype(np.float64) for a in f], storage)
    for k, (x, mag) in sums(stored).items():
        assert abs(np.longdouble(got[k]) - x) <= 64 * 2.0 ** -53 * mag, (k, got[k], x)
    assert got["finite"]


@pytest.mark.parametrize("bad", [math.inf, math.nan, 1e30])
@pytest.mark.parametrize("field", [0, 2])
def test_diagnostics_of_extreme_values(lw, field, bad):
    """A planted infinity or NaN is reported, a huge finite value summed as FP64 does."""
    rng = np.random.default_rng(62)
    f = [(rng.normal(size=(64, 64, 66)) * 1e-2).astype(np.float32) for _ in range(4)]
    f[field][13, 17, 19] = bad
    got, stored = diagnose(lw, [a.astype(np.float64) for a in f])
    assert got["finite"] == math.isfinite(bad)
    if math.isfinite(bad):
        for k, (x, mag) in sums(stored).items():
            assert abs(np.longdouble(got[k]) - x) <= 64 * 2.0 ** -53 * mag, (k, got[k], x)
