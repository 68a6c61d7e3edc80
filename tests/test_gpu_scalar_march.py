"""The passive scalar on the marching D3Q19 kernel (kernels_scalar3.cu): edges of strips,
tiles and runs of planes, 256-node rows and the general flow kernel before it, forcing,
against the FP64 oracle."""
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


@pytest.mark.parametrize("shape", [(1, 4, 1), (2, 5, 29), (3, 6, 30), (1, 7, 31), (5, 17, 61), (40, 9, 7), (3, 66, 91),
                                   (37, 24, 256), (4, 12, 128)])
def test_marching_scalar_matches_oracle(lw, shape):
    f = inputs.smooth_random(shape, seed=91, u_amp=0.05, d_amp=0.01)
    T0 = 1.0 + 0.2 * inputs.smooth_random(shape, seed=92, u_amp=0.0, d_amp=1.0)[0]
    nz, ny, nx = shape
    sim = lw.Lwacm(19, nx, ny, nz, 0.02, scalar_alpha=0.03)
    sim.set_fields(*f)
    sim.set_scalar(T0)
    sim.step(13)
    got, gT = sim.get_fields(), sim.get_scalar()
    sim.close()
    ref = oracle.step_scalar(19, *f, T=T0, nu=0.02, alpha=0.03, nsteps=13)
    eu = max(float(np.max(np.abs(g - r))) for g, r in zip(got[1:], ref[1:-1])) / 0.05
    # T ~ 1 is the sum of 19 values and rounded once a step: a few units in the last place a step
    assert eu < 1e-5 and float(np.max(np.abs(gT - ref[-1]))) < 13 * 4 * 2.0 ** -24


@pytest.mark.parametrize("storage,half_ulp", [(1, 2.0 ** -8), (2, 2.0 ** -11)])
def test_marching_scalar_half_storage(lw, storage, half_ulp):
    """One step from a rounded state: half a unit in the last place of the scalar (relative, at
    most 2^-8 of a BF16 and 2^-11 of an FP16 value) and the FP32 sum."""
    shape = (5, 17, 61)
    import torch
    t = {1: torch.bfloat16, 2: torch.float16}[storage]
    r = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float32)).to(t).double().numpy()  # noqa: E731
    f = [r(a) for a in inputs.smooth_random(shape, seed=93, u_amp=0.05, d_amp=0.01)]
    T0 = r(1.0 + 0.2 * inputs.smooth_random(shape, seed=94, u_amp=0.0, d_amp=1.0)[0])
    sim = lw.Lwacm(19, 61, 17, 5, 0.02, scalar_alpha=0.03, storage=storage)
    sim.set_fields(*f)
    sim.set_scalar(T0)
    sim.step(1)
    gT = sim.get_scalar()
    sim.close()
    ref = oracle.step_scalar(19, *f, T=T0, nu=0.02, alpha=0.03, nsteps=1)[-1]
    assert np.all(np.abs(gT - ref) <= np.abs(ref) * half_ulp + 4e-7)
