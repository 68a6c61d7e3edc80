"""The half-row D3Q19 kernel asked for by LWACM_OPT_KERNEL 5, where the automatic choice takes the
marching warps: recorded runs, stochastic rounding, omega_p and cavities still run on it."""
import numpy as np
import pytest

import oracle
from paper_1111_2142_gb300 import inputs
from test_gpu_parity import HALF_SHAPES, HALF_ULP, _tgv_box, errs, round_storage, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


@pytest.mark.parametrize("shape,storage", [((3, 8, 256), 0), ((6, 16, 256), 2), ((4, 16, 384), 0), ((3, 8, 512), 2),
                                           ((4, 9, 200), 0), ((3, 13, 100), 0)])
def test_constant_force(lw, shape, storage):
    """Whole rows and segments of them, 60 steps against the oracle (FP16 storage: 60 roundings to 11
    significant bits of O(0.03) velocities)."""
    f = inputs.smooth_random(shape, seed=31, u_amp=0.03, d_amp=0.01)
    g = (1e-4, 2e-5, -1e-4)
    got, name = run_gpu(lw, 19, f, 0.02, 60, force=g, storage=storage, kernel=5)
    assert name == "half_d3q19_tma"
    eu, ed = errs(got, oracle.step(19, *f, nu=0.02, force=g, nsteps=60), 0.03)
    assert eu < (60 * 2.0 ** -11 if storage else 1e-5) and ed < (60 * 2.0 ** -11 if storage else 1e-4)


@pytest.mark.parametrize("shape", HALF_SHAPES[1:])
@pytest.mark.parametrize("storage", [2, 1])
def test_half_storage_one_step(lw, storage, shape):
    """From a state rounded to the storage type one step differs from the oracle by the final
    rounding only (floors: FP16 subnormals, the FP32 rounding of O(u0) terms that cancel)."""
    f = [round_storage(a, storage) for a in _tgv_box(shape)]
    got, name = run_gpu(lw, 19, f, 0.005, 1, storage=storage, kernel=5)
    assert name == "half_d3q19_tma"
    for g, r in zip(got, oracle.step(19, *f, nu=0.005, nsteps=1)):
        tol = 1.05 * HALF_ULP[storage] * np.abs(r) + max(2.0 ** -25 if storage == 2 else 0.0, 4 * 2.0 ** -24 * 0.02)
        assert np.all(np.abs(g - r) <= tol)


def test_many_steps_from_graphs(lw):
    """256-node rows over three graph replays and single steps."""
    f = inputs.smooth_random((24, 40, 256), seed=33, u_amp=0.03, d_amp=0.01)
    got, name = run_gpu(lw, 19, f, 0.005, 200, kernel=5)
    assert name == "half_d3q19_tma"
    eu, ed = errs(got, oracle.step(19, *f, nu=0.005, nsteps=200), 0.03)
    assert eu < 1e-5 and ed < 1e-4


def test_offsets_beyond_32_bits(lw):
    """537M nodes, the fourth field beyond 2^31 elements: one step at sampled nodes, each the centre
    of its 3 x 3 x 3 neighbourhood stepped by the oracle as a periodic box."""
    import torch
    nx, ny, nz = 256, 2048, 1024
    g = torch.Generator(device="cuda").manual_seed(8)
    src = [(torch.rand((nz, ny, nx), generator=g, device="cuda") - 0.5) * s for s in (0.02, 0.1, 0.1, 0.1)]
    sim = lw.Lwacm(lw.D3Q19, nx, ny, nz, 0.02, kernel=5)
    assert sim.kernel_name == "half_d3q19_tma"
    sim.set_fields(*src)
    sim.step(1)
    out = sim.fields()
    rng = np.random.default_rng(9)
    pts = [(int(rng.integers(nz)), int(rng.integers(ny)), int(rng.integers(nx))) for _ in range(100)]
    for z, y, x in pts + [(0, 0, 0), (nz - 1, ny - 1, nx - 1)]:
        zi, yi, xi = ([(c + k) % n for k in (-1, 0, 1)] for c, n in ((z, nz), (y, ny), (x, nx)))
        ref = oracle.step(19, *[f[zi][:, yi][:, :, xi].double().cpu().numpy() for f in src], nu=0.02, nsteps=1)
        for o, r, tol in zip(out, ref, (1e-6, 5e-8, 5e-8, 5e-8)):  # 1e-6 of the velocities' scale 0.05
            assert abs(float(o[z, y, x]) - float(r[1, 1, 1])) < tol
    sim.close()
