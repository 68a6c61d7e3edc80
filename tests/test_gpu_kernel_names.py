"""lwacm_kernel_name says which kernel runs, also where two kernels share a class of
LWACM_OPT_KERNEL (the first part of the name)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


# (lattice, (nx, ny, nz), keyword arguments, options, name)
CASES = [
    (19, (24, 24, 24), {}, {}, "generic_d3q19_march"),
    (19, (24, 24, 24), dict(bc=1), {}, "generic_d3q19_march"),
    (19, (24, 3, 24), {}, {}, "generic_d3q19"),
    (19, (24, 24, 24), {}, dict(NU_P=0.1), "generic_d3q19"),
    (19, (24, 24, 24), dict(scalar_alpha=0.02), {}, "generic_d3q19_march+scalar_march"),
    (19, (24, 24, 24), dict(scalar_alpha=0.02), dict(NU_P=0.1), "generic_d3q19"),
    (19, (256, 16, 8), {}, {}, "half_d3q19_march"),
    (19, (256, 16, 8), {}, dict(KERNEL=5), "half_d3q19_tma"),
    (19, (256, 16, 8), {}, dict(KERNEL=1), "generic_d3q19_march"),
    (19, (256, 16, 8), dict(bc=1), {}, "half_d3q19_tma"),
    (19, (256, 16, 8), {}, dict(NU_P=0.1), "half_d3q19_tma+nu_p_sum"),
    (19, (256, 16, 8), dict(scalar_alpha=0.02), {}, "half_d3q19_tma+scalar_rows_march"),
    (19, (128, 16, 8), dict(scalar_alpha=0.02), {}, "half_d3q19_tma+scalar_rows"),
    (19, (128, 16, 8), {}, {}, "half_d3q19_tma"),
    (9, (64, 64, 1), {}, {}, "tiles2d_d2q9_rows+cluster"),
    (9, (64, 64, 1), dict(semi_implicit=True), {}, "tiles2d_d2q9_rows"),
    (9, (400, 300, 1), {}, {}, "tiles2d_d2q9_rows"),
    (9, (64, 64, 1), {}, dict(BATCH_TILE=2), "tiles2d_d2q9_30x14"),
    (9, (64, 64, 1), dict(scalar_alpha=0.02), {}, "generic_d2q9"),
]


@pytest.mark.parametrize("Q,dims,kw,opts,name", CASES)
def test_single_domains(lw, Q, dims, kw, opts, name):
    kw = dict(kw)
    sim = lw.Lwacm(Q, *dims, 0.02, kw.pop("bc", 0), **kw)
    for k, v in opts.items():
        sim.set_option(getattr(lw, "OPT_" + k), v)
    assert sim.kernel_name == name
    sim.close()


@pytest.mark.parametrize("Q,mode,tile,name", [(9, 0, 0, "batch_rows_step"), (9, 1, 0, "batch_rows_persistent"),
                                              (9, 0, 2, "batch_tiles30x14_step"), (19, 0, 0, "batch_step"),
                                              (19, 1, 0, "batch_persistent")])
def test_ensembles(lw, Q, mode, tile, name):
    dims = [(33, 20), (40, 31)] if Q == 9 else [(9, 8, 7), (5, 6, 7)]
    sim = lw.LwacmBatch(Q, dims, [0.02, 0.03], mode=mode, tile=tile)
    assert sim.kernel_name == name
    sim.close()


def test_the_force_field_changes_the_name(lw):
    """Switched on, a field takes a 256-node row from kernel 5 to kernel 1, and back."""
    import torch
    sim = lw.Lwacm(19, 256, 16, 8, 0.02, force_field=True)
    assert sim.kernel_name == "half_d3q19_march"
    g = [torch.zeros(8, 16, 256, device="cuda") for _ in range(3)]
    sim.set_force_field(*g)
    assert sim.kernel_name == "generic_d3q19_march"
    sim.set_force_field(None, None)
    assert sim.kernel_name == "half_d3q19_march"
    sim.close()
