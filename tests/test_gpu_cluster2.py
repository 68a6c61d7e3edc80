"""Several steps of a small D2Q9 domain in one launch of a cluster (kernels_cluster2.cu): the
same fields, bit for bit, as single steps on the marching kernel, which the oracle checks."""
import numpy as np
import pytest

from paper_1111_2142_gb300 import inputs

pytestmark = pytest.mark.gpu

# fewer rows than CTAs, one column, one node to two nodes a thread, uneven rows, the largest
SHAPES = [(1, 1), (7, 1), (1, 7), (2, 2), (3, 29), (16, 31), (17, 33), (33, 60), (128, 128), (150, 100), (16, 1664)]


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


def both(lw, shape, T, bc=0, nu_p=None, **kw):
    ny, nx = shape
    f = inputs.smooth_random(shape, seed=71, u_amp=0.05, d_amp=0.01)
    out = []
    for calls in ([T], [1] * T):
        sim = lw.Lwacm(9, nx, ny, 1, 0.02, bc, lid=(0.05, 0.01) if bc else None, **kw)
        if nu_p:
            sim.set_option(lw.OPT_NU_P, nu_p)
        sim.set_fields(*f)
        for n in calls:
            sim.step(n)
        assert sim.step_count() == T
        got = list(sim.get_fields())
        if kw.get("bulk_gamma"):
            got.append(sim.get_trace())
        sim.close()
        out.append(got)
    for a, b in zip(*out):
        assert np.array_equal(a, b), (shape, bc, nu_p, kw)


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_equals_single_steps(lw, shape, storage):
    both(lw, shape, 5, storage=storage)
    both(lw, shape, 6, storage=storage, force=(1e-4, 2e-5))
    both(lw, shape, 5, storage=storage, nu_p=0.1)
    both(lw, shape, 5, storage=storage, bulk_gamma=0.4)
    both(lw, shape, 6, storage=storage, bulk_gamma=0.3, nu_p=0.08)
    if min(shape) >= 2:
        both(lw, shape, 5, bc=1, storage=storage)
        both(lw, shape, 5, bc=2, storage=storage, force=(1e-4, 0.0))


def test_cluster_then_single_steps_and_long_runs(lw):
    """Any split of a run gives the same fields: more steps than one launch takes, odd
    remainders, a graph prepared for the whole run."""
    f = inputs.smooth_random((20, 24), seed=72, u_amp=0.03, d_amp=0.005)
    out = []
    for calls in ([8192 + 131], [1, 64, 3, 8192 + 63]):
        sim = lw.Lwacm(9, 24, 20, 1, 0.02)
        sim.set_fields(*f)
        sim.prepare(sum(calls))
        for n in calls:
            sim.step(n)
        assert sim.step_count() == 8192 + 131
        out.append(sim.get_fields())
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [4, 5, 64])
def test_cluster_leaves_the_state_in_the_buffer_of_single_steps(lw, n):
    """An even number of steps ends in the buffer it started from, so that a caller's own graph
    of them advances the state at every replay."""
    import torch
    f = inputs.smooth_random((20, 24), seed=73, u_amp=0.03, d_amp=0.005)
    sim = lw.Lwacm(9, 24, 20, 1, 0.02, stream=torch.cuda.Stream())
    sim.set_fields(*f)
    before = sim.fields()[0].data_ptr()
    sim.step(n)
    assert (sim.fields()[0].data_ptr() == before) == (n % 2 == 0)
    if n % 2 == 0:
        sim.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=sim.stream):
            sim.step(n)
        with torch.cuda.stream(sim.stream):
            g.replay()
            g.replay()
        sim.sync()
        ref = lw.Lwacm(9, 24, 20, 1, 0.02)
        ref.set_fields(*f)
        for _ in range(3 * n):
            ref.step(1)
        for a, b in zip(sim.get_fields(), ref.get_fields()):
            assert np.array_equal(a, b)
        ref.close()
    sim.close()


def takes_cluster(shape, nu_p):
    """The bounds of the cluster kernel: at most 1664 nodes and 227 KB of link arrays a CTA."""
    ny, nx = shape
    rows = -(-ny // min(ny, 16))
    return rows * nx <= 1664 and 2 * (12 if nu_p else 8) * (rows + 2) * nx * 4 <= 227 * 1024


# two nodes a thread: square, uneven rows, tall, two rows and one row a CTA up to the largest
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(160, 160), (165, 130), (255, 97), (175, 150), (17, 800), (16, 1100), (16, 1210)])
def test_two_nodes_a_thread(lw, shape, storage):
    assert takes_cluster(shape, False) and -(-shape[0] // 16) * shape[1] > 1024
    both(lw, shape, 5, storage=storage)
    both(lw, shape, 6, storage=storage, force=(1e-4, 2e-5))
    both(lw, shape, 5, storage=storage, nu_p=0.1)
    both(lw, shape, 5, storage=storage, bulk_gamma=0.4)
    both(lw, shape, 6, storage=storage, bulk_gamma=0.3, nu_p=0.08)
    both(lw, shape, 5, bc=1, storage=storage)
    both(lw, shape, 5, bc=2, storage=storage, force=(1e-4, 0.0))


@pytest.mark.parametrize("nu_p", [None, 0.1])
@pytest.mark.parametrize("shape", SHAPES + [(160, 160), (17, 800), (16, 1210), (16, 1211), (176, 152)])
def test_the_cluster_ran(lw, shape, nu_p):
    """Where the domain is within its bounds the cluster takes the steps: the name keeps saying so
    after them (a device that refused it would have fallen back to single steps)."""
    ny, nx = shape
    sim = lw.Lwacm(9, nx, ny, 1, 0.02)
    if nu_p:
        sim.set_option(lw.OPT_NU_P, nu_p)
    sim.set_fields(*inputs.smooth_random(shape, seed=74, u_amp=0.05, d_amp=0.01))
    sim.step(8)
    sim.sync()
    assert sim.kernel_name == "tiles2d_d2q9_rows" + ("+cluster" if takes_cluster(shape, nu_p) else "")
    sim.close()
