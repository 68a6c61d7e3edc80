"""Fields and forces copied in by one launch for all arrays: vector and single loads (aligned
and unaligned sources, counts that are no multiple of four), every type."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1111_2142_gb300 import lwacm
    return lwacm


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 3), (3, 5, 7), (4, 8, 64), (33, 65, 129)])
@pytest.mark.parametrize("shift", [0, 1])
def test_fields_from_device_arrays(lw, shape, storage, dtype, shift):
    """The stored values are those of the same arrays handed over as FP64 host arrays (one copy
    and one launch an array), the sources at 16-byte boundaries or one element past them."""
    import torch
    n = int(np.prod(shape))
    g = torch.Generator(device="cuda").manual_seed(81)
    f = [(torch.randn(n + shift, generator=g, device="cuda", dtype=getattr(torch, dtype)) * 0.05)[shift:].view(shape)
         for _ in range(4)]
    sim = lw.Lwacm(19, shape[2], shape[1], shape[0], 0.02, storage=storage)
    sim.set_fields(*f)
    got = [v.clone() for v in sim.fields()]
    sim.set_fields(*[a.double().cpu().numpy() for a in f])
    for a, v in zip(got, sim.fields()):
        assert torch.equal(a, v)
    sim.close()


@pytest.mark.parametrize("shape", [(1, 1, 3), (5, 6, 7), (24, 80, 100)])
@pytest.mark.parametrize("order", [(0, 2, 3, None), (1, 2, 3, None), (0, 2, 1, 3), (3, 3, 0, 1), (0, 1, 2, 3)])
def test_fields_from_views_of_the_state(shape, order, lw):
    """The state's own views as sources: the arrays are copied one after the other, so that field k
    takes what its source holds once the fields before it are in place (None: another array)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(83)
    f = [torch.randn(shape, generator=g, device="cuda") * 0.05 for _ in range(5)]
    sim = lw.Lwacm(19, shape[2], shape[1], shape[0], 0.02)
    sim.set_fields(*f[:4])
    views = list(sim.fields())
    want = [t.clone() for t in f[:4]]
    for k, o in enumerate(order):
        want[k] = f[4].clone() if o is None else want[o].clone()
    sim.set_fields(*[f[4] if o is None else views[o] for o in order])
    for a, v in zip(want, sim.fields()):
        assert torch.equal(a, v)
    sim.close()


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_force_field_from_unaligned_arrays(lw, dtype):
    """A force field from arrays one element past a 16-byte boundary acts as from aligned ones."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(82)
    flat = [torch.randn(35 * 27 + 1, generator=g, device="cuda", dtype=getattr(torch, dtype)) * 1e-4 for _ in range(2)]
    out = []
    for a in ([t[1:].view(27, 35) for t in flat], [t[1:].view(27, 35).clone() for t in flat]):
        sim = lw.Lwacm(9, 35, 27, 1, 0.02, force_field=True)
        sim.set_fields(*[np.zeros((27, 35))] * 3)
        sim.set_force_field(*a)
        sim.step(3)
        out.append(sim.get_fields())
        sim.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    assert float(np.max(np.abs(out[0][1]))) > 1e-5


def test_force_field_from_memory_of_another_device(lw):
    """An FP32 force array that is not in this GPU's memory goes through a copy and not through a
    kernel that reads it, which may have no access to it. Pinned host memory stands in for another
    GPU's; the nodes of a captured call show the route."""
    import torch
    n = 24 * 20
    sim = lw.Lwacm(9, 24, 20, 1, 0.02, force_field=True, stream=torch.cuda.Stream())
    sim.set_fields(*[np.zeros((20, 24))] * 3)
    host = [(torch.arange(n, dtype=torch.float32) * s).pin_memory() for s in (1e-6, -2e-6)]
    here = [t.cuda() for t in host]
    torch.cuda.synchronize()

    def nodes(arrays):
        sim.set_force_field(*here)  # on already: nothing is chosen anew under capture
        sim.sync()
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g, stream=sim.stream):
            status = sim._lib.lwacm_set_force_field(sim._h, *[t.data_ptr() for t in arrays], None, lw.F32, lw.DEVICE)
        assert status == lw.OK
        cu, graph, count = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t()
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
        found, kind, kinds = (ctypes.c_void_p * count.value)(), ctypes.c_int(), []
        assert cu.cuGraphGetNodes(graph, found, ctypes.byref(count)) == 0
        for node in found:
            assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
            kinds.append(kind.value)
        return kinds

    assert nodes(here) == [0]  # one kernel
    assert nodes(host) == [1, 1]  # two copies
    out = []
    for arrays in (here, host):
        sim.set_fields(*[np.zeros((20, 24))] * 3)
        assert sim._lib.lwacm_set_force_field(sim._h, *[t.data_ptr() for t in arrays], None, lw.F32, lw.DEVICE) == lw.OK
        sim.step(3)
        out.append(sim.get_fields())
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    assert float(np.max(np.abs(out[0][1]))) > 1e-5
    sim.close()


def test_fields_outlive_the_call_on_another_stream(lw):
    """Arrays that are dropped right after set_fields are not handed out again while the copy still
    waits on the context's own stream."""
    import torch
    n = 64
    st = torch.cuda.Stream()
    sim = lw.Lwacm(9, n, n, 1, 0.02, stream=st)
    g = torch.Generator(device="cuda").manual_seed(84)
    f = [torch.randn(n, n, generator=g, device="cuda") * 0.05 for _ in range(3)]
    want = [t.cpu().numpy().astype(np.float64) for t in f]
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(50_000_000)  # some 30 ms during which the copy cannot start
    sim.set_fields(*f)
    del f
    other = [torch.full((n, n), 7.0, device="cuda") for _ in range(6)]
    torch.cuda.current_stream().synchronize()
    for a, b in zip(want, sim.get_fields()):
        assert np.array_equal(a, b)
    assert all(float(t[0, 0]) == 7.0 for t in other)
    sim.close()


@pytest.mark.parametrize("call", ["set_fields", "set_force_field", "set_scalar"])
def test_strided_arrays_on_another_stream(lw, call):
    """The copies made of strided arrays come from torch's current stream: the context's own stream
    reads them after it, also when that is busy."""
    import torch
    n = 96
    st = torch.cuda.Stream()
    sim = lw.Lwacm(9, n, n, 1, 0.02, stream=st, force_field=call == "set_force_field",
                   scalar_alpha=0.02 if call == "set_scalar" else None)
    ref = lw.Lwacm(9, n, n, 1, 0.02, force_field=call == "set_force_field",
                   scalar_alpha=0.02 if call == "set_scalar" else None)
    g = torch.Generator(device="cuda").manual_seed(85)
    f = [torch.randn(n, n, generator=g, device="cuda") * 0.05 for _ in range(3)]
    t = [1e-3 * v.t() for v in f]
    for s, src in ((ref, [v.contiguous() for v in t]), (sim, t)):
        s.set_fields(*f)
        torch.cuda.synchronize()
        if s is sim:
            for _ in range(8):  # memory that a copy may get holds other values
                torch.full((n, n), 7.0, device="cuda")
            torch.cuda._sleep(50_000_000)  # the copies wait on the current stream
        if call == "set_fields":
            s.set_fields(*src)
        elif call == "set_force_field":
            s.set_force_field(*src[1:])
        else:
            s.set_scalar(src[0])
        s.step(2)
        s.sync()
    for a, b in zip(ref.get_fields(), sim.get_fields()):
        assert np.array_equal(a, b)
    if call == "set_scalar":
        assert np.array_equal(ref.get_scalar(), sim.get_scalar())
    sim.close()
    ref.close()


def test_backward_on_another_stream(lw):
    """Seeds that are still being computed on torch's current stream when backward is called."""
    import torch
    n = 64
    out = []
    for st in (None, torch.cuda.Stream()):
        sim = lw.Lwacm(9, n, n, 1, 0.02, stream=st)
        g = torch.Generator(device="cuda").manual_seed(86)
        f = [torch.randn(n, n, generator=g, device="cuda") * 0.02 for _ in range(6)]
        torch.cuda.synchronize()
        sim.set_fields(*f[:3])
        sim.forward_record(6)
        sim.sync()
        torch.cuda._sleep(50_000_000)
        grads, gnu = sim.backward([v.t() for v in f[3:]])
        out.append([v.cpu().numpy() for v in grads] + [gnu])
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
