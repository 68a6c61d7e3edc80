"""Kernels that overlap the grid before them (griddepcontrol.wait, programmatic stream
serialization) must not read device memory through the read-only path: that path is defined only
for data nobody writes while the kernel is alive, and such a kernel is alive while the grid before
it still writes the state. Nor must kernels that run many steps in one launch, whose CTAs read what
others wrote before a barrier. Read from the sources, since a stale value cannot be provoked at
will."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1111_2142_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s*(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^)]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), m.group(2), text[m.end():i]


def overlapped():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            for k, params, body in kernels(source(name)):
                if "griddepcontrol.launch_dependents" in body:
                    yield name, k, params


def test_every_overlapped_kernel_is_known():
    assert {k for _, k, _ in overlapped()} == {"k_d2q9_rows", "k_batch_rows", "k_d3q19_rows", "k_adj_rows", "k_d3q19_half"}


@pytest.mark.parametrize("kernel", ["k_d2q9_rows", "k_batch_rows", "k_d3q19_rows", "k_adj_rows"])
def test_no_read_only_pointers(kernel):
    """A load through a pointer marked const __restrict__ may be compiled to the read-only path
    (the half-row kernel's goes to bulk copies only)."""
    params = {k: p for _, k, p in overlapped()}[kernel]
    assert "__restrict__" not in params


@pytest.mark.parametrize("name", ["rows2.cuh", "kernels_rows2.cu", "kernels_rows3.cu"])
def test_no_read_only_loads(name):
    """The marches read state and force field with ordinary loads (kernels_batch.cu has the
    2D-tile kernels too, which overlap nothing; its march is that of rows2.cuh)."""
    text = source(name)
    assert "__ldg" not in text and not re.search(r"\bldf\s*\(", text)


def test_persistent_kernels_read_with_ordinary_loads():
    """Their updates are the single-step kernels' with RO (read-only) off; the march past L1."""
    bodies = {k: (p, b) for k, p, b in kernels(source("kernels_batch.cu"))}
    want = {"k_batch_persistent": "tile_update<Q, false>(", "k_batch_tiles_persistent": "tile2_update<TW, TH, false>(",
            "k_batch_rows_persistent": "rows2_update<NS, T, true>("}
    assert set(want) == {k for k in bodies if "grid_barrier" in bodies[k][1]}
    for k, call in want.items():
        params, body = bodies[k]
        assert call in body and "__restrict__" not in params
    for name in ("node_update.cuh", "kernels_batch.cu"):  # the state only through ldx<RO>
        text = source(name)
        assert not re.search(r"\bldf\s*\(", text)
        assert all("field" in m for m in re.findall(r"__ldg\(([^)]*)\)", text))
