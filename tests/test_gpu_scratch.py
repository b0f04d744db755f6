"""Calls that split the directions of their lines need more scratch than calls that
do not. A call up to the size of an earlier one of its kind finds its scratch in
place, whatever differs that decides on splitting (the plane's place, the seeds'
spacing, blocks_per_sm); and splitting is no reason for a call to fail where
whole lines would fit. Allocation is refused by the library's cap, so nothing
is exhausted."""
import numpy as np
import pytest
import torch

import synth
from parity import to_np

pytestmark = pytest.mark.gpu

N = (40, 36, 24)


@pytest.fixture(scope="module")
def fq():
    import paper_2208_12569_gb300 as fq

    return fq


@pytest.fixture(autouse=True)
def _no_cap(fq):
    yield
    fq.debug_alloc_cap(0)


def _field(fq, pack=("f32",)):
    grid = synth.Grid(N, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    B = synth.monopole_cube(grid, synth.random_charges(np.random.default_rng(5), 6, ((0.0, 39.0), (0.0, 35.0))), dtype=np.float32)
    return fq.Field(torch.from_numpy(B).cuda(), grid.origin, grid.spacing, pack=pack)


def _plane(z, nu, nv):
    return dict(origin=(0.0, 0.0, z), u=(39.0 / nu, 0.0, 0.0), v=(0.0, 35.0 / nv, 0.0), nu=nu, nv=nv)


def _same(a, b):
    for k in a:
        assert a[k].tobytes() == b[k].tobytes(), k


def test_inside_after_face_method2(fq):
    f = _field(fq)
    p = fq.params(precision="f32", method=2, gradb_way=2)
    ref = to_np(fq.qmap_plane(_field(fq), p=p, **_plane(9.5, 150, 150)))
    fq.qmap_plane(f, p=p, **_plane(0.0, 150, 150))
    fq.debug_alloc_cap(1)
    _same(to_np(fq.qmap_plane(f, p=p, **_plane(9.5, 150, 150))), ref)


def test_default_after_few_blocks(fq):
    f = _field(fq)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nv = 96 * 4 * sms // 250 + 6  # above what one block per SM splits, far below what four do
    ref = to_np(fq.qmap_plane(_field(fq), p=fq.params(precision="f32"), **_plane(9.5, 250, nv)))
    fq.qmap_plane(f, p=fq.params(precision="f32", blocks_per_sm=1), **_plane(9.5, 250, nv))
    fq.debug_alloc_cap(1)
    _same(to_np(fq.qmap_plane(f, p=fq.params(precision="f32"), **_plane(9.5, 250, nv))), ref)


def test_dense_after_sparse_in_a_large_cube(fq):
    n = (1024, 512, 86)
    z, y, x = torch.meshgrid(*[torch.arange(k, dtype=torch.float32, device="cuda") for k in n[::-1]], indexing="ij")
    B = torch.stack((0.1 + 0.0 * x, 0.2 * torch.sin(0.01 * x), 1.0 + 0.001 * y), -1)
    del x, y, z
    f = fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f32",))
    p = fq.params(precision="f32")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lines = 96 * 12 * sms + 15000  # sparse: 3 blocks, not split; dense: 4 blocks, split
    nz = 50
    nx = ny = int((lines / nz) ** 0.5) + 1
    fq.qmap_volume(f, (0.0, 0.0, 0.0), (4.0, 4.0, 1.5), nx, ny, nz, p)
    fq.debug_alloc_cap(1)
    fq.qmap_volume(f, (0.0, 0.0, 0.0), (0.5, 0.5, 0.5), nx, ny, nz - 1, p)
    f.check()
    f.close()


@pytest.mark.parametrize("kind", ["plane", "list"])
def test_whole_lines_where_split_ones_do_not_fit(fq, kind):
    p = fq.params(precision="f32")
    seeds = torch.rand((1000, 3), generator=torch.Generator().manual_seed(1), dtype=torch.float64).cuda() * 20.0 + 1.0

    def call(f):
        return to_np(fq.qmap_plane(f, p=p, **_plane(9.5, 100, 100)) if kind == "plane" else fq.twist(f, seeds, p))

    ref = call(_field(fq))
    # the least cap under which a new field's call succeeds, to 1/64: with split
    # directions it is 63 (list: 71) bytes a line and a few, with whole lines 8 to 40 less
    lo, hi = 0, 1 << 23
    while hi - lo > max(64, lo // 64):
        mid = (lo + hi) // 2
        f = _field(fq)
        fq.debug_alloc_cap(mid)
        try:
            _same(call(f), ref)
            hi = mid
        except fq.FqslError as e:
            assert e.status == 3
            lo = mid
        fq.debug_alloc_cap(0)
        f.close()
    n = 10000 if kind == "plane" else 1000
    assert hi < n * (240 if kind == "plane" else 67) + 4096, hi / n


def test_capture_with_room_for_whole_lines(fq):
    # the scratch of a list call holds whole lines of a small Method II interior plane
    f = _field(fq)
    p = fq.params(precision="f32", method=2, gradb_way=2)
    pl = _plane(9.5, 100, 100)
    ref = to_np(fq.qmap_plane(_field(fq), p=p, **pl))
    per = 4 * 12 + 4 * 12 + 32 + 63 + 8 + 17 + 64  # a line's scratch, generously; a list's line takes 63 bytes
    seeds = torch.rand((10000 * per // 63, 3), dtype=torch.float64, device="cuda") * 20.0
    fq.twist(f, seeds, p=fq.params(precision="f32"))
    out = fq.alloc_out(10000)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            fq.qmap_plane(f, p=p, out=out, **pl)
    g.replay()
    torch.cuda.synchronize()
    _same(to_np(out), ref)
