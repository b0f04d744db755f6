"""Maps small enough to have the directions of their lines split give the bytes of
the same maps with whole lines: Method II (deviation vectors of two lanes), grids
of every kind, planes and volumes, step budgets that end lines before, between
and after the two directions, and with the extra lines of rotated seeds in the
lattice's launch or, timed, in their own. blocks_per_sm = 1 lowers the limit for
splitting; the sizes lie between the two limits."""
import numpy as np
import pytest
import torch

import synth
from parity import to_np

pytestmark = pytest.mark.gpu

N = (36, 33, 22)


def _field(kind):
    import paper_2208_12569_gb300 as fq

    d = (0.5, 0.3, 0.7) if kind == "aniso" else (1.0, 1.0, 1.0)
    hi = tuple((k - 1) * v for k, v in zip(N, d))
    g = synth.stretched_grid(N, (0.0, 0.0, 0.0), hi) if kind == "stretched" else synth.Grid(N, (0.0, 0.0, 0.0), d)
    ch = synth.random_charges(np.random.default_rng(13), 8, ((0.0, hi[0]), (0.0, hi[1])), depth=(3.0 * d[2], 8.0 * d[2]))
    B = torch.from_numpy(synth.monopole_cube(g, ch, dtype=np.float32)).cuda()
    pack = ("f32", "gradb")
    f = fq.Field(B, coords=g.coords, pack=pack) if kind == "stretched" else fq.Field(B, g.origin, g.spacing, pack=pack)
    return fq, f, hi


def _warps(blocks):
    return 4 * blocks * torch.cuda.get_device_properties(0).multi_processor_count


def _same(a, b):
    for k in a:
        assert a[k].tobytes() == b[k].tobytes(), k


@pytest.mark.parametrize("max_steps", [1, 9, 17, 33, 150, 100000])
@pytest.mark.parametrize("kind", ["unit", "aniso", "stretched"])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("way", [1, 2])
def test_method2(way, scheme, kind, max_steps):
    fq, f, hi = _field(kind)
    nu = 107
    nv = 16 * _warps(1) // nu + 3  # split with the default's blocks, whole with one
    pl = dict(origin=(0.0, 0.47 * hi[1], 0.0), u=(hi[0] / nu, 0.0, 0.0), v=(0.0, 0.0, hi[2] / nv), nu=nu, nv=nv)
    kw = dict(precision="f32", method=2, gradb_way=way, scheme=scheme, step=1.1, max_steps=max_steps)
    split, whole = [to_np(fq.qmap_plane(f, p=fq.params(blocks_per_sm=b, **kw), **pl)) for b in (0, 1)]
    _same(split, whole)
    f.close()


@pytest.mark.parametrize("max_steps", [9, 33, 150, 100000])
@pytest.mark.parametrize("kind", ["aniso", "stretched"])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("precision", ["f32", "f32acc64"])
def test_method1(precision, scheme, kind, max_steps):
    fq, f, hi = _field(kind)
    n = 96 * _warps(1)
    kw = dict(precision=precision, scheme=scheme, step=1.1, max_steps=max_steps, rot_thresh=0.3)
    nu = 251
    nv = n // nu + 3
    pl = dict(origin=(0.0, 0.47 * hi[1], 0.0), u=(hi[0] / nu, 0.0, 0.0), v=(0.0, 0.0, hi[2] / nv), nu=nu, nv=nv)
    split, whole = [to_np(fq.qmap_plane(f, p=fq.params(blocks_per_sm=b, **kw), **pl)) for b in (0, 1)]
    assert int((split["status"] & fq.LINE_ROTATED != 0).sum()) > 50
    _same(split, whole)
    f.set_timing(True)
    _same(split, to_np(fq.qmap_plane(f, p=fq.params(**kw), **pl)))
    f.set_timing(False)
    mu, mv = 41, 37
    mw = n // (mu * mv) + 3
    v = [to_np(fq.qmap_volume(f, (0.0, 0.0, 0.0), (hi[0] / mu, hi[1] / mv, hi[2] / mw), mu, mv, mw,
                              fq.params(blocks_per_sm=b, **kw))) for b in (0, 1)]
    _same(*v)
    f.close()


@pytest.mark.parametrize("kind", ["aniso", "stretched"])
@pytest.mark.parametrize("scheme", [0, 1])
def test_list(scheme, kind):
    fq, f, hi = _field(kind)
    n = _warps(1) // 2 + 3
    s = (torch.rand((n, 3), generator=torch.Generator().manual_seed(3), dtype=torch.float64) * torch.tensor(hi, dtype=torch.float64)).cuda()
    for max_steps in (9, 33, 100000):
        kw = dict(precision="f32", scheme=scheme, step=1.1, max_steps=max_steps)
        split, whole = [to_np(fq.twist(f, s, fq.params(blocks_per_sm=b, **kw))) for b in (0, 1)]
        _same(split, whole)
    f.close()
