"""Small FP32 maps and lists give the two directions of a line to two lanes and
few lines to a warp; batches and long lists do neither. Both must give the same
bytes, whatever ends a line first (its footpoints, or max_steps before, between
or after the two directions)."""
import numpy as np
import pytest
import torch

import synth
from parity import to_np

pytestmark = pytest.mark.gpu

N = (40, 36, 24)


@pytest.fixture(scope="module")
def field():
    import paper_2208_12569_gb300 as fq

    grid = synth.Grid(N, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    ch = synth.random_charges(np.random.default_rng(11), 8, ((0.0, N[0] - 1.0), (0.0, N[1] - 1.0)), depth=(3.0, 9.0))
    B = synth.monopole_cube(grid, ch, dtype=np.float32)
    f = fq.Field(torch.from_numpy(B).cuda(), grid.origin, grid.spacing, pack=("f32",))
    yield fq, f
    f.close()


def _same(a, b):
    for k in a:
        assert a[k].tobytes() == b[k].tobytes(), k


@pytest.mark.parametrize("max_steps", [1, 4, 9, 17, 33, 100000])
@pytest.mark.parametrize("precision,scheme", [("f32", 0), ("f32acc64", 0), ("f32", 1)])
@pytest.mark.parametrize("nu,nv", [(1, 1), (9, 5), (61, 37)])
def test_split_lattice_equals_batch_entry(field, max_steps, precision, scheme, nu, nv):
    fq, f = field
    p = fq.params(precision=precision, scheme=scheme, max_steps=max_steps)
    pl = dict(origin=(0.0, 17.3, 0.0), u=((N[0] - 1.0) / nu, 0.0, 0.0), v=(0.0, 0.0, (N[2] - 1.0) / nv), nu=nu, nv=nv)
    one = to_np(fq.qmap_plane(f, p=p, **pl))
    b = fq.Batch([f], [pl], p)
    _same(one, to_np(b.run()[0]))
    b.close()


@pytest.mark.parametrize("max_steps", [1, 6, 18, 100000])
@pytest.mark.parametrize("n", [1, 33, 1216, 1217, 2433])
def test_short_list_equals_the_same_seeds_in_a_long_one(field, n, max_steps):
    fq, f = field
    g = torch.Generator().manual_seed(n)
    seeds = (torch.rand((n, 3), generator=g, dtype=torch.float64) * 1.1 - 0.05) * torch.tensor([v - 1.0 for v in N], dtype=torch.float64)
    seeds = seeds.cuda()  # a few outside the box
    p = fq.params(precision="f32", max_steps=max_steps)
    short = to_np(fq.twist(f, seeds, p))
    reps = 100000 // n
    long = to_np(fq.twist(f, seeds.repeat(reps, 1), p))
    _same(short, {k: v[:n] for k, v in long.items()})
    _same(short, {k: v[(reps - 1) * n:] for k, v in long.items()})
