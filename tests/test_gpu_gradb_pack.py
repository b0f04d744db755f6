"""The tiled gradient-grid kernel at the sizes where its 16 x 8 x 4 tiles, their
halo and the one-sided face stencils can go wrong: axes of 2 and 3 nodes, one
node more or less than a tile, uniform, anisotropic and stretched. Method II
way 1 in FP64 reads every component of the grid, and has to be the oracle's map
bit for bit (the grid is formed as the oracle forms it)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2, 2, 2), (3, 2, 5), (16, 8, 4), (17, 9, 5), (15, 7, 3), (33, 16, 9)])
@pytest.mark.parametrize("kind", ["unit", "aniso", "stretched"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_way1_reads_the_oracles_gradient_grid(n, kind, dtype):
    import paper_2208_12569_gb300 as fq

    d = (0.5, 0.25, 0.75) if kind == "aniso" else (1.0, 1.0, 1.0)
    hi = tuple((k - 1) * v for k, v in zip(n, d))
    g = (synth.stretched_grid(n, (0.0, 0.0, 0.0), hi, ratios=(1.2, 1.1, 1.3)) if kind == "stretched"
         else synth.Grid(n, (0.0, 0.0, 0.0), d))
    rng = np.random.default_rng(sum(n))
    B = rng.standard_normal((n[2], n[1], n[0], 3)).astype(dtype)
    B[..., 2] += 3.0
    B[0, 0, 0] = 0.0  # |B| = 0 at a node: its B/|B| is taken as 0
    t = torch.from_numpy(B).cuda()
    pack = ("f64", "gradb")
    f = fq.Field(t, coords=g.coords, pack=pack) if kind == "stretched" else fq.Field(t, g.origin, g.spacing, pack=pack)
    f.update(t)
    pl = ((0.0, 0.0, 0.0), (hi[0] / 13, 0.0, 0.0), (0.0, hi[1] / 11, 0.0), 13, 11)
    got = to_np(fq.qmap_plane(f, *pl, fq.params(precision="f64", method=2, gradb_way=1)))
    ref = oracle.plane(B.astype(np.float64), g, *pl, oracle.params(method=2, way=1))
    for k in ("Q", "Tw", "length", "r2", "face2", "status"):
        a, b = got[k], np.asarray(ref[k]).astype(got[k].dtype)
        assert np.array_equal(a.reshape(-1), b.reshape(-1), equal_nan=a.dtype.kind == "f"), k
    f.close()
