"""The gradient grid of a cube with a short x axis (or x and y), which has a tile
shape of its own: the oracle's bit for bit around the edges of those tiles (through a Method II
way 1 map in FP64, which reads every component), and no dearer than the same
number of nodes the other way round (three times is allowed: its rows are short and
its one-sided differences form B/|B| again)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 32, 4), (5, 33, 5), (8, 31, 3), (9, 32, 4), (2, 65, 9), (4, 4, 32), (5, 8, 33),
                               (2, 3, 65)])
@pytest.mark.parametrize("kind", ["aniso", "stretched"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_short_x_axis(n, kind, dtype):
    import paper_2208_12569_gb300 as fq

    d = (0.5, 0.25, 0.75)
    hi = tuple((k - 1) * v for k, v in zip(n, d))
    g = (synth.stretched_grid(n, (0.0, 0.0, 0.0), hi, ratios=(1.2, 1.1, 1.3)) if kind == "stretched"
         else synth.Grid(n, (0.0, 0.0, 0.0), d))
    B = np.random.default_rng(sum(n)).standard_normal((n[2], n[1], n[0], 3)).astype(dtype)
    B[..., 2] += 3.0
    t = torch.from_numpy(B).cuda()
    pack = ("f64", "gradb")
    f = fq.Field(t, coords=g.coords, pack=pack) if kind == "stretched" else fq.Field(t, g.origin, g.spacing, pack=pack)
    pl = ((0.0, 0.0, 0.0), (hi[0] / 7, 0.0, 0.0), (0.0, hi[1] / 40, 0.0), 7, 40)
    got = to_np(fq.qmap_plane(f, *pl, fq.params(precision="f64", method=2, gradb_way=1)))
    ref = oracle.plane(B.astype(np.float64), g, *pl, oracle.params(method=2, way=1))
    for k in ("Q", "Tw", "length", "r2", "face2", "status"):
        a, b = got[k], np.asarray(ref[k]).astype(got[k].dtype)
        assert np.array_equal(a.reshape(-1), b.reshape(-1), equal_nan=a.dtype.kind == "f"), k
    f.close()


def test_short_x_axis_is_not_dearer():
    import paper_2208_12569_gb300 as fq

    ms = []
    for n in ((2, 512, 512), (512, 512, 2)):
        B = torch.randn((n[2], n[1], n[0], 3), generator=torch.Generator().manual_seed(2)).cuda()
        f = fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f32", "gradb"))
        ts = []
        for _ in range(11):
            e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e[0].record()
            for _ in range(4):
                f.update(B)
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        ms.append(sorted(ts)[5])
        f.close()
    assert ms[0] < 3.0 * ms[1], ms
