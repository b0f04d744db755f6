"""FP64 planes of more than 6 to 16 times 1,024 seeds per SM (by scheme, grid and
place) give a line one lane, smaller ones eight: the rows that a large and a small
plane share have the same bytes, whatever ends their lines."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

N = (22, 19, 15)


@pytest.mark.parametrize("max_steps", [7, 100000])
@pytest.mark.parametrize("cut", ["bottom", "xz"])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("kind", ["unit", "aniso", "stretched"])
def test_large_plane_equals_its_rows(kind, scheme, cut, max_steps):
    import paper_2208_12569_gb300 as fq

    d = (0.5, 0.25, 0.75) if kind == "aniso" else (1.0, 1.0, 1.0)
    hi = tuple((k - 1) * v for k, v in zip(N, d))
    g = synth.stretched_grid(N, (0.0, 0.0, 0.0), hi) if kind == "stretched" else synth.Grid(N, (0.0, 0.0, 0.0), d)
    ch = synth.random_charges(np.random.default_rng(9), 6, ((0.0, hi[0]), (0.0, hi[1])), depth=(2.0 * d[2], 6.0 * d[2]))
    B = torch.from_numpy(synth.monopole_cube(g, ch, dtype=np.float64)).cuda()
    f = fq.Field(B, coords=g.coords, pack=("f64",)) if kind == "stretched" else fq.Field(B, g.origin, g.spacing, pack=("f64",))
    p = fq.params(precision="f64", scheme=scheme, step=1.3, max_steps=max_steps)
    nu = 1001
    nv = (16 if kind == "unit" and cut == "xz" else 8) * 1024 * torch.cuda.get_device_properties(0).multi_processor_count // nu + 2
    w = 1 if cut == "bottom" else 2
    v = tuple(hi[w] / nv if a == w else 0.0 for a in range(3))
    pl = dict(origin=(0.0, 0.0 if cut == "bottom" else 0.41 * hi[1], 0.0), u=(hi[0] / nu, 0.0, 0.0), v=v)
    large = fq.qmap_plane(f, nu=nu, nv=nv, p=p, **pl)
    few = nu * 299  # Q and the mixed-ends bit of the small plane's last row have no row above them
    small = fq.qmap_plane(f, nu=nu, nv=300, p=p, **pl)
    for k in large:
        a, b = large[k][:few].cpu().numpy(), small[k][:few].cpu().numpy()
        assert a.tobytes() == b.tobytes(), k
    assert int(((large["status"] & fq.LINE_ROTATED) != 0).sum()) > (100 if cut == "xz" else -1)
    f.close()
