"""FP32 Method II way 2 forms B at the offset points from the corners that the
stage's own evaluation read, and gathers where an offset leaves the cell: with
offsets of 0.001 cells (nearly all stay), 0.2 and 0.45 cells (many leave) the
map follows the FP64 tracer, which gathers every point, and lines that start on
nodes and faces do too. Bound: the median error that the FP32 way-2 maps are
held to elsewhere (1e-3); 0.45-cell offsets average over kinks, so an error in
the cell's choice would show at the size of Q itself."""
import numpy as np
import pytest
import torch

import synth
from parity import q_rel, to_np, tw_rel

pytestmark = pytest.mark.gpu

N = (33, 29, 21)


@pytest.mark.parametrize("eps", [1e-3, 0.2, 0.45])
@pytest.mark.parametrize("grid", ["unit", "aniso", "stretched"])
@pytest.mark.parametrize("scheme", [0, 1])
def test_way2_offsets_inside_and_outside_the_cell(eps, grid, scheme):
    import paper_2208_12569_gb300 as fq

    hi = tuple(float(v - 1) for v in N)
    d = (1.0, 1.0, 1.0)
    if grid == "stretched":
        g = synth.stretched_grid(N, (0.0, 0.0, 0.0), hi)
    else:
        d = (1.0, 1.0, 1.0) if grid == "unit" else (0.5, 0.25, 0.75)
        g = synth.Grid(N, (0.0, 0.0, 0.0), d)
    hi = tuple(h * v for h, v in zip(hi, d))
    ch = synth.random_charges(np.random.default_rng(3), 6, ((0.0, hi[0]), (0.0, hi[1])), depth=(4.0 * d[2], 9.0 * d[2]))
    B = torch.from_numpy(synth.monopole_cube(g, ch, dtype=np.float32)).cuda()
    f = fq.Field(B, coords=g.coords) if grid == "stretched" else fq.Field(B, g.origin, g.spacing)
    # seeds half a cell apart, every second one on a node row (the lattice starts a quarter cell before one)
    nu, nv = 2 * (N[0] - 2), 2 * (N[1] - 2)
    org = (0.75 * d[0], 0.75 * d[1], 0.0)
    pl = dict(origin=org, u=(0.5 * d[0], 0.0, 0.0), v=(0.0, 0.5 * d[1], 0.0), nu=nu, nv=nv)
    out = {}
    for prec in ("f32", "f64"):
        p = fq.params(precision=prec, method=2, gradb_way=2, eps_way2=eps, scheme=scheme, step=1.0)
        out[prec] = to_np(fq.qmap_plane(f, p=p, **pl))
    assert np.mean(out["f32"]["status"] == out["f64"]["status"]) > 0.99
    assert np.median(q_rel(out["f32"], out["f64"])) < 1e-3
    assert np.median(tw_rel(out["f32"], out["f64"])) < 1e-3
    f.close()
