"""The FP64 tracer's groups of eight lanes at the sizes where their scheduling
changes: fewer lines than a warp's four groups, ragged last warps, one, two and
four groups per warp, and step budgets that end lines anywhere. Every output is
the oracle's, bit for bit (it is the same arithmetic)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import to_np

pytestmark = pytest.mark.gpu

N = (28, 24, 18)


def _field(kind):
    import paper_2208_12569_gb300 as fq

    hi = tuple(float(v - 1) for v in N)
    if kind == "stretched":
        g = synth.stretched_grid(N, (-3.0, 1.0, -2.0), tuple(h + o for h, o in zip(hi, (-3.0, 1.0, -2.0))))
        lo = (-3.0, 1.0, -2.0)
    else:
        d = (1.0, 1.0, 1.0) if kind == "unit" else (0.5, 0.3, 0.7)
        lo = (0.0, 0.0, 0.0)
        g = synth.Grid(N, lo, d)
        hi = tuple(h * v for h, v in zip(hi, d))
    ch = synth.random_charges(np.random.default_rng(5), 7, ((lo[0], lo[0] + hi[0]), (lo[1], lo[1] + hi[1])),
                              depth=(3.0 - lo[2], 7.0 - lo[2]))
    B = synth.monopole_cube(g, ch, dtype=np.float64)
    t = torch.from_numpy(B).cuda()
    f = fq.Field(t, coords=g.coords, pack=("f64",)) if kind == "stretched" else fq.Field(t, g.origin, g.spacing, pack=("f64",))
    return fq, f, B, g, lo, hi


def _same(got, ref, keys):
    for k in keys:
        a, b = np.asarray(got[k]), np.asarray(ref[k]).astype(np.asarray(got[k]).dtype)
        assert np.array_equal(a.reshape(-1), b.reshape(-1), equal_nan=a.dtype.kind == "f"), k


@pytest.mark.parametrize("kind", ["unit", "aniso", "stretched"])
@pytest.mark.parametrize("scheme", [0, 1])
def test_list_sizes(kind, scheme):
    fq, f, B, g, lo, hi = _field(kind)
    rng = np.random.default_rng(1)
    s = np.array(lo) + (rng.random((9731, 3)) * 1.04 - 0.02) * np.array(hi)
    s[:8, 2] = lo[2]  # on the bottom face, and on nodes
    s[4:8] = np.round((s[4:8] - lo)) + lo if kind == "unit" else s[4:8]
    ref = oracle.twist(B, g, s, oracle.params(scheme=scheme, step=1.3) if scheme else oracle.params())
    p = fq.params(precision="f64", scheme=scheme, step=1.3)
    for n in (1, 2, 3, 4, 5, 8, 33, 608, 2432, 2433, 4865, 9731):
        got = to_np(fq.twist(f, torch.from_numpy(s[:n].copy()).cuda(), p))
        _same(got, {k: v[:n] for k, v in ref.items()}, ("Tw", "length", "r1", "r2", "face1", "face2", "status", "steps"))
    f.close()


@pytest.mark.parametrize("max_steps", [1, 5, 13, 29])
@pytest.mark.parametrize("nu,nv", [(1, 1), (3, 1), (11, 7)])
def test_step_budgets_on_an_interior_plane(max_steps, nu, nv):
    fq, f, B, g, lo, hi = _field("aniso")
    pl = ((0.0, 0.37 * hi[1], 0.0), (hi[0] / nu, 0.0, 0.0), (0.0, 0.0, hi[2] / nv), nu, nv)
    ref = oracle.plane(B, g, *pl, oracle.params(max_steps=max_steps))
    got = to_np(fq.qmap_plane(f, *pl, fq.params(precision="f64", max_steps=max_steps)))
    _same(got, ref, ("Q", "Tw", "length", "r1", "r2", "face1", "face2", "status", "steps"))
    f.close()
