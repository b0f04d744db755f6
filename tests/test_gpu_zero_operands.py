"""Exact zeros (a field component that vanishes everywhere, the curl of a
current-free field, the error of a straight line's step) are ordinary operands
of the FP64 tracer and of the gradient grid. Work on a field that holds them
may take no longer than on the same field with 1e-9 in their place, which takes
the same steps: a quarter is allowed for the noise of the clock."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ms(fns, reps=9):
    """Median times of the functions, run in turn."""
    ts = [[] for _ in fns]
    for k in range(reps + 2):
        for t, fn in zip(ts, fns):
            e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e[0].record()
            fn()
            e[1].record()
            torch.cuda.synchronize()
            if k >= 2:
                t.append(e[0].elapsed_time(e[1]))
    return [sorted(t)[reps // 2] for t in ts]


def _cubes(n, b):
    """The constant field b, and the same with a small field of nonzero curl
    whose three components vanish nowhere."""
    z, y, x = torch.meshgrid(*[torch.arange(1.0, k + 1.0, dtype=torch.float64, device="cuda") for k in n[::-1]], indexing="ij")
    B = torch.tensor(b, dtype=torch.float64, device="cuda").expand(n[2], n[1], n[0], 3).contiguous()
    return B, B + 1e-9 * torch.stack((y + 2 * z, z + 3 * x, x + 5 * y), -1)


@pytest.mark.parametrize("grid", ["unit", "aniso", "stretched"])
@pytest.mark.parametrize("b", [(0.25, 0.125, 1.0), (0.0, 0.0, 1.0)])
def test_fp64_map(grid, b):
    import paper_2208_12569_gb300 as fq

    n, m = (64, 64, 32), 256
    d = (0.5, 0.25, 0.75) if grid == "aniso" else (1.0, 1.0, 1.0)
    fields = []
    for B in _cubes(n, b):
        if grid == "stretched":
            coords = [[0.0] + [i * (1.0 + 0.001 * i) for i in range(1, k)] for k in n]
            fields.append(fq.Field(B, coords=coords, pack=("f64",)))
            hi = [c[-1] for c in coords]
        else:
            fields.append(fq.Field(B, (0.0, 0.0, 0.0), d, pack=("f64",)))
            hi = [(k - 1) * v for k, v in zip(n, d)]
    p = fq.params(precision="f64")
    out = fq.alloc_out(m * m)
    pl = dict(origin=(0.0, 0.0, 0.0), u=(hi[0] / m, 0.0, 0.0), v=(0.0, hi[1] / m, 0.0), nu=m, nv=m)
    zero, small = _ms([lambda f=f: fq.qmap_plane(f, p=p, out=out, **pl) for f in fields])
    assert zero < 1.25 * small, (zero, small)
    for f in fields:
        f.close()


def test_gradient_grid():
    import paper_2208_12569_gb300 as fq

    n = (256, 128, 64)
    fns, fields = [], []
    for B in _cubes(n, (0.0, 0.0, 1.0)):
        f = fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f64", "gradb"))
        fields.append(f)
        fns.append(lambda f=f, B=B: [f.update(B) for _ in range(4)])
    zero, small = _ms(fns)
    assert zero < 1.25 * small, (zero, small)
    for f in fields:
        f.close()
