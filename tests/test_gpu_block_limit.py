"""FP32 launches over a large cube hold fewer resident blocks only where their
lines share few cells. Seeds a cell apart share them: such a call may not be
slower than with as many blocks as fit (a sixteenth is allowed for noise), and
neither may seeds four cells apart. A plane two cells apart has to be faster."""
import pytest
import torch

pytestmark = pytest.mark.gpu

N = (1024, 512, 86)  # 1.44e9 bytes of records


@pytest.fixture(scope="module")
def field():
    import paper_2208_12569_gb300 as fq

    z, y, x = torch.meshgrid(*[torch.arange(k, dtype=torch.float32, device="cuda") for k in N[::-1]], indexing="ij")
    B = torch.zeros((N[2], N[1], N[0], 3), dtype=torch.float32, device="cuda")
    g = torch.Generator().manual_seed(4)
    for q in torch.rand((24, 4), generator=g).tolist():  # buried sources of both signs
        d = torch.stack((x - q[0] * N[0], y - q[1] * N[1], z + 6.0 + 40.0 * q[2]), -1)
        B += (q[3] - 0.5) * d / d.square().sum(-1, keepdim=True).pow(1.5)
    f = fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f32",))
    yield fq, f
    f.close()


def _ms(fns, reps=9):
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


def _calls(fq, call):
    return [lambda p=fq.params(precision="f32", blocks_per_sm=b): call(p) for b in (0, 8)]


@pytest.mark.parametrize("shape,apart", [("plane", 1.0), ("plane", 1.3), ("plane", 1.99), ("plane", 4.0), ("volume", 1.0),
                                         ("volume", 1.3), ("volume", 4.0)])
def test_lattice(field, shape, apart):
    fq, f = field
    w, h = min(800, int((N[0] - 2) / apart)), min(500, int((N[1] - 2) / apart))
    if shape == "plane":
        out = fq.alloc_out(w * h)

        def call(p):
            fq.qmap_plane(f, (0.2, 0.2, 21.8), (apart, 0.0, 0.0), (0.0, apart, 0.0), w, h, p=p, out=out)
    else:
        w, h, d = 96, 96, min(40, int((N[2] - 2) / apart))
        out = fq.alloc_out(w * h * d)

        def call(p):
            fq.qmap_volume(f, (0.2, 0.2, 0.2), (apart,) * 3, w, h, d, p=p, out=out)
    limited, free = _ms(_calls(fq, call))
    assert limited < (0.97 if apart == 1.99 else 1.0625) * free, (limited, free)


def _rows(apart):
    w, h = min(600, int((N[0] - 2) / apart)), min(500, int((N[1] - 2) / apart))
    j, i = torch.meshgrid(torch.arange(h), torch.arange(w), indexing="ij")
    return torch.stack((apart * i + 0.3, apart * j + 0.4, torch.full_like(i, 21.8, dtype=torch.float64)), -1).double().reshape(-1, 3)


def _curves(g):
    d = torch.randn((300, 1, 3), generator=g, dtype=torch.float64)
    s = 0.3 * d / d.norm(dim=-1, keepdim=True) * torch.arange(1000.0).view(1, -1, 1)
    s = s + torch.rand((300, 1, 3), generator=g, dtype=torch.float64) * torch.tensor(N, dtype=torch.float64)
    return s.reshape(-1, 3).remainder(torch.tensor(N, dtype=torch.float64) - 1.0)


@pytest.mark.parametrize("order", ["rows 0.5", "rows 1", "curves", "rows 3", "rows 1 shuffled"])
def test_list(field, order):
    fq, f = field
    g = torch.Generator().manual_seed(1)
    seeds = _curves(g) if order == "curves" else _rows(float(order.split()[1]))
    if "shuffled" in order:
        seeds = seeds[torch.randperm(seeds.shape[0], generator=g)]
    seeds = seeds.cuda()
    out = [fq.alloc_out(seeds.shape[0], q=False) for _ in range(2)]
    fns = [lambda p=fq.params(precision="f32", blocks_per_sm=b), o=o: fq.twist(f, seeds, p, o) for b, o in zip((0, 8), out)]
    limited, free = _ms(fns)
    # rows 3 cells apart and scattered seeds run with fewer blocks, which has to pay
    assert limited < (0.95 if order in ("rows 3", "rows 1 shuffled") else 1.0625) * free, (limited, free)
    for k, t in out[0].items():
        if t is not None:
            assert t.cpu().numpy().tobytes() == out[1][k].cpu().numpy().tobytes(), k
