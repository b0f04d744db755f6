"""Where every seed of a small interior map is rotated there are four extra lines
to each of its lines, and lanes enough have to take them: such a map may not be
slower than with whole warps (FP32), nor than one of more seeds, which has more
lanes of each warp at work (FP64). A sixth is allowed for noise."""
import pytest
import torch

pytestmark = pytest.mark.gpu

N = (128, 128, 64)


def _ms(fns, reps=11):
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


def _field(dtype, pack):
    import paper_2208_12569_gb300 as fq

    z, y, x = torch.meshgrid(*[torch.arange(k, dtype=dtype, device="cuda") for k in N[::-1]], indexing="ij")
    B = torch.stack((1.0 + 0.0 * x, 0.3 + 0.001 * x, 0.004 * (z - N[2] / 2) + 0.03), -1)
    return fq, fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=(pack,))


def _call(fq, f, m, **kw):
    p, out = fq.params(**kw), fq.alloc_out(m * m)
    return lambda: fq.qmap_plane(f, (0.0, 0.0, 31.51), (127.0 / m, 0.0, 0.0), (0.0, 127.0 / m, 0.0), m, m, p=p, out=out)


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("m", [40, 48, 64])
def test_fp32(m, scheme):
    fq, f = _field(torch.float32, "f32")
    few, whole = [_call(fq, f, m, precision="f32", scheme=scheme, chunk_tiles=c) for c in (0, 1)]
    out, ref = few(), whole()
    assert bool((out["status"] & fq.LINE_ROTATED).all())
    for k in out:
        assert out[k].cpu().numpy().tobytes() == ref[k].cpu().numpy().tobytes(), k
    a, b = _ms([few, whole])
    assert a < 7 / 6 * b, (a, b)
    f.close()


@pytest.mark.parametrize("scheme", [0, 1])
def test_fp64(scheme):
    fq, f = _field(torch.float64, "f64")
    a, b = _ms([_call(fq, f, m, precision="f64", scheme=scheme) for m in (48, 50)])
    assert a < 7 / 6 * b, (a, b)
    f.close()
