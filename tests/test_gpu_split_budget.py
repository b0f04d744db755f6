"""A line whose second direction never leaves the box (it winds onto a closed
line) runs into max_steps. Small interior maps trace its two directions in two
lanes: the outputs are those of the same map in a batch, which uses one lane per
line, and the call takes no longer than the batch (a quarter more allowed for
noise), that is, the line's budget is traced once."""
import pytest
import torch

from parity import to_np

pytestmark = pytest.mark.gpu

N = (48, 48, 16)


def _cycle(sign):
    """B winds around the z axis of the box and away from the circle of 8 cells."""
    z, y, x = torch.meshgrid(*[torch.arange(k, dtype=torch.float64, device="cuda") for k in N[::-1]], indexing="ij")
    x, y = x - 23.4, y - 23.6
    r = (x * x + y * y).sqrt() + 0.1
    out = 0.15 * (r - 8.0) / r
    return sign * torch.stack((-y / r + out * x, x / r + out * y, 0.0 * z), -1).float()


def _ms(fns, reps=5):
    ts = [[] for _ in fns]
    for k in range(reps + 1):
        for t, fn in zip(ts, fns):
            e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e[0].record()
            fn()
            e[1].record()
            torch.cuda.synchronize()
            if k:
                t.append(e[0].elapsed_time(e[1]))
    return [sorted(t)[reps // 2] for t in ts]


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("max_steps", [100, 127, 128, 255, 300, 1000, 20000])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("precision", ["f32", "f32acc64"])
def test_trapped_second_direction(sign, max_steps, scheme, precision):
    import paper_2208_12569_gb300 as fq

    f = fq.Field(_cycle(sign), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f32",))
    # small steps: the circle's 50 cells take hundreds of trials
    p = fq.params(precision=precision, scheme=scheme, step=0.3, tol=1e-6, h0=0.4, h_max=0.4, max_steps=max_steps)
    pl = dict(origin=(26.0, 0.0, 0.0), u=(0.0, 47.0 / 19, 0.0), v=(0.0, 0.0, 15.0 / 7), nu=19, nv=7)
    b = fq.Batch([f], [pl], p)
    out = fq.alloc_out(19 * 7)
    one, ref = to_np(fq.qmap_plane(f, p=p, out=out, **pl)), to_np(b.run()[0])
    for k in ref:
        assert one[k].tobytes() == ref[k].tobytes(), k
    if max_steps == 20000:
        trapped = (ref["status"] & fq.LINE_MAXSTEPS) != 0
        second = trapped & (ref["face1"] >= 0)
        assert trapped.sum() > 10 and (second.sum() > 10 if sign > 0 else True), (trapped.sum(), second.sum())
        split, single = _ms([lambda: fq.qmap_plane(f, p=p, out=out, **pl), b.run])
        assert split < 1.25 * single, (split, single)
    b.close()
    f.close()
