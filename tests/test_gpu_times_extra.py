"""fqsl_field_times counts the rotated seeds' extra lines, their set-up included: what
a timed call takes beside its three times (the seed pre-pass and gaps) is no more
where every seed is rotated than where none is (half as much again is allowed)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("static", [False, True])
def test_set_up_of_extra_lines_is_timed(static):
    import paper_2208_12569_gb300 as fq

    n = (64, 64, 32)
    z, y, x = torch.meshgrid(*[torch.arange(k, dtype=torch.float32, device="cuda") for k in n[::-1]], indexing="ij")
    B = torch.stack((1.0 + 0.0 * x, 0.3 + 0.001 * x, 0.001 * (z - n[2] / 2)), -1)
    f = fq.Field(B, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), pack=("f32",))
    f.set_timing(True)
    m = 256 if static else 1000
    out = fq.alloc_out(m * m)
    rest = []
    for rot in (0.5, 0.0):
        p = fq.params(precision="f32", rot_thresh=rot, max_steps=1)
        got = []
        for _ in range(11):
            e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e[0].record()
            (fq.qmap_plane_static if static else fq.qmap_plane)(f, (0.0, 0.0, 15.3), (63.0 / m, 0.0, 0.0), (0.0, 63.0 / m, 0.0),
                                                                m, m, p, out=out)
            e[1].record()
            torch.cuda.synchronize()
            got.append(e[0].elapsed_time(e[1]) - sum(f.times()))
        assert bool((out["status"] & fq.LINE_ROTATED).all()) == (rot > 0)
        rest.append(sorted(got)[5])
    assert rest[0] < 1.5 * rest[1], rest
    f.close()
