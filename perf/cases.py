"""The work that a user of this framework has it do, as cases to time.

Every case goes through the public binding: seed lists (twist), Q/Tw maps on
planes and volumes (Methods I and II, both step schemes, FP32, FP32 with FP64
sums and FP64, uniform and stretched grids), a batch of uneven cubes, a time
series step (repack + map) and a gradient step (repack + taped map + loss +
reverse sweep). The fields are sums of buried point monopoles over the cube,
the stand-in for an extrapolated active-region field, with a rigid-twist tube
added where the twist matters.
"""
import math
import random

import torch

import paper_2208_12569_gb300 as fq

DEV = "cuda"

# cube sizes of the batched workload
BATCH_CUBES = ((64, 64, 64), (128, 128, 64), (256, 256, 128), (384, 384, 192))


def listed():
    base = dict(nx=256, ny=256, nz=128, spacing="unit", cut="bottom", precision="f32", method=1, scheme=0)
    return [
        # a few lines picked by hand to be drawn or measured: latency and launches count
        dict(base, name="twist-few", kind="twist", nx=64, ny=64, nz=64, seeds=37),
        # a quick look: the small test cube, the plane at 2x its nodes
        dict(base, name="plane-small", kind="plane", nx=64, ny=64, nz=64, nu=128, nv=128, spacing="aniso"),
        # the headline map: 4x oversampled bottom plane of a 256x256x128 cube
        dict(base, name="plane-1024", kind="plane", nu=1024, nv=1024),
        # the same cube in FP64, the precision that reproduces the method to the last bit
        dict(base, name="plane-f64", kind="plane", nu=512, nv=512, precision="f64"),
        # a vertical cut through an odd-sized cube: interior seeds rotate S0 and trace extra lines
        dict(base, name="slice-acc64", kind="plane", nx=301, ny=151, nz=76, nu=601, nv=151, cut="xz", spacing="aniso",
             precision="f32acc64"),
        # Method II with the gradient grid, Q_perp (the paper's deviation-vector setting)
        dict(base, name="deviation-way1", kind="plane", nu=512, nv=384, method=2, way=1, qperp=1),
        # Method II by differences around the line: no gradient grid to store
        dict(base, name="deviation-way2", kind="plane", nu=384, nv=256, method=2, way=2, qperp=0),
        # an extrapolation grid whose cells grow upward and outward
        dict(base, name="stretched", kind="plane", nu=768, nv=512, spacing="stretched"),
        # Q in a volume: every layer its own S0, lines through a cube larger than L2
        dict(base, name="volume", kind="volume", nx=512, ny=512, nz=256, nu=96, nv=96, nw=48),
        # many cubes of uneven sizes in one set of launches
        dict(base, name="batch", kind="batch", count=7, mix=3, nu=512, nv=256),
        # a time series: each snapshot is repacked, then mapped
        dict(base, name="series", kind="series", nu=400, nv=300),
        # one step of an inversion: repack, taped map, loss, gradient with respect to B
        dict(base, name="gradient", kind="gradient", nx=128, ny=128, nz=64, nu=256, nv=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("twist", "plane", "plane", "plane", "plane", "volume", "batch", "series", "gradient"))
    big = dict(twist=256, plane=320, volume=448, batch=0, series=288, gradient=160)[kind]
    c = dict(kind=kind, spacing=rng.choice(("unit", "unit", "aniso", "stretched")), cut=rng.choice(("bottom", "bottom", "xz")),
             precision=rng.choice(("f32", "f32", "f32", "f32acc64", "f64")), method=1, scheme=rng.choice((0, 0, 0, 1)))
    if kind == "batch":
        c.update(nx=256, ny=256, nz=128, spacing=rng.choice(("unit", "aniso")), count=rng.randint(2, 7), mix=rng.randint(0, 999),
                 nu=_log_int(rng, 32, 512), nv=_log_int(rng, 32, 256), precision=rng.choice(("f32", "f32", "f32acc64")))
    else:
        c["nx"] = _log_int(rng, 32, big)
        c["ny"] = max(24, min(big, int(c["nx"] * rng.uniform(0.5, 1.2))))
        c["nz"] = max(20, int(c["nx"] * rng.uniform(0.4, 0.8)))
    if kind == "twist":
        c["seeds"] = _log_int(rng, 1, 100000)
    elif kind == "volume":
        c.update(nu=_log_int(rng, 8, 96), nv=_log_int(rng, 8, 96), nw=_log_int(rng, 4, 48))
    elif kind == "gradient":
        c.update(nu=_log_int(rng, 16, 256), nv=_log_int(rng, 16, 256), cut="bottom")
    elif kind != "batch":
        c.update(nu=_log_int(rng, 16, 1024), nv=_log_int(rng, 16, 1024))
        if rng.random() < 0.3:
            c.update(method=2, way=rng.choice((1, 2)), qperp=rng.choice((0, 1)))
            if c["precision"] == "f32acc64":
                c["precision"] = "f32"  # Method II has one FP32 form
    # keep the map below the largest listed ones, by estimated device time
    size = ("seeds",) if kind == "twist" else ("nu", "nv") + (("nw",) if kind == "volume" else ())
    while _cost(c) > MOST_COST:
        k = max(size, key=lambda s: c[s])
        c[k] = max(1, int(c[k] * 0.8))
    return c


# ---------------------------------------------------------------------------
# the work of a case
# ---------------------------------------------------------------------------
def _batch_parts(case):
    """The entries of a batch: (nx, ny, nz), charges, cut."""
    r = random.Random(case["mix"])
    return [(r.choice(BATCH_CUBES), r.randint(8, 64), r.choice(("bottom", "xz"))) for _ in range(case["count"])]


def _parts(case):
    """(nodes, lines, trial steps a line) of each map of the case. Lines from
    the bottom plane mostly close low down (about 18 trials), lines from inside
    cross the cube."""
    if case["kind"] == "batch":
        got = [(n, case["nu"] * case["nv"], cut) for n, _, cut in _batch_parts(case)]
    else:
        n = (case["nx"], case["ny"], case["nz"])
        if case["kind"] == "twist":
            got = [(n, case["seeds"], "inside")]
        elif case["kind"] == "volume":
            got = [(n, case["nu"] * case["nv"] * case["nw"], "inside")]
        else:
            got = [(n, case["nu"] * case["nv"], case["cut"])]
    return [(n[0] * n[1] * n[2], m, 18.0 if cut == "bottom" else 12.0 + 0.2 * (n[0] + n[1] + n[2]) / 3.0) for n, m, cut in got]


def work(case):
    f64 = case["precision"] == "f64"
    stages = 4 if case["scheme"] else 6
    trials = 2.6 if case["scheme"] else 1.0
    # per stage: 8 corners x 6 components, the weights and the right-hand side;
    # Method II: 9 more components (way 1) or 6 more points (way 2)
    per = 165.0
    if case["method"] == 2:
        per = 360.0 if case["way"] == 1 else 700.0
    nbytes = flops = 0.0
    for nodes, lines, t in _parts(case):
        out = lines * (71 if case["kind"] == "twist" else 79)
        nbytes += nodes * (24 if f64 else 12) + out
        flops += lines * t * trials * stages * per
        if case["kind"] == "gradient":
            nbytes += nodes * (24 if f64 else 12) + 16 * lines
            flops *= 4
        if case["kind"] in ("series", "gradient"):
            flops += 18.0 * nodes
    return dict(bytes=nbytes, flops=flops)


def _cost(case):
    """Estimated device time (arbitrary units): FP64 runs at a small fraction of the FP32 rate."""
    return work(case)["flops"] * (45.0 if case["precision"] == "f64" else 1.0)


MOST_COST = max(_cost(c) for c in listed() if c["precision"] == "f64")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _axis(n, d, ratio, edges):
    if ratio == 1.0:
        return [d * i for i in range(n)]
    w = [ratio ** (abs(i - 0.5 * (n - 2)) if edges else i) for i in range(n - 1)]
    s = d * (n - 1) / sum(w)
    x = [0.0]
    for v in w:
        x.append(x[-1] + s * v)
    return x


def _coords(n, spacing):
    if spacing == "stretched":
        return [_axis(n[0], 1.0, 1.01, True), _axis(n[1], 1.0, 1.01, True), _axis(n[2], 1.0, 1.02, False)]
    return [_axis(k, d, 1.0, False) for k, d in zip(n, _spacing(spacing))]


def _spacing(spacing):
    return (0.02, 0.02, 0.03) if spacing == "aniso" else (1.0, 1.0, 1.0)


def _charges(r, n, spacing, count, scale):
    """Signed point sources below z = 0, no net flux, depths 4 to 16 cells of a 256-node footprint."""
    d = _spacing(spacing)
    q = [r.gauss(0.0, 1.0) for _ in range(count)]
    mean = sum(q) / count
    return [(r.uniform(0.0, (n[0] - 1) * d[0]), r.uniform(0.0, (n[1] - 1) * d[1]),
             -d[2] * (1.0 + scale * n[0] * r.uniform(4.0, 16.0)), v - mean) for v in q]


def _cube(n, spacing, charges, dtype, tube=False):
    x, y, z = [torch.tensor(c, dtype=torch.float64, device=DEV) for c in _coords(n, spacing)]
    B = torch.empty((n[2], n[1], n[0], 3), dtype=dtype, device=DEV)
    layers = max(1, (1 << 22) // (n[0] * n[1]))
    for k in range(0, n[2], layers):
        zk = z[k:k + layers, None, None]
        acc = [0.0, 0.0, 0.0]
        for cx, cy, cz, q in charges:
            dx, dy, dz = x - cx, (y - cy)[:, None], zk - cz
            r2 = dx * dx + dy * dy + dz * dz
            s = q / (r2 * r2.sqrt())
            acc = [acc[0] + s * dx, acc[1] + s * dy, acc[2] + s * dz]
        for c in range(3):
            B[k:k + layers, :, :, c] = acc[c]
    if tube:  # a vertical rigid-twist flux tube through the middle: 1.5 turns over the height
        xp, yp = x - 0.5 * (x[0] + x[-1]), (y - 0.5 * (y[0] + y[-1]))[:, None]
        rad = 10.0 / 128.0 * (x[-1] - x[0])
        w = B[0].double().square().sum(-1).mean().sqrt() * torch.exp(-(xp * xp + yp * yp) / (rad * rad))
        q = 2.0 * math.pi * 1.5 / (z[-1] - z[0])
        for c, t in enumerate((-q * yp * w, q * xp * w, w)):
            B[..., c] += t.to(dtype)
    return B


def _field(B, n, spacing, pack):
    if spacing == "stretched":
        return fq.Field(B, coords=_coords(n, spacing), pack=pack)
    return fq.Field(B, (0.0, 0.0, 0.0), _spacing(spacing), pack=pack)


def _plane(n, spacing, cut, nu, nv):
    """Seed plane over the whole bottom, or over the vertical cut at mid-y."""
    x, y, z = _coords(n, spacing)
    if cut == "bottom":
        return dict(origin=(0.0, 0.0, 0.0), u=(x[-1] / nu, 0.0, 0.0), v=(0.0, y[-1] / nv, 0.0), nu=nu, nv=nv)
    return dict(origin=(0.0, 0.5 * y[-1], 0.0), u=(x[-1] / nu, 0.0, 0.0), v=(0.0, 0.0, z[-1] / nv), nu=nu, nv=nv)


def _params(case, **kw):
    p = dict(precision=case["precision"], method=case["method"], scheme=case["scheme"])
    if case["method"] == 2:
        p.update(gradb_way=case["way"], qperp=case["qperp"])
    if case["scheme"]:
        p.update(step=4.0 if case["method"] == 2 else 3.0)
    return fq.params(**p, **kw)


def _inputs(case, seed):
    """The case's inputs from the seed: cubes and seed points."""
    r = random.Random(1000003 * seed + 17)
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    if case["kind"] == "batch":
        parts = _batch_parts(case)
        cubes = [_cube(n, case["spacing"], _charges(r, n, case["spacing"], count, 1.0 / 256.0), dtype) for n, count, _ in parts]
        return dict(cubes=cubes, planes=[_plane(n, case["spacing"], cut, case["nu"], case["nv"]) for n, _, cut in parts],
                    sizes=[n for n, _, _ in parts])
    n = (case["nx"], case["ny"], case["nz"])
    ch = _charges(r, n, case["spacing"], 24, 1.0 / 128.0 if case["kind"] == "gradient" else 1.0 / 256.0)
    tube = case["kind"] in ("twist", "gradient")
    got = dict(n=n, B=_cube(n, case["spacing"], ch, dtype, tube))
    if case["kind"] == "gradient":  # the map to be fitted: the same sources, 5 % off in strength
        other = [(a, b, c, q * (1.0 + 0.05 * r.gauss(0.0, 1.0))) for a, b, c, q in ch]
        got["target"] = _cube(n, case["spacing"], other, dtype, tube)
    if case["kind"] == "series":  # the snapshot before
        other = [(a, b, c, q * (1.0 + 0.05 * r.gauss(0.0, 1.0))) for a, b, c, q in ch]
        got["before"] = _cube(n, case["spacing"], other, dtype, tube)
    if case["kind"] == "twist":
        hi = [c[-1] for c in _coords(n, case["spacing"])]
        g = torch.Generator().manual_seed(seed)
        s = torch.rand((case["seeds"], 3), generator=g, dtype=torch.float64)
        s[:, 2] *= 0.5  # in the lower half, where the closed lines are
        got["seeds"] = (s * torch.tensor(hi, dtype=torch.float64)).to(DEV)
    elif case["kind"] == "volume":
        m = (case["nu"], case["nv"], case["nw"])
        got["step"] = tuple(c[-1] / k for c, k in zip(_coords(n, case["spacing"]), m))
    else:
        got["plane"] = _plane(n, case["spacing"], case["cut"], case["nu"], case["nv"])
    return got


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    pack = ("f64",) if case["precision"] == "f64" else ("f32",)
    if case["method"] == 2 and case["way"] == 1:
        pack += ("gradb",)
    if case["kind"] == "batch":
        s["fields"] = [_field(B, n, case["spacing"], pack) for B, n in zip(s["cubes"], s["sizes"])]
        s["batch"] = fq.Batch(s["fields"], s["planes"], _params(case))
        return s
    s["field"] = _field(s["before"] if case["kind"] == "series" else s["B"], s["n"], case["spacing"], pack)
    s["p"] = _params(case, tape=1) if case["kind"] == "gradient" else _params(case)
    if case["kind"] == "gradient":
        f = _field(s["target"], s["n"], case["spacing"], pack)
        t = fq.qmap_plane(f, p=_params(case), **s["plane"])
        s["Qt"], s["Twt"] = t["Q"], t["Tw"]
        torch.cuda.synchronize()
        f.close()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "twist":
        return fq.twist(s["field"], s["seeds"], s["p"])
    if kind == "volume":
        return fq.qmap_volume(s["field"], (0.0, 0.0, 0.0), s["step"], case["nu"], case["nv"], case["nw"], s["p"])
    if kind == "batch":
        return s["batch"].run()
    if kind == "plane":
        return fq.qmap_plane(s["field"], p=s["p"], **s["plane"])
    s["field"].update(s["B"])
    out = fq.qmap_plane(s["field"], p=s["p"], **s["plane"])
    if kind == "series":
        return out
    loss, dQ, dTw = fq.loss_logq_tw(out["Q"], out["Tw"], s["Qt"], s["Twt"], out["status"])
    dB = fq.backward(s["field"], dQ, dTw, dtype=s["B"].dtype)
    return dict(Q=out["Q"], Tw=out["Tw"], loss=loss, dB=dB)


# ---------------------------------------------------------------------------
# the same in 64 bits: a plain torch evaluation of the method, line by line
# ---------------------------------------------------------------------------
_RKF_A = ((), (1 / 4,), (3 / 32, 9 / 32), (1932 / 2197, -7200 / 2197, 7296 / 2197), (439 / 216, -8.0, 3680 / 513, -845 / 4104),
          (-8 / 27, 2.0, -3544 / 2565, 1859 / 4104, -11 / 40))
_RKF_B4 = (25 / 216, 0.0, 1408 / 2565, 2197 / 4104, -1 / 5, 0.0)
_RKF_B5 = (16 / 135, 0.0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55)
_K38_A = ((), (1 / 3,), (-1 / 3, 1.0), (1.0, -1.0, 1.0))
_K38_B = (1 / 8, 3 / 8, 3 / 8, 1 / 8)
_LONGEST = 2500  # trial steps after which the reference gives up (it would take too long)


class _Lines:
    """Field lines of one cube. Positions are in cells on a uniform grid and
    physical on a stretched one."""

    def __init__(self, B, n, spacing):
        B = B.double()
        xyz = _coords(n, spacing)
        self.rect = spacing == "stretched"
        t = [torch.tensor(c, dtype=torch.float64, device=DEV) for c in xyz]
        sp = [t[2], t[1], t[0]] if self.rect else [_spacing(spacing)[a] for a in (2, 1, 0)]
        g = [torch.gradient(B[..., c], spacing=sp, edge_order=2) for c in range(3)]  # g[c] = d/dz, d/dy, d/dx
        J = torch.stack((g[2][1] - g[1][0], g[0][0] - g[2][2], g[1][2] - g[0][1]), -1)
        self.rec = torch.cat((B, J), -1).reshape(-1, 6)
        self.n, self.axes = n, t
        self.d = torch.tensor(_spacing(spacing), dtype=torch.float64, device=DEV)
        self.lo = torch.zeros(3, dtype=torch.float64, device=DEV)
        self.hi = torch.stack([c[-1] for c in t]) if self.rect else torch.tensor([k - 1.0 for k in n], dtype=torch.float64, device=DEV)

    def cells(self, x):
        """Lower cell index and its weight omega_0 on the three axes, and the cells' widths."""
        c, w, d = [], [], []
        for a in range(3):
            p = x[:, a].contiguous()
            if self.rect:
                ax = self.axes[a]
                i = (torch.searchsorted(ax, p, right=True) - 1).clamp(0, self.n[a] - 2)
                d.append(ax[i + 1] - ax[i])
                w.append((ax[i + 1] - p) / d[a])
            else:
                f = p.floor().clamp(0.0, self.n[a] - 2.0)
                i = f.long()
                d.append(self.d[a].expand_as(p))
                w.append((f + 1.0) - p)
            c.append(i)
        return c, w, torch.stack(d, 1)

    def at(self, x):
        c, w, _ = self.cells(x)
        base = (c[2] * self.n[1] + c[1]) * self.n[0] + c[0]
        v = 0.0
        for i in range(2):
            for j in range(2):
                for k in range(2):
                    wt = (w[0] if i == 0 else 1.0 - w[0]) * (w[1] if j == 0 else 1.0 - w[1]) * (w[2] if k == 0 else 1.0 - w[2])
                    v = v + wt[:, None] * self.rec[base + (k * self.n[1] + j) * self.n[0] + i]
        return v[:, :3], v[:, 3:]

    def rhs(self, x, D, sgn):
        B, J = self.at(x)
        bt = B / D
        bb, BB = (bt * bt).sum(1), (B * B).sum(1)
        ok = (bb > 0) & (bb < math.inf)
        nbt = bb.sqrt()
        F = sgn[:, None] * (B if self.rect else bt) / nbt[:, None]
        dl = BB.sqrt() / nbt
        dtw = (J * B).sum(1) / (4.0 * math.pi * BB) * dl
        return torch.cat((F, dl[:, None], dtw[:, None]), 1), ok

    def state_of(self, r):
        return r if self.rect else r / self.d

    def phys_of(self, x):
        return x if self.rect else x * self.d

    def trace(self, x0, sgn, ctl, scheme):
        """Every line from x0 along sgn B to its end: (end, face, length, Tw); a line on a null field has NaN sums.
        None where lines are too long."""
        m = len(x0)
        A, B4, B5 = (_K38_A, _K38_B, None) if scheme else (_RKF_A, _RKF_B4, _RKF_B5)
        hmin, hmax, graze = 1e-6, 4.0, 1e-3
        f8 = dict(dtype=torch.float64, device=DEV)
        end, face = x0.clone(), torch.full((m,), -1, device=DEV)
        length, tw = torch.full((m,), math.nan, **f8), torch.full((m,), math.nan, **f8)
        lim = torch.stack((self.lo, self.hi), 1).reshape(-1)  # by face
        S = dict(id=torch.arange(m, device=DEV), x=x0.clone(), sgn=sgn.clone(), tol=ctl.clone(), h=ctl.clone() if scheme else torch.full((m,), 0.5, **f8),
                 acc=torch.zeros((m, 2), **f8), hen=torch.zeros(m, dtype=torch.bool, device=DEV), face=torch.zeros(m, dtype=torch.long, device=DEV),
                 tries=torch.zeros(m, dtype=torch.long, device=DEV), out=torch.zeros((m, 5), **f8), t0=torch.zeros(m, **f8), f0=torch.zeros(m, dtype=torch.long, device=DEV))
        for _ in range(_LONGEST):
            if not len(S["id"]):
                return end, face, length, tw
            x, h, hen, fc = S["x"], S["h"], S["hen"], S["face"]
            ax = fc // 2
            pick = lambda v: v.gather(1, ax[:, None])[:, 0]  # noqa: E731
            side = torch.where(fc % 2 == 1, 1.0, -1.0).double()
            hh = torch.where(hen, lim[fc] - pick(x), h)
            D = self.cells(x)[2]
            k, fine, flat = [], torch.ones_like(hen), torch.zeros_like(hen)
            for s in range(len(A)):
                p = 0.0
                for q in range(s):
                    p = p + A[s][q] * k[q][:, :3]
                o, ok = self.rhs(x + hh[:, None] * p if s else x, D, S["sgn"])
                fa = pick(o[:, :3])
                low = hen & ~((fa / pick(D) if self.rect else fa) * side >= graze)
                flat |= fine & ok & low  # the first failing stage says what failed
                fine &= ok | flat
                k.append(torch.where((hen & ~low)[:, None], o / torch.where(low, 1.0, fa)[:, None], o))
            a4 = sum(B4[s] * k[s] for s in range(len(k)) if B4[s])
            new = x + hh[:, None] * a4[:, :3]
            sums = hh[:, None] * a4[:, 3:]
            step = fine & ~hen
            if scheme:
                over, hn = torch.zeros_like(hen), h
            else:
                a5 = sum(B5[s] * k[s][:, :3] for s in range(len(k)) if B5[s])
                e = (x + hh[:, None] * a5) - new
                err = (e / D if self.rect else e).square().sum(1).sqrt()
                q = 0.9 * (S["tol"] / err).sqrt().sqrt()
                over = step & (err > S["tol"]) & (h > hmin)
                hn = torch.where(over, h * q.clamp(min=0.1), h * torch.where(err > 0, q.clamp(max=4.0), torch.full_like(q, 4.0)))
                hn = hn.clamp(hmin, hmax)
            inside = ((new >= self.lo) & (new <= self.hi)).all(1)
            go, leave = step & ~over & inside, step & ~over & ~inside
            # the first face that the chord crosses
            t = torch.full((len(x), 6), math.inf, **f8)
            for a in range(3):
                t[:, 2 * a] = torch.where(new[:, a] < self.lo[a], (self.lo[a] - x[:, a]) / (new[:, a] - x[:, a]), math.inf)
                t[:, 2 * a + 1] = torch.where(new[:, a] > self.hi[a], (self.hi[a] - x[:, a]) / (new[:, a] - x[:, a]), math.inf)
            tmin, first = t.min(1)
            # exit steps: onto the face, or back with half the step, or along the chord
            land = fine & hen & ~flat
            at = new.scatter(1, ax[:, None], lim[fc][:, None])
            off = torch.stack([(at[:, a // 2] < self.lo[a // 2]) if a % 2 == 0 else (at[:, a // 2] > self.hi[a // 2]) for a in range(6)], 1)
            off &= torch.arange(6, device=DEV)[None] // 2 != ax[:, None]
            again = land & off.any(1) & (S["tries"] < 2)
            done = land & ~again
            back = hen & flat & fine
            chord = back & ~(0.5 * h >= hmin)
            f0 = S["f0"]
            on = (x + S["t0"][:, None] * (S["out"][:, :3] - x)).scatter(1, (f0 // 2)[:, None], lim[f0][:, None])
            stop = done | chord | ~fine
            i = S["id"][stop]
            end[i] = torch.where(done[:, None], at.clamp(self.lo, self.hi), torch.where(chord[:, None], on, x))[stop]
            face[i] = torch.where(done, fc, torch.where(chord, f0, -1))[stop]
            total = S["acc"] + torch.where(done[:, None], sums, S["t0"][:, None] * S["out"][:, 3:])
            total = torch.where(fine[:, None], total, math.nan)
            length[i], tw[i] = total[stop, 0], total[stop, 1]
            S["out"] = torch.where(leave[:, None], torch.cat((new, sums), 1), S["out"])
            S["t0"], S["f0"] = torch.where(leave, tmin, S["t0"]), torch.where(leave, first, f0)
            S["face"] = torch.where(leave, first, torch.where(again, off.long().argmax(1), fc))
            S["tries"] = torch.where(leave, 0, S["tries"] + again.long())
            S["hen"] = (hen | leave) & ~back
            S["x"] = torch.where(go[:, None], new, x)
            S["acc"] = torch.where(go[:, None], S["acc"] + sums, S["acc"])
            S["h"] = torch.where(go | over, hn, torch.where(back & ~chord, 0.5 * h, h))
            keep = ~stop
            S = {a: v[keep] for a, v in S.items()}
        return None

    def both(self, r0, normal, case, method):
        """The lines of physical seeds r0 (n, 3) both ways: footpoints, faces, length, Tw and B at the seeds."""
        x0 = self.state_of(r0)
        B0 = self.at(x0)[0]
        nB = B0.square().sum(1).sqrt()
        s0 = torch.ones_like(nB)
        perp = 10.0 ** -3.2
        if case["scheme"]:
            perp = 4.0 if method == 2 else 3.0
        ctl = torch.full_like(nB, perp)
        if normal is not None:
            a, sign, on_face = normal
            s0 = torch.where(B0[:, a] * sign < 0, -1.0, 1.0).double()
            if method == 1:
                ratio = B0[:, a].abs() / nB
                scaled = (perp * ratio).clamp(min=0.15) if case["scheme"] else perp * ratio.clamp(min=0.05) ** 1.5
                ctl = scaled if on_face else torch.where(ratio < 0.05, ctl, scaled)
        one, two = self.trace(x0, -s0, ctl, case["scheme"]), None
        if one is not None:
            two = self.trace(x0, s0, ctl, case["scheme"])
        if two is None:
            return None
        return dict(r1=self.phys_of(one[0]), r2=self.phys_of(two[0]), f1=one[1], f2=two[1], length=one[2] + two[2], Tw=one[3] + two[3], B0=B0)

    def q_bottom(self, m, nu, nv, du, dv):
        """Method I on the bottom plane: differences of neighbouring footpoints on the same face."""
        J = []
        for r, f in ((m["r1"], m["f1"]), (m["r2"], m["f2"])):
            a = f // 2
            uv = torch.stack((torch.where(a == 0, r[:, 1], r[:, 0]), torch.where(a == 2, r[:, 1], r[:, 2])), 1).reshape(nv, nu, 2)
            f = f.reshape(nv, nu)
            cols = []
            for dim, d in ((1, du), (0, dv)):
                p, q = torch.roll(uv, -1, dim), torch.roll(uv, 1, dim)
                okp, okq = torch.roll(f, -1, dim) == f, torch.roll(f, 1, dim) == f
                okp.select(dim, -1).fill_(False)
                okq.select(dim, 0).fill_(False)
                mixed = torch.where(okp[..., None], (p - uv) / d, torch.where(okq[..., None], (uv - q) / d, math.nan))
                cols.append(torch.where((okp & okq)[..., None], (p - q) / (2.0 * d), mixed))
            J.append(torch.stack(cols, -1).reshape(-1, 2, 2))
        a, b = J
        adj = torch.stack((torch.stack((a[:, 1, 1], -a[:, 0, 1]), 1), torch.stack((-a[:, 1, 0], a[:, 0, 0]), 1)), 1)
        norm2 = (b @ adj).square().sum((1, 2))
        bn = [self.at(self.state_of(r))[0].gather(1, (f // 2).clamp(min=0)[:, None])[:, 0] for r, f in ((m["r1"], m["f1"]), (m["r2"], m["f2"]))]
        Q = norm2 * (bn[0] * bn[1]).abs() / m["B0"][:, 2].square()
        return torch.where((m["f1"] < 0) | (m["f2"] < 0), math.nan, Q)


def _lattice(origin, steps, counts):
    r = torch.zeros((1, 3), dtype=torch.float64, device=DEV) + torch.tensor(origin, dtype=torch.float64, device=DEV)
    for a, k in zip(reversed(steps), reversed(counts)):
        t = (torch.arange(k, dtype=torch.float64, device=DEV) + 0.5)[:, None] * torch.tensor(a, dtype=torch.float64, device=DEV)
        r = (r[:, None, :] + t[None]).reshape(-1, 3)
    return r


def exact(case, seed):
    """Footpoints, length and Tw of every line in 64 bits, and Q of FP64 maps of
    the bottom plane. FP32 maps have no value of Q to be held to: lines beside
    a separatrix take other steps in other roundings, and the norm of all Q is
    theirs. The same goes for gradients, which are taken along the steps that
    the traced map took."""
    s = _inputs(case, seed)
    names = ("Q", "Tw", "length", "r1", "r2", "face1", "face2", "status", "steps")

    def lines(L, r0, normal):
        m = L.both(r0, normal, case, case["method"])
        return None if m is None else dict({k: None for k in names}, **{k: m[k] for k in ("Tw", "length", "r1", "r2")}), m

    def plane(B, n, pl):
        normal = (2, 1.0, True) if pl["v"][1] else (1, -1.0, False)  # unit(u x v)
        L = _Lines(B, n, case["spacing"])
        got, m = lines(L, _lattice(pl["origin"], (pl["u"], pl["v"]), (pl["nu"], pl["nv"])), normal)
        if got is not None and case["precision"] == "f64" and normal[2] and case["method"] == 1:
            got["Q"] = L.q_bottom(m, pl["nu"], pl["nv"], pl["u"][0], pl["v"][1])
        return got

    if case["kind"] == "batch":
        got = [plane(B, n, pl) for B, n, pl in zip(s["cubes"], s["sizes"], s["planes"])]
        return None if any(g is None for g in got) else got
    if case["kind"] == "twist":
        return lines(_Lines(s["B"], s["n"], case["spacing"]), s["seeds"], None)[0]
    if case["kind"] == "volume":
        st = s["step"]
        r0 = _lattice((0.0, 0.0, 0.0), ((st[0], 0.0, 0.0), (0.0, st[1], 0.0), (0.0, 0.0, st[2])), (case["nu"], case["nv"], case["nw"]))
        return lines(_Lines(s["B"], s["n"], case["spacing"]), r0, (2, 1.0, False))[0]
    got = plane(s["B"], s["n"], s["plane"])
    if case["kind"] == "gradient" and got is not None:
        got = dict(Q=got["Q"], Tw=got["Tw"], loss=None, dB=None)
    return got
