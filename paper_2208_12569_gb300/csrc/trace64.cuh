// FP64 field-line tracer with eight lanes per line (Method I maps and seed
// lists, both step schemes, uniform and stretched grids, batches, the step
// tape). The method and every rounding are trace.cuh's FP64 form; what differs
// is who computes what.
//
// GB300 holds its FP64 pipe for 64 cycles per warp instruction and SM partition,
// however many lanes take part (1.06 TFLOP/s of FMAs against 71 in FP32,
// measured). With a line per lane a trial step is a chain of about 1600 such
// instructions, 50 us and more for a lone warp, and a map ends on its longest
// lines. A line's arithmetic is mostly the same operation on several
// components, so a group of eight lanes takes a line: lanes 0 to 5 interpolate
// Bx, By, Bz, Jx, Jy, Jz (8 bytes each of a corner's 64-byte record), each lane
// forms the weight of one of the eight corners, lanes 0 to 4 carry the five
// components of the right-hand side {F (3), dl/dtau, dTw/dtau} through the
// stages, lanes 0 to 2 (and 4 to 6) the position, and lanes 5 to 7 the
// 5th-order solution. Shuffles move values between the lanes; what is one
// value per line (the error, the step factor, the control flow) every lane
// computes. A trial step is then a chain of about 200 FP64-pipe instructions,
// for four lines at once. Divisions and square roots, about ten FP64
// instructions each, run on the integer pipe (soft64.cuh); products and sums
// stay on the FP64 pipe (products on the integer pipe too: 35.1 ms against 25.5
// ms for a map of 512x512 seeds in an earlier build, half of the gather's 27.2
// ms: 30 issue slots and an instruction cache that runs out cost more than 64
// cycles of a pipe that other warps leave idle).
//
// Measured against the line-per-lane form (256x256x128 cube, outputs
// bit-identical; spacing 1 / anisotropic / stretched, ms): bottom plane of
// 512x512 seeds 31.0 -> 21.5 / 30.4 -> 23.0 / 44.2 -> 35.9 (FP64 pipe 76 % busy), of
// 1024x1024 94.9 -> 80.8 / 91.4 -> 87.0 / 143 -> 139, a list of 400,000 seeds 135 ->
// 66.5 / 157 -> 84.1 / 196 -> 105. Larger planes: api.cu, line_per_lane.
#pragma once

#include "soft64.cuh"
#include "trace.cuh"

namespace fqsl {
namespace trace64 {

using soft64::div64;
using soft64::sqrt64;
using trace::sel3;

constexpr int kGroup = 8;  // lanes per line
constexpr unsigned kFull = 0xffffffffu;

// Stage coefficients [scheme][stage]: the Fehlberg pair's 4th-order form and
// the 3/8 rule; the 5th-order weights of the pair.
static __constant__ double kA[2][6][5] = {
    {{0},
     {1.0 / 4.0},
     {3.0 / 32.0, 9.0 / 32.0},
     {1932.0 / 2197.0, -7200.0 / 2197.0, 7296.0 / 2197.0},
     {439.0 / 216.0, -8.0, 3680.0 / 513.0, -845.0 / 4104.0},
     {-8.0 / 27.0, 2.0, -3544.0 / 2565.0, 1859.0 / 4104.0, -11.0 / 40.0}},
    {{0}, {1.0 / 3.0}, {-1.0 / 3.0, 1.0}, {1.0, -1.0, 1.0}, {0}, {0}}};
static __constant__ double kB[2][6] = {
    {25.0 / 216.0, 0.0, 1408.0 / 2565.0, 2197.0 / 4104.0, -1.0 / 5.0, 0.0}, {1.0 / 8.0, 3.0 / 8.0, 3.0 / 8.0, 1.0 / 8.0}};
static __constant__ double kB5[6] = {16.0 / 135.0, 0.0, 6656.0 / 12825.0, 28561.0 / 56430.0, -9.0 / 50.0, 2.0 / 55.0};

// A lane's place: its group's lanes, its number in it, and the axis whose
// position component it holds (lanes a and 4 + a: axis a; lanes 3 and 7: none)
struct Place {
    unsigned mask;
    int sub, a;
};

__device__ __forceinline__ double get(const Place &g, double v, int src)
{
    const int hi = __shfl_sync(g.mask, __double2hiint(v), src, kGroup);
    const int lo = __shfl_sync(g.mask, __double2loint(v), src, kGroup);
    return __hiloint2double(hi, lo);
}

// (v of lane src) + (v of lane src + 1) + (v of lane src + 2), left to right
__device__ __forceinline__ double sum3(const Place &g, double v, int src)
{
    return __dadd_rn(__dadd_rn(get(g, v, src), get(g, v, src + 1)), get(g, v, src + 2));
}

// x + 0.0 (-0 becomes +0)
__device__ __forceinline__ double plus_zero(double x)
{
    return __double_as_longlong(x) == (long long)0x8000000000000000ull ? 0.0 : x;
}

// 0 < x < infinity, read off the bits (a comparison would take the FP64 pipe)
__device__ __forceinline__ bool positive_finite(double x)
{
    return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull - 1ull;
}

// An integer that orders as its double does (-0 as +0); NaNs lie above
// kInfKey or below -kInfKey.
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 ? -(b & 0x7fffffffffffffffll) : b;
}
constexpr long long kInfKey = 0x7ff0000000000000ll;

// s x for s = +1 or -1
__device__ __forceinline__ double turn(double s, double x)
{
    return __hiloint2double(__double2hiint(x) ^ (__double2hiint(s) & (int)0x80000000), __double2loint(x));
}

// A lane's axis of the field: box bounds in state coordinates, spacing and
// origin, and on a stretched grid its cell tables. Lanes without an axis get a
// harmless one (their position is 0).
struct Axis {
    int n;
    double lo, hi, d, o;
    const double2 *cell;
    const int *bkt;
    int nbkt;
    double bsc;
};

template <bool RECT>
__device__ __forceinline__ Axis axis_of(const FieldView &f, int a)
{
    Axis x;
    x.n = a == 3 ? 2 : sel3<int>(a, f.nx, f.ny, f.nz);
    x.d = a == 3 ? 1.0 : sel3<double>(a, f.d[0], f.d[1], f.d[2]);
    x.o = a == 3 ? 0.0 : sel3<double>(a, f.o[0], f.o[1], f.o[2]);
    x.lo = 0.0;
    x.hi = (double)(x.n - 1);
    if constexpr (RECT) {
        x.lo = sel3<double>(a, f.lo64[0], f.lo64[1], f.lo64[2]);
        x.hi = sel3<double>(a, f.hi64[0], f.hi64[1], f.hi64[2]);
        x.cell = a == 0 ? f.cell64[0] : (a == 1 ? f.cell64[1] : f.cell64[2]);
        x.bkt = a == 0 ? f.bkt[0] : (a == 1 ? f.bkt[1] : f.bkt[2]);
        x.nbkt = sel3<int>(a, f.nbkt[0], f.nbkt[1], f.nbkt[2]);
        x.bsc = sel3<double>(a, f.bsc64[0], f.bsc64[1], f.bsc64[2]);
    }
    return x;
}

// The cell of a lane's coordinate, its weight (omega_0 in lanes 0-3, omega_1 in
// lanes 4-7) and its width.
template <bool RECT>
__device__ __forceinline__ int cell_of(const Axis &ax, const Place &g, double X, double &w, double &width)
{
    double w0;
    int c = 0;
    if constexpr (RECT) {
        width = 1.0;
        w0 = 1.0;
        if (g.a < 3) {
            // (trace.cuh rect_cell: the largest c in [0, n - 2] with x_c <= X; the
            // comparisons and the bucket on the integer pipe)
            const long long kx = order_key(X);
            if (kx >= order_key(ax.lo) && kx <= kInfKey) {
                const double bf = __dmul_rn(__dadd_rn(X, -ax.lo), ax.bsc);
                c = __ldg(ax.bkt + trace::cell_floor64(bf, ax.nbkt + 1));
            }
            double2 cr = __ldg(ax.cell + c);
            if (kx <= kInfKey) {
                while (c < ax.n - 2 && kx >= order_key(cr.y)) cr = __ldg(ax.cell + (++c));
                while (c > 0 && kx < order_key(cr.x)) cr = __ldg(ax.cell + (--c));
            }
            width = cr.y - cr.x;
            w0 = div64(cr.y - X, width);
        }
    } else {
        c = trace::cell_floor64(X, ax.n);
        w0 = __dadd_rn(trace::int_f64(c + 1), -X);
        width = ax.d;
    }
    const double w1 = __dadd_rn(1.0, -w0);
    w = g.sub < 4 ? w0 : w1;
    return c;
}

// Component sub (lanes 0 to 5: Bx, By, Bz, Jx, Jy, Jz) at the position whose
// components the lanes hold, Eq. interp term by term: the sum over m (x), n (y),
// p (z) in that nesting of (w_m w_n) w_p times the corner's value.
// Given the lanes' cells c and weights w.
__device__ __forceinline__ double gather_cell(const FieldView &f, const Place &g, int c, double w)
{
    const long long sy = f.nx, sz = (long long)f.nx * f.ny;
    const long long base = (long long)__shfl_sync(g.mask, c, 2, kGroup) * sz +
                           (long long)__shfl_sync(g.mask, c, 1, kGroup) * sy + __shfl_sync(g.mask, c, 0, kGroup);
    const double *r = (const double *)f.rec + 8 * base + (g.sub < 6 ? g.sub : 5);
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __ldg(r + 8 * ((i & 1 ? sz : 0) + (i & 2 ? sy : 0) + (i & 4 ? 1 : 0)));
    // this lane's corner: m = bit 2, n = bit 1, p = bit 0 of sub
    const double wm = get(g, w, g.sub & 4), wn = get(g, w, (g.sub & 2 ? 4 : 0) + 1), wp = get(g, w, (g.sub & 1 ? 4 : 0) + 2);
    const double wt = __dmul_rn(__dmul_rn(wm, wn), wp);
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const double t = __dmul_rn(v[i], get(g, wt, i));
        s = i ? __dadd_rn(s, t) : plus_zero(t);
    }
    return s;
}

template <bool RECT>
__device__ __forceinline__ double gather(const FieldView &f, const Axis &ax, const Place &g, double X, double &width)
{
    double w;
    const int c = cell_of<RECT>(ax, g, X, w, width);
    return gather_cell(f, g, c, w);
}

// Right-hand side at a position: lanes 0 to 4 get {F (3), dl/dtau, dTw/dtau}
// (bt_a = B_a / D_a, F = sigma bt / |bt| or, stretched, sigma B / |bt|; dl/dtau =
// |B| / |bt|; dTw/dtau = (J.B) / (4 pi B^2) dl/dtau). Returns false on a null or
// non-finite field. On a unit grid bt = B and dl/dtau = 1 exactly.
// c, w: the lanes' cells and weights there.
template <bool RECT>
__device__ __forceinline__ bool rhs(const FieldView &f, const Place &g, int c, double w, const soft64::Divisor &D,
                                    double sgn, double &o)
{
    const double v = gather_cell(f, g, c, w);
    const double b0 = get(g, v, 0), b1 = get(g, v, 1), b2 = get(g, v, 2);
    // lanes 0-2: B_c^2, lanes 3-5: J_c B_c
    const double pr = __dmul_rn(v, g.sub < 3 ? v : sel3<double>(g.sub - 3, b0, b1, b2));
    const double S = sum3(g, pr, g.sub < 4 ? 0 : 3);  // lanes 0-3: B^2, lanes 4-7: J.B
    const double BB = get(g, S, 0);
    const bool unit = !RECT && f.unit;
    double bt = v, bb = BB;
    if (!unit) {
        bt = div64(v, D);
        bb = sum3(g, __dmul_rn(bt, bt), 0);
    }
    if (!positive_finite(bb)) return false;
    // both roots at once: lanes 0-3 |bt|, lanes 4-7 |B|
    const double root = sqrt64(g.sub < 4 ? bb : BB);
    const double nbt = get(g, root, 0), nB = unit ? nbt : get(g, root, 4);
    double num = g.sub < 3 ? turn(sgn, RECT ? v : bt) : (g.sub == 4 ? S : nB);
    const double den = g.sub == 4 ? __dmul_rn(12.566370614359172, BB) : nbt;
    o = div64(num, den);
    if (!unit) {
        const double dl = get(g, o, 3);
        if (g.sub == 4) o = __dmul_rn(o, dl);
    }
    return true;
}

// The line of a group. X, S: the lane's position component and its seed; the
// others are the same in all lanes unless noted.
struct Line {
    long long line;
    double X, S;
    double h, tol, s0;
    double O;     // end of the exiting step: lanes 0-2 position, 3 length, 4 Tw
    double t0;    // chord parameter of the first crossed face
    double acc;   // lanes 3, 4: length and Tw of the current direction
    double tot1;  // lanes 3, 4: totals of end 1
    int steps, st, end, mode, hface, tries, fc0;
    int tcur, tn;  // step tape (see trace::Lane)
};

__device__ __forceinline__ bool all_of(const Place &g, bool p)
{
    return (__ballot_sync(g.mask, p) & g.mask) == g.mask;
}

template <bool RECT>
__device__ __forceinline__ double phys(const Axis &ax, double x)
{
    return RECT ? x : trace::to_phys(ax.o, ax.d, x);
}

template <bool RECT>
__device__ __forceinline__ void write_end(const LineRecs &R, const Axis &ax, const Place &g, long long line, int e,
                                          double X, int face, double bn)
{
    if (g.sub < 3) (e == 0 ? R.r1 : R.r2)[3 * line + g.sub] = phys<RECT>(ax, X);
    if (g.sub == 0) {
        (e == 0 ? R.f1 : R.f2)[line] = (int8_t)face;
        double *bnp = e == 0 ? R.bn1 : R.bn2;
        if (bnp) bnp[line] = bn;
    }
}

__device__ __forceinline__ void nan_sums(const LineRecs &R, const Place &g, long long line)
{
    if (g.sub == 0) {
        if (R.tw) R.tw[line] = NAN;
        if (R.len) R.len[line] = NAN;
    }
}

// --- step tape (trace.cuh) ---
__device__ __forceinline__ bool tape_chunk(const Tape &tp, const Place &g, Line &L)
{
    unsigned long long c = 0;
    if (g.sub == 0) c = atomicAdd(tp.next, 1ull);
    c = __shfl_sync(g.mask, c, 0, kGroup);
    if (c >= (unsigned long long)tp.cap) {
        L.tcur = -2;
        return false;
    }
    if (g.sub == 0) {
        tp.prev[c] = L.tcur;
        tp.owner[c] = (int32_t)(tp.hl_base + 2 * L.line + L.end);
    }
    const double x = g.sub < 3 ? L.X : 0.0;
    if (g.sub < 4) {
        ((double *)tp.xi)[4 * c + g.sub] = x;
        if (tp.wx && (long long)c < tp.wcap)
            ((double *)tp.wx)[c * (unsigned long long)(tp.k + 1) * kStateStride + g.sub] = x;
    }
    L.tcur = (int)c;
    L.tn = 0;
    return true;
}

// NS stages' derivatives k (the lane's component) and the end state x1
template <int NS>
__device__ __forceinline__ void tape_step(const Tape &tp, const Place &g, Line &L, double h, const double k[], double x1)
{
    if (L.tcur == -2) return;
    if ((L.tcur < 0 || L.tn == tp.k) && !tape_chunk(tp, g, L)) return;
    const long long j = (long long)L.tcur * tp.k + L.tn;
    if (g.sub == 0) ((double *)tp.h)[j] = h;
    if (tp.wx && L.tcur < tp.wcap) {
        double *wk = (double *)tp.wk + j * kStageStride;
        if (g.sub < 3) {
#pragma unroll 1
            for (int s = 0; s < NS; s++) wk[3 * s + g.sub] = k[s];
        }
        if (NS == 5 && g.sub == 3) wk[15] = 0.0;
        if (g.sub < 4)
            ((double *)tp.wx)[((long long)L.tcur * (tp.k + 1) + L.tn + 1) * kStateStride + g.sub] = g.sub < 3 ? x1 : 0.0;
    }
    L.tn++;
}

__device__ __forceinline__ void tape_end(const Tape &tp, const Place &g, Line &L, int code, double X, double hx)
{
    if (L.tcur == -1) tape_chunk(tp, g, L);
    const long long hl = tp.hl_base + 2 * L.line + L.end;
    const int sg = (L.end == 0) == (L.s0 > 0.0) ? -1 : 1;
    if (g.sub == 0) tp.head[hl] = make_int4(L.tcur, L.tn, L.tcur >= 0 ? code : -2, sg);
    if (g.sub < 4) ((double *)tp.xe)[4 * hl + g.sub] = g.sub < 3 ? X : hx;
}

// split directions of the taped lattice tracer (trace::split_finish)
__device__ __forceinline__ void split_finish(const TraceArgs &A, const LineRecs &R, const Place &g, Line &L, bool bad)
{
    int before = 0;
    if (g.sub == 0) before = atomicAdd(R.steps + L.line, L.steps);
    before = __shfl_sync(g.mask, before, 0, kGroup);
    unsigned st = (unsigned)L.st;
    if ((long long)before + L.steps > A.p.max_steps) {
        st |= FQSL_LINE_MAXSTEPS;
        bad = true;
    }
    if (g.sub == 0) trace::or_status(R.st, L.line, st);
    if (bad) nan_sums(R, g, L.line);
}

template <bool SPLIT, bool RECT>
__device__ __forceinline__ void finish_bad(const TraceArgs &A, const LineRecs &R, const Axis &ax, const Place &g, Line &L,
                                           unsigned bit)
{
    L.st |= bit;
    write_end<RECT>(R, ax, g, L.line, L.end, L.X, -1, 0.0);
    if (L.end == 0 && !SPLIT) write_end<RECT>(R, ax, g, L.line, 1, L.S, -1, 0.0);
    nan_sums(R, g, L.line);
    if constexpr (SPLIT) {
        split_finish(A, R, g, L, true);
    } else if (g.sub == 0) {
        R.st[L.line] = (uint8_t)L.st;
        R.steps[L.line] = L.steps;
    }
}

// A direction reached a face at X. Returns whether the line goes on (its
// second direction).
template <bool SPLIT, bool RECT>
__device__ __forceinline__ bool finish_dir(const TraceArgs &A, const LineRecs &R, const Axis &ax, const Place &g, Line &L,
                                           double X, int face)
{
    X = get(g, X, g.a);
    if (g.a == 3) X = 0.0;
    double width;
    const double v = gather<RECT>(A.f, ax, g, X, width);
    write_end<RECT>(R, ax, g, L.line, L.end, X, face, get(g, v, face >> 1));
    if constexpr (SPLIT) {
        if (g.sub == 4 && R.tw) atomicAdd(R.tw + L.line, L.acc);
        if (g.sub == 3 && R.len) atomicAdd(R.len + L.line, L.acc);
        split_finish(A, R, g, L, false);
        return false;
    }
    if (L.end == 0) {
        L.tot1 = L.acc;
        L.end = 1;
        L.X = L.S;
        L.h = A.p.scheme == 1 ? L.tol : A.p.h0;
        L.mode = 0;
        L.tcur = -1;
        L.tn = 0;
        L.acc = 0.0;
        return true;
    }
    if (g.sub == 0) {
        R.st[L.line] = (uint8_t)L.st;
        R.steps[L.line] = L.steps;
    }
    if (g.sub == 4 && R.tw) R.tw[L.line] = L.tot1 + L.acc;
    if (g.sub == 3 && R.len) R.len[L.line] = L.tot1 + L.acc;
    return false;
}

// Start a line at the state position X (lanes' components) with B there (v,
// lanes 0 to 2), orientation sign s0 and tolerance or step tol. Returns false
// if it ends at once.
template <bool RECT>
__device__ __forceinline__ bool start_line(const TraceArgs &A, const LineRecs &R, const Axis &ax, const Place &g, Line &L,
                                           double X, bool in, double v, double width, double s0, double tol, int st0)
{
    L.X = L.S = X;
    L.st = st0;
    L.steps = 0;
    L.end = 0;
    L.mode = 0;
    L.tcur = -1;
    L.tn = 0;
    L.acc = 0.0;
    L.tol = tol;
    L.h = A.p.scheme == 1 ? tol : A.p.h0;
    unsigned bad = 0;
    if (!in) {
        bad = FQSL_LINE_OUTSIDE;
    } else {
        const double b = div64(v, width);
        const double bb = sum3(g, __dmul_rn(b, b), 0);
        if (!positive_finite(bb)) bad = FQSL_LINE_NULL_B;
    }
    if (bad) {
        write_end<RECT>(R, ax, g, L.line, 0, X, -1, 0.0);
        write_end<RECT>(R, ax, g, L.line, 1, X, -1, 0.0);
        nan_sums(R, g, L.line);
        if (g.sub == 0) {
            R.st[L.line] = (uint8_t)(L.st | (int)bad);
            R.steps[L.line] = 0;
        }
        return false;
    }
    L.s0 = s0;
    return true;
}

// component a of a lattice seed (trace::lattice_seed)
__device__ __forceinline__ double seed_of(const Lattice &G, int a, long long i, long long j, long long k)
{
    double v = __dadd_rn(sel3<double>(a, G.o[0], G.o[1], G.o[2]),
                         __dmul_rn((double)i + 0.5, sel3<double>(a, G.a1[0], G.a1[1], G.a1[2])));
    v = __dadd_rn(v, __dmul_rn((double)j + 0.5, sel3<double>(a, G.a2[0], G.a2[1], G.a2[2])));
    return __dadd_rn(v, __dmul_rn((double)k + 0.5, sel3<double>(a, G.a3[0], G.a3[1], G.a3[2])));
}

// state coordinate of a physical one
template <bool RECT>
__device__ __forceinline__ double state_of(const Axis &ax, const Place &g, double r)
{
    if (g.a == 3) return 0.0;
    return RECT ? r : div64(r - ax.o, ax.d);
}

// Lattice seed (trace::init_lattice): frame, tolerance and rotation decision.
template <bool RECT>
__device__ __forceinline__ bool init_lattice(const TraceArgs &A, const Axis &ax, const Place &g, Line &L, long long item,
                                             bool reg_rot)
{
    const Lattice &G = A.lat;
    const long long per_tile = kTileU * kTileV;
    const long long w = item % per_tile;
    long long t = item / per_tile;
    const long long tu = t % G.tiles_u;
    t /= G.tiles_u;
    const long long tv = t % G.tiles_v;
    const long long k = t / G.tiles_v;
    const long long i = tu * kTileU + (w % kTileU);
    const long long j = tv * kTileV + (w / kTileU);
    if (i >= G.n1 || j >= G.n2 || k >= G.n3) return false;
    const long long idx = i + G.n1 * (j + G.n2 * k);
    L.line = idx;
    const double X = state_of<RECT>(ax, g, seed_of(G, g.a, i, j, k));
    const bool in = all_of(g, g.a == 3 || (X >= ax.lo && X <= ax.hi));
    double tol = trace::ctl_perp(A.p), bn0 = 0.0, v = 0.0, width = 1.0, bn = 0.0;
    int st0 = 0;
    if (in) {
        v = gather<RECT>(A.f, ax, g, X, width);
        const double nB = sqrt64(sum3(g, __dmul_rn(v, v), 0));
        const double n0 = sel3<double>(g.sub, G.n0[0], G.n0[1], G.n0[2]);
        bn = sum3(g, __dmul_rn(v, n0), 0);
        if (positive_finite(nB)) {
            const double ratio = div64(fabs(bn), nB);
            bool on_face = false;
            if (G.normal_axis >= 0) {
                const bool mine = X == ax.lo || X == ax.hi;
                on_face = __shfl_sync(g.mask, (int)mine, G.normal_axis, kGroup) != 0;
            }
            if (G.allow_rot && ratio < A.p.rot && !on_face) {
                st0 = FQSL_LINE_ROTATED;
                bn0 = nB;
                if (reg_rot && g.sub == 0) {
                    const unsigned slot = atomicAdd(A.q.rot_count, 1u);
                    A.q.rot_seed[slot] = (int32_t)idx;
                    A.q.rot_slot[idx] = (int32_t)slot + 1;
                }
            } else {
                bn0 = bn;
                if (A.p.scheme == 1) tol = fmax(A.p.step * ratio, A.p.step_min);  // Eq. step
                else tol = A.p.tol * trace::obliq_pow(fmax(ratio, A.p.rot), A.p.texp);
            }
        }
    }
    if (g.sub == 0) A.rec.bn0[idx] = bn0;
    return start_line<RECT>(A, A.rec, ax, g, L, X, in, v, width, bn < 0.0 ? -1.0 : 1.0, tol, st0);
}

// Rotated extra line q of rotated slot s (trace::init_extra).
template <bool RECT>
__device__ __forceinline__ bool init_extra(const TraceArgs &A, const Axis &ax, const Place &g, Line &L, long long item)
{
    const Lattice &G = A.lat;
    const long long s = item >> 2;
    const int q = (int)(item & 3);
    const long long idx = A.q.rot_seed[s];
    const long long i = idx % G.n1, j = (idx / G.n1) % G.n2, k = idx / (G.n1 * G.n2);
    const double r0 = seed_of(G, g.a, i, j, k);
    double width;
    const double v0 = gather<RECT>(A.f, ax, g, state_of<RECT>(ax, g, r0), width);
    const double nB = sqrt64(sum3(g, __dmul_rn(v0, v0), 0));
    const double b = div64(v0, nB);
    const double bh[3] = {get(g, b, 0), get(g, b, 1), get(g, b, 2)};
    double u[3], v[3];
    trace::perp_frame(bh, u, v);
    const double n0 = sel3<double>(g.sub, G.n0[0], G.n0[1], G.n0[2]);
    const double sc = sum3(g, __dmul_rn(v0, n0), 0) < 0.0 ? -1.0 : 1.0;
    const double dir = q < 2 ? sel3<double>(g.a, u[0], u[1], u[2]) : sel3<double>(g.a, v[0], v[1], v[2]);
    const double sg = (q & 1) ? -1.0 : 1.0;
    const double X = state_of<RECT>(ax, g, __dadd_rn(r0, __dmul_rn(__dmul_rn(sg, G.drot), dir)));
    const bool in = all_of(g, g.a == 3 || (X >= ax.lo && X <= ax.hi));
    double B = 0.0, s0 = 1.0;
    if (in) {
        B = gather<RECT>(A.f, ax, g, X, width);
        // B . n with n = sc bh
        const double nr = turn(sc, sel3<double>(g.sub, bh[0], bh[1], bh[2]));
        if (sum3(g, __dmul_rn(B, nr), 0) < 0.0) s0 = -1.0;
    }
    L.line = item;
    return start_line<RECT>(A, A.ext, ax, g, L, X, in, B, width, s0, trace::ctl_perp(A.p), 0);
}

template <bool RECT>
__device__ __forceinline__ bool init_list(const TraceArgs &A, const Axis &ax, const Place &g, Line &L, long long item)
{
    L.line = item;
    const double X = state_of<RECT>(ax, g, g.a < 3 ? A.seeds[3 * item + g.a] : 0.0);
    const bool in = all_of(g, g.a == 3 || (X >= ax.lo && X <= ax.hi));
    double v = 0.0, width = 1.0;
    if (in) v = gather<RECT>(A.f, ax, g, X, width);
    return start_line<RECT>(A, A.rec, ax, g, L, X, in, v, width, 1.0, trace::ctl_perp(A.p), 0);
}

// The persistent kernel body (the template parameters are trace::trace_body's).
// p.lanes / 8 groups of each warp take lines, each as soon as its last one is
// done: groups of a warp share no cells that matter here, the FP64 and integer
// pipes do.
template <int SRC, bool BATCH = false, bool TAPE = false, bool RECT = false, int SCH = 0>
__device__ __forceinline__ void trace_body(const TraceArgs &A0, const BatchArgs &BA)
{
    constexpr bool SPLIT = TAPE && SRC == kSrcLattice;
    const int lane = threadIdx.x & 31;
    const int lead = lane & ~(kGroup - 1);
    const Place g{0xffu << lead, lane & (kGroup - 1), lane & 3};
    const double hmin = A0.p.hmin, hmax = A0.p.hmax, graze = A0.p.graze;
    const int max_steps = (int)A0.p.max_steps;

    long long nitems = A0.nitems;
    if (BATCH) nitems = BA.ibase[BA.nent];
    else if (SRC == kSrcExtra) nitems = 4LL * (long long)(*(volatile unsigned *)A0.q.rot_count);
    // lanes that take lines: the host chose them by the lattice's lines, and there
    // may be four times as many extra lines (48x48 seeds, all rotated: 5.9 -> 4.0 ms)
    int take = A0.p.lanes, chunk = A0.p.chunk;  // (chunk divides 32 with BATCH)
    if (SRC == kSrcExtra)
        for (; take < 32 && nitems > (long long)gridDim.x * (blockDim.x / 32) * chunk; chunk *= 2) take *= 2;
    const unsigned gmask = 0x01010101u & (take >= 32 ? kFull : (1u << take) - 1u);

    long long ck_cur = 0, ck_end = 0, ck_base = 0;
    int ck_ent = 0, eb = 0;
    bool exhausted = false, active = false;
    Line L;
    L.line = 0;
    Axis ax = axis_of<RECT>(BATCH ? BA.desc[0].f : A0.f, g.a);
    auto ent = [&]() -> const TraceArgs & {
        if constexpr (BATCH) return BA.desc[eb];
        else return A0;
    };

    for (;;) {
        unsigned idle = __ballot_sync(kFull, !active) & gmask;
        while (idle != 0u && !exhausted) {
            if (ck_cur >= ck_end) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(A0.q.head, (unsigned long long)chunk);
                base = __shfl_sync(kFull, base, 0);
                if ((long long)base >= nitems) {
                    exhausted = true;
                    break;
                }
                ck_cur = (long long)base;
                ck_end = min(ck_cur + chunk, nitems);
                ck_base = 0;
                if constexpr (BATCH) {
                    int lo = 0, hi = BA.nent - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (BA.ibase[mid] <= ck_cur) lo = mid;
                        else hi = mid - 1;
                    }
                    ck_ent = lo;
                    ck_base = BA.ibase[lo];
                }
            }
            const long long avail = ck_end - ck_cur;
            const int rank = __popc(idle & ((1u << lead) - 1u));
            if (((idle >> lead) & 1u) && rank < avail) {
                const long long item = ck_cur + rank - ck_base;
                eb = ck_ent;
                const TraceArgs &E = ent();
                if constexpr (BATCH) ax = axis_of<RECT>(E.f, g.a);
                if constexpr (SRC == kSrcLattice) {
                    if constexpr (SPLIT) {
                        // 32 items' first directions, then the same items' second ones
                        const long long q = item >> 5;
                        active = init_lattice<RECT>(E, ax, g, L, ((q >> 1) << 5) | (item & 31), (q & 1) == 0);
                        if (active && (q & 1)) L.end = 1;
                    } else {
                        active = init_lattice<RECT>(E, ax, g, L, item, true);
                    }
                } else if constexpr (SRC == kSrcExtra) {
                    active = item < 4LL * (long long)*E.q.rot_count && init_extra<RECT>(E, ax, g, L, item);
                } else {
                    active = item < A0.nitems && init_list<RECT>(E, ax, g, L, item);
                }
            }
            ck_cur += min((long long)__popc(idle), avail);
            idle = __ballot_sync(kFull, !active) & gmask;
        }
        if (__ballot_sync(kFull, active) == 0u) break;
        if (!active) continue;

        const TraceArgs &A = ent();
        const FieldView &f = A.f;
        const LineRecs &R = (SRC == kSrcExtra) ? A.ext : A.rec;
        // the step's scale per axis: the spacing, or the start cell's widths
        // (the first stage is there too)
        double D, wx;
        int cx = cell_of<RECT>(ax, g, L.X, wx, D);
        const soft64::Divisor dD = soft64::divisor(D);
        const bool henon = L.mode != 0;
        const int hax = L.hface >> 1;
        const double hsign = (L.hface & 1) ? 1.0 : -1.0;
        const double target = get(g, (L.hface & 1) ? ax.hi : ax.lo, henon ? hax : 0);
        const double sgn = (L.end == 0) ? -L.s0 : L.s0;
        double hh = L.h;
        if (!henon) {
            if (L.steps >= max_steps) {
                finish_bad<SPLIT, RECT>(A, R, ax, g, L, FQSL_LINE_MAXSTEPS);
                active = false;
                continue;
            }
        } else {
            hh = target - get(g, L.X, hax);
        }
        L.steps++;

        constexpr int NST = SCH ? 4 : 6;
        // stage derivatives: lanes 0-2 and 4-6 their axis'
        double k[5];
        // weighted sums of the stages: lanes 0-4 with the 4th-order weights
        // (position, length, Tw), lanes 5-7 position with the 5th-order ones
        double ws = 0.0;
        const int own = g.sub < 5 ? g.sub : g.sub - 5;
        int fail = 0;  // first failing stage: 1 null field, 2 grazing exit step
        // (an exit step of length 0 evaluates one point: see trace.cuh)
        const bool still = henon && hh == 0.0;
        double o = 0.0;
#pragma unroll 1
        for (int s = 0; s < NST; s++) {
            if (s > 0 && !still) {
                // sum of a(s, r) k_r over r, left to right; lanes 0-2 form the
                // products of even r, lanes 4-6 those of the odd r behind them
                double p = 0.0;
#pragma unroll 1
                for (int r = 0; r < s; r += 2) {
                    const int q = g.sub < 4 || r + 1 == s ? r : r + 1;
                    const double t = __dmul_rn(k[q], kA[SCH][s][q]);
                    p = r ? __dadd_rn(p, t) : plus_zero(t);
                    if (r + 1 < s) p = __dadd_rn(p, get(g, t, 4 + g.a));
                }
                double x = get(g, __dadd_rn(L.X, __dmul_rn(hh, p)), g.a), width;
                if (g.a == 3) x = 0.0;
                cx = cell_of<RECT>(ax, g, x, wx, width);
            }
            if (s == 0 || !still) {
                o = 0.0;
                const bool ok = rhs<RECT>(f, g, cx, wx, dD, sgn, o);
                if (!ok && !fail) fail = 1;
                if (henon) {
                    const double fa = get(g, o, hax);
                    const double fn = RECT ? div64(fa, get(g, D, hax)) : fa;
                    const bool bad = !(turn(hsign, fn) >= graze);
                    if (bad && !fail) fail = 2;
                    o = div64(o, bad ? 1.0 : fa);
                }
            }
            const double ka = get(g, o, g.a);
            if (s < 5) k[s] = ka;
            const double t = __dmul_rn(g.sub < 5 || SCH ? kB[SCH][s] : kB5[s], get(g, o, own));
            ws = s ? __dadd_rn(ws, t) : plus_zero(t);
        }

        if (fail == 1) {
            finish_bad<SPLIT, RECT>(A, R, ax, g, L, FQSL_LINE_NULL_B);
            active = false;
            continue;
        }
        // the step's end: lanes 0-2 position, 3 and 4 the sums with the step,
        // 5-7 the 5th-order position
        const double xo = get(g, L.X, own);
        const double E = __dadd_rn(g.sub == 3 || g.sub == 4 ? L.acc : xo, __dmul_rn(hh, ws));
        if (!henon) {
            double hn = L.h;
            if constexpr (SCH == 0) {
                double e = __dadd_rn(get(g, E, g.sub < 3 ? g.sub + 5 : g.sub), -E);
                if constexpr (RECT) e = div64(e, dD);
                const double err = sqrt64(sum3(g, __dmul_rn(e, e), 0));
                const bool over = err > L.tol;
                double q = 0.0;
                if (err > 0.0) q = sqrt64(sqrt64(div64(L.tol, err)));
                if (over) {
                    if (L.h > hmin) {
                        const double hr = L.h * fmax(0.1, 0.9 * q);
                        L.h = hr < hmin ? hmin : hr;
                        continue;
                    }
                    L.st |= FQSL_LINE_STALL;
                }
                hn = err > 0.0 ? L.h * fmin(4.0, 0.9 * q) : 4.0 * L.h;
                hn = hn < hmin ? hmin : (hn > hmax ? hmax : hn);
            }
            if (all_of(g, g.sub > 2 || (E >= ax.lo && E <= ax.hi))) {
                if constexpr (TAPE) tape_step<SCH ? 4 : 5>(A.tape, g, L, hh, k, E);
                L.X = get(g, E, g.a);
                if (g.a == 3) L.X = 0.0;
                L.acc = E;
                L.h = hn;
                continue;
            }
            // exit: the first face the chord crosses (ties: lower axis first)
            double t = INFINITY;
            int fc = -1;
            if (g.sub < 3) {
                if (E < ax.lo) {
                    t = div64(ax.lo - L.X, E - L.X);
                    fc = 2 * g.sub;
                } else if (E > ax.hi) {
                    t = div64(ax.hi - L.X, E - L.X);
                    fc = 2 * g.sub + 1;
                }
            }
            int best = -1;
            double tb = INFINITY;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const double ta = get(g, t, a);
                const int fa = __shfl_sync(g.mask, fc, a, kGroup);
                if (fa >= 0 && ta < tb) {
                    tb = ta;
                    best = fa;
                }
            }
            L.O = E;
            L.t0 = tb;
            L.fc0 = best;
            L.hface = best;
            L.tries = 0;
            L.mode = 1;
            continue;
        }
        // exit step
        if (fail == 2) {
            L.mode = 0;
            if (0.5 * L.h >= hmin) {
                L.h = 0.5 * L.h;
                continue;
            }
            // chord fallback onto the first crossed face
            const double c = g.sub < 3 ? L.X : L.acc;
            double e = __dadd_rn(c, __dmul_rn(L.t0, __dadd_rn(L.O, -c)));
            if (g.sub == 3 || g.sub == 4) L.acc = e;
            const double v0 = get(g, (L.fc0 & 1) ? ax.hi : ax.lo, L.fc0 >> 1);
            if (g.sub == L.fc0 >> 1) e = v0;
            L.st |= FQSL_LINE_CHORD;
            if constexpr (TAPE) tape_end(A.tape, g, L, kTapeChord + L.fc0, e, L.h);
            active = finish_dir<SPLIT, RECT>(A, R, ax, g, L, e, L.fc0);
            continue;
        }
        double tx = E;
        if (g.sub == hax) tx = target;
        const unsigned below = __ballot_sync(g.mask, g.sub < 3 && g.sub != hax && tx < ax.lo) >> lead;
        const unsigned above = __ballot_sync(g.mask, g.sub < 3 && g.sub != hax && tx > ax.hi) >> lead;
        const unsigned off = (below | above) & 7u;
        const int nf = off ? 2 * (__ffs(off) - 1) + ((below >> (__ffs(off) - 1)) & 1u ? 0 : 1) : -1;
        if (nf >= 0 && L.tries < 2) {
            L.hface = nf;
            L.tries++;
            continue;
        }
        if (nf >= 0) tx = fmin(fmax(tx, ax.lo), ax.hi);
        L.acc = E;
        if constexpr (TAPE) tape_end(A.tape, g, L, (nf >= 0 ? kTapeExitClamped : kTapeExit) + L.hface, tx, 0.0);
        active = finish_dir<SPLIT, RECT>(A, R, ax, g, L, tx, L.hface);
    }
}

}  // namespace trace64
}  // namespace fqsl
