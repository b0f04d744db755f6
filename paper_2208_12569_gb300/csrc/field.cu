// curl_pack: curl B at the nodes and the packed B+J node records.
//
// The twist number Tw = int (curl B . B)/(4 pi B^2) dl (Sec. 1, Eq. tw) needs
// curl B along the line; it is precomputed once per field on the node grid
// with 2nd-order central differences inside (the stencil of Eq. grad_B),
// 2nd-order one-sided differences on the faces and first order on a 2-node
// axis, and packed next to B so that one trilinear gather (Sec. 2.2, Eq.
// interp) fetches both. FP64 records (and FP32 records of an FP64 cube) use
// FP64 stencils written as plain expressions; FP32 records of an FP32 cube use
// float stencils. On a stretched grid the three-point stencils of a
// non-uniform axis are used, in FP64. One thread per node, grid-stride;
// streaming and HBM-bound.
#include "fqsl_internal.cuh"
#include "soft64.cuh"

namespace fqsl {
namespace {

template <typename TI>
__device__ __forceinline__ double node_diff(const TI *__restrict__ B, int c, long long node, long long stride,
                                            long long i, long long n, const soft64::Divisor &h)
{
    // value of component c at index kk along the axis (node is at index i);
    // h: the spacing (2 nodes) or twice it
    auto F = [&](long long kk) -> double { return (double)B[(node + (kk - i) * stride) * 3 + c]; };
    double v;
    if (n == 2) v = F(1) - F(0);
    else if (i == 0) v = -3.0 * F(0) + 4.0 * F(1) - F(2);
    else if (i == n - 1) v = 3.0 * F(n - 1) - 4.0 * F(n - 2) + F(n - 3);
    else v = F(i + 1) - F(i - 1);
    return soft64::div64(v, h);
}

template <typename TI>
__global__ void __launch_bounds__(256) k_curl_pack(const TI *__restrict__ B, int nx, int ny, int nz, double dx,
                                                   double dy, double dz, float4 *__restrict__ rec32,
                                                   double2 *__restrict__ rec64)
{
    const long long total = (long long)nx * ny * nz;
    const long long sy = nx, sz = (long long)nx * ny;
    // the six divisions of a node run on the integer pipe (same bits): they held
    // the FP64 pipe for about 60 of the node's 75 instructions (FP64 records of
    // 256x256x128 nodes of an FP64 cube 1.09 -> 0.62 ms)
    const soft64::Divisor hx = soft64::divisor(nx == 2 ? dx : 2.0 * dx), hy = soft64::divisor(ny == 2 ? dy : 2.0 * dy),
                          hz = soft64::divisor(nz == 2 ? dz : 2.0 * dz);
    for (long long node = blockIdx.x * (long long)blockDim.x + threadIdx.x; node < total;
         node += (long long)gridDim.x * blockDim.x) {
        const long long i = node % nx;
        const long long j = (node / nx) % ny;
        const long long k = node / sz;
        const double dyBz = node_diff(B, 2, node, sy, j, ny, hy);
        const double dzBy = node_diff(B, 1, node, sz, k, nz, hz);
        const double dzBx = node_diff(B, 0, node, sz, k, nz, hz);
        const double dxBz = node_diff(B, 2, node, 1, i, nx, hx);
        const double dxBy = node_diff(B, 1, node, 1, i, nx, hx);
        const double dyBx = node_diff(B, 0, node, sy, j, ny, hy);
        const double Jx = dyBz - dzBy, Jy = dzBx - dxBz, Jz = dxBy - dyBx;
        const double Bx = (double)B[node * 3 + 0], By = (double)B[node * 3 + 1], Bz = (double)B[node * 3 + 2];
        if (rec32) {
            rec32[2 * node + 0] = make_float4((float)Bx, (float)By, (float)Bz, (float)Jx);
            rec32[2 * node + 1] = make_float4((float)Jy, (float)Jz, 0.f, 0.f);
        }
        if (rec64) {
            rec64[4 * node + 0] = make_double2(Bx, By);
            rec64[4 * node + 1] = make_double2(Bz, Jx);
            rec64[4 * node + 2] = make_double2(Jy, Jz);
            rec64[4 * node + 3] = make_double2(0.0, 0.0);
        }
    }
}

// Stretched grid (Sec. 2.2): d f/d x_a at node index i along an axis, as the
// derivative of the quadratic through three neighbouring nodes (one-sided at
// the ends, first order on a 2-node axis); on a uniform axis these are the
// stencils above. co = the node's three coefficients, formed on the host
// from the node coordinates X (fqsl_field_create_rect); with them each
// derivative is a plain sum of products in a fixed order:
//   inside: c0 f_{i-1} + c1 f_i + c2 f_{i+1}; first node: c0 f_0 + c1 f_1 -
//   c2 f_2; last node: c0 f_{n-3} - c1 f_{n-2} + c2 f_{n-1}.
template <typename TI>
__device__ __forceinline__ double node_diff_rect(const TI *__restrict__ B, int c, long long node, long long stride,
                                                 long long i, long long n, const double *__restrict__ X,
                                                 const double *__restrict__ co)
{
    auto F = [&](long long kk) -> double { return (double)B[(node + (kk - i) * stride) * 3 + c]; };
    if (n == 2) return (F(1) - F(0)) / (X[1] - X[0]);
    const double c0 = co[3 * i], c1 = co[3 * i + 1], c2 = co[3 * i + 2];
    if (i == 0) return c0 * F(0) + c1 * F(1) - c2 * F(2);
    if (i == n - 1) return c0 * F(n - 3) - c1 * F(n - 2) + c2 * F(n - 1);
    return c0 * F(i - 1) + c1 * F(i) + c2 * F(i + 1);
}

template <typename TI>
__global__ void __launch_bounds__(256) k_curl_pack_rect(const TI *__restrict__ B, const FieldView g,
                                                        float4 *__restrict__ rec32, double2 *__restrict__ rec64)
{
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const long long total = (long long)nx * ny * nz;
    const long long sy = nx, sz = (long long)nx * ny;
    for (long long node = blockIdx.x * (long long)blockDim.x + threadIdx.x; node < total;
         node += (long long)gridDim.x * blockDim.x) {
        const long long i = node % nx;
        const long long j = (node / nx) % ny;
        const long long k = node / sz;
        const double dyBz = node_diff_rect(B, 2, node, sy, j, ny, g.x64[1], g.dco[1]);
        const double dzBy = node_diff_rect(B, 1, node, sz, k, nz, g.x64[2], g.dco[2]);
        const double dzBx = node_diff_rect(B, 0, node, sz, k, nz, g.x64[2], g.dco[2]);
        const double dxBz = node_diff_rect(B, 2, node, 1, i, nx, g.x64[0], g.dco[0]);
        const double dxBy = node_diff_rect(B, 1, node, 1, i, nx, g.x64[0], g.dco[0]);
        const double dyBx = node_diff_rect(B, 0, node, sy, j, ny, g.x64[1], g.dco[1]);
        const double Jx = dyBz - dzBy, Jy = dzBx - dxBz, Jz = dxBy - dyBx;
        const double Bx = (double)B[node * 3 + 0], By = (double)B[node * 3 + 1], Bz = (double)B[node * 3 + 2];
        if (rec32) {
            rec32[2 * node + 0] = make_float4((float)Bx, (float)By, (float)Bz, (float)Jx);
            rec32[2 * node + 1] = make_float4((float)Jy, (float)Jz, 0.f, 0.f);
        }
        if (rec64) {
            rec64[4 * node + 0] = make_double2(Bx, By);
            rec64[4 * node + 1] = make_double2(Bz, Jx);
            rec64[4 * node + 2] = make_double2(Jy, Jz);
            rec64[4 * node + 3] = make_double2(0.0, 0.0);
        }
    }
}

// FP32 records only: the same stencils in float with reciprocal spacings (the
// FP64 kernel above is the one whose rounding matches a plain evaluation).
__device__ __forceinline__ float node_diff32(const float *__restrict__ B, int c, unsigned node, unsigned stride,
                                             unsigned i, unsigned n, float rh, float rh2)
{
    auto F = [&](unsigned kk) -> float { return B[(size_t)(node + kk * stride - i * stride) * 3 + c]; };
    if (n == 2) return (F(1) - F(0)) * rh;
    if (i == 0) return (-3.f * F(0) + 4.f * F(1) - F(2)) * rh2;
    if (i == n - 1) return (3.f * F(n - 1) - 4.f * F(n - 2) + F(n - 3)) * rh2;
    return (F(i + 1) - F(i - 1)) * rh2;
}

// 32-bit index arithmetic (a cube with FP32 records holds fewer than 2^31 nodes)
__global__ void __launch_bounds__(256) k_curl_pack32(const float *__restrict__ B, int nx, int ny, int nz, float rx,
                                                     float ry, float rz, float4 *__restrict__ rec32)
{
    const unsigned total = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned sy = (unsigned)nx, sz = (unsigned)nx * (unsigned)ny;
    for (unsigned node = blockIdx.x * blockDim.x + threadIdx.x; node < total; node += gridDim.x * blockDim.x) {
        const unsigned t = node / sy;
        const unsigned i = node - t * sy;
        const unsigned k = t / (unsigned)ny;
        const unsigned j = t - k * (unsigned)ny;
        const float dyBz = node_diff32(B, 2, node, sy, j, ny, ry, 0.5f * ry);
        const float dzBy = node_diff32(B, 1, node, sz, k, nz, rz, 0.5f * rz);
        const float dzBx = node_diff32(B, 0, node, sz, k, nz, rz, 0.5f * rz);
        const float dxBz = node_diff32(B, 2, node, 1, i, nx, rx, 0.5f * rx);
        const float dxBy = node_diff32(B, 1, node, 1, i, nx, rx, 0.5f * rx);
        const float dyBx = node_diff32(B, 0, node, sy, j, ny, ry, 0.5f * ry);
        rec32[2 * (size_t)node + 0] = make_float4(B[(size_t)node * 3 + 0], B[(size_t)node * 3 + 1], B[(size_t)node * 3 + 2], dyBz - dzBy);
        rec32[2 * (size_t)node + 1] = make_float4(dzBx - dxBz, dxBy - dyBx, 0.f, 0.f);
    }
}

// B/|B| at a node (0 where |B| = 0), the divisions and the root on the integer
// pipe (soft64.cuh; same bits).
struct Unit {
    double v[3];
};

template <typename TI>
__device__ __forceinline__ Unit bhat(const TI *__restrict__ B, long long q)
{
    const double b0 = (double)B[3 * q], b1 = (double)B[3 * q + 1], b2 = (double)B[3 * q + 2];
    const double m = soft64::sqrt64(b0 * b0 + b1 * b1 + b2 * b2);
    const soft64::Divisor d = soft64::divisor(m);
    Unit u;
    u.v[0] = m > 0 ? soft64::div64(b0, d) : 0.0;
    u.v[1] = m > 0 ? soft64::div64(b1, d) : 0.0;
    u.v[2] = m > 0 ? soft64::div64(b2, d) : 0.0;
    return u;
}

// grad(B/|B|) at the nodes for Method II way 1 (Sec. 4, Eq. grad_B): G[a*3+b]
// = d(B_b/|B|)/dx_a with the stencils of the curl grid (RECT: node_diff_rect's).
// A block holds B/|B| of a tile of GX x GY x GZ nodes and its one-node halo in
// shared memory, so that a node's is formed about twice and not 18 times (its
// root and divisions are what the kernel spends its time on: repacking 256x256x128
// nodes with the gradient took 9.54 ms when a thread formed all of a node's
// differences from B, and takes 1.54 ms); the one-sided differences on the
// faces, which reach two nodes, form theirs.
constexpr int kGradThreads = 128;

template <typename TI, bool RECT, int GX, int GY, int GZ>
__global__ void __launch_bounds__(kGradThreads) k_gradb_pack(const TI *__restrict__ B, const FieldView g,
                                                             float4 *__restrict__ g32, double *__restrict__ g64)
{
    __shared__ double U[3][GZ + 2][GY + 2][GX + 2];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const long long stride[3] = {1, nx, (long long)nx * ny};
    const int n[3] = {nx, ny, nz};
    const int tx = (nx + GX - 1) / GX, ty = (ny + GY - 1) / GY;
    const long long tiles = (long long)tx * ty * ((nz + GZ - 1) / GZ);
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int x0 = (int)(t % tx) * GX, y0 = (int)(t / tx % ty) * GY, z0 = (int)(t / ((long long)tx * ty)) * GZ;
        __syncthreads();
        for (int q = threadIdx.x; q < (GZ + 2) * (GY + 2) * (GX + 2); q += kGradThreads) {
            const int i = q % (GX + 2), j = q / (GX + 2) % (GY + 2), k = q / ((GX + 2) * (GY + 2));
            const int x = x0 + i - 1, y = y0 + j - 1, z = z0 + k - 1;
            if (x < 0 || y < 0 || z < 0 || x >= nx || y >= ny || z >= nz) continue;
            const Unit u = bhat(B, x + nx * (y + (long long)ny * z));
#pragma unroll
            for (int c = 0; c < 3; c++) U[c][k][j][i] = u.v[c];
        }
        __syncthreads();
#pragma unroll 1
        for (int q = threadIdx.x; q < GX * GY * GZ; q += kGradThreads) {
            const int i = q % GX, j = q / GX % GY, k = q / (GX * GY);
            if (x0 + i >= nx || y0 + j >= ny || z0 + k >= nz) continue;
            const int at[3] = {x0 + i, y0 + j, z0 + k};
            const long long node = at[0] + nx * (at[1] + (long long)ny * at[2]);
            double G[3][3];
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const int p = at[a], m = n[a];
                const bool inner = m > 2 && p > 0 && p < m - 1;
                // B/|B| at the three nodes of the stencil, in its order
                Unit f[3];
                if (inner) {
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        f[0].v[c] = U[c][k + 1 - (a == 2)][j + 1 - (a == 1)][i + 1 - (a == 0)];
                        f[1].v[c] = U[c][k + 1][j + 1][i + 1];
                        f[2].v[c] = U[c][k + 1 + (a == 2)][j + 1 + (a == 1)][i + 1 + (a == 0)];
                    }
                } else {
#pragma unroll 1
                    for (int r = 0; r < 3; r++) {
                        // first node: 0, 1, 2; last: n - 1, n - 2, n - 3; two nodes: 0, 1
                        const int q = m == 2 ? min(r, 1) : (p == 0 ? r : m - 1 - r);
                        const Unit u = bhat(B, node + (long long)(q - p) * stride[a]);
                        if (r == 0) f[0] = u;
                        else if (r == 1) f[1] = u;
                        else f[2] = u;
                    }
                }
                if constexpr (RECT) {
                    const double *X = g.x64[a], *co = g.dco[a] + 3 * p;
                    const soft64::Divisor w = soft64::divisor(m == 2 ? X[1] - X[0] : 1.0);
#pragma unroll
                    for (int b = 0; b < 3; b++) {
                        const double f0 = f[0].v[b], f1 = f[1].v[b], f2 = f[2].v[b];
                        if (m == 2) G[a][b] = soft64::div64(f1 - f0, w);
                        else if (p == 0) G[a][b] = co[0] * f0 + co[1] * f1 - co[2] * f2;
                        else if (p == m - 1) G[a][b] = co[0] * f2 - co[1] * f1 + co[2] * f0;
                        else G[a][b] = co[0] * f0 + co[1] * f1 + co[2] * f2;
                    }
                } else {
                    const soft64::Divisor w = soft64::divisor(m == 2 ? g.d[a] : 2.0 * g.d[a]);
#pragma unroll
                    for (int b = 0; b < 3; b++) {
                        const double f0 = f[0].v[b], f1 = f[1].v[b], f2 = f[2].v[b];
                        double v;
                        if (m == 2) v = f1 - f0;
                        else if (p == 0) v = -3.0 * f0 + 4.0 * f1 - f2;
                        else if (p == m - 1) v = 3.0 * f0 - 4.0 * f1 + f2;
                        else v = f2 - f0;
                        G[a][b] = soft64::div64(v, w);
                    }
                }
            }
            if (g64) {
#pragma unroll
                for (int c = 0; c < 9; c++) g64[node * 10 + c] = G[c / 3][c % 3];
                g64[node * 10 + 9] = 0.0;
            }
            if (g32) {
                g32[3 * node + 0] = make_float4((float)G[0][0], (float)G[0][1], (float)G[0][2], (float)G[1][0]);
                g32[3 * node + 1] = make_float4((float)G[1][1], (float)G[1][2], (float)G[2][0], (float)G[2][1]);
                g32[3 * node + 2] = make_float4((float)G[2][2], 0.f, 0.f, 0.f);
            }
        }
    }
}

template <typename TI, bool RECT, int GX, int GY, int GZ>
void gradb_tiled(const void *B, const FieldView &g, float4 *g32, double *g64, int sms, cudaStream_t s)
{
    const long long tiles = (long long)((g.nx + GX - 1) / GX) * ((g.ny + GY - 1) / GY) * ((g.nz + GZ - 1) / GZ);
    const unsigned blocks = (unsigned)(tiles < (long long)sms * 32 ? tiles : (long long)sms * 32);
    k_gradb_pack<TI, RECT, GX, GY, GZ><<<blocks, kGradThreads, 0, s>>>((const TI *)B, g, g32, g64);
}

template <typename TI, bool RECT>
void gradb_tiles(int shape, const void *B, const FieldView &g, float4 *g32, double *g64, int sms, cudaStream_t s)
{
    if (shape == 0) gradb_tiled<TI, RECT, 16, 8, 4>(B, g, g32, g64, sms, s);
    else if (shape == 1) gradb_tiled<TI, RECT, 4, 32, 4>(B, g, g32, g64, sms, s);
    else gradb_tiled<TI, RECT, 4, 4, 32>(B, g, g32, g64, sms, s);
}

}  // namespace

cudaError_t launch_gradb_pack(const void *B, fqsl_dtype bt, const FieldView &g, void *grad32, void *grad64,
                              cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // Tiles of 16 x 8 x 4 nodes; where an axis would leave most of that empty, of
    // 4 x 32 x 4 or 4 x 4 x 32 (four updates of an FP32 cube of 2 x 512 x 512 nodes with
    // the gradient 3.3 -> 1.03 ms, of 2 x 2 x 40,000 2.5 -> 0.77).
    const int shape = g.nx > 8 ? 0 : (g.ny > 8 ? 1 : 2);
    const bool f32 = bt == FQSL_F32;
    if (f32 && g.rect) gradb_tiles<float, true>(shape, B, g, (float4 *)grad32, (double *)grad64, sms, s);
    else if (f32) gradb_tiles<float, false>(shape, B, g, (float4 *)grad32, (double *)grad64, sms, s);
    else if (g.rect) gradb_tiles<double, true>(shape, B, g, (float4 *)grad32, (double *)grad64, sms, s);
    else gradb_tiles<double, false>(shape, B, g, (float4 *)grad32, (double *)grad64, sms, s);
    return cudaGetLastError();
}

cudaError_t launch_curl_pack(const void *B, fqsl_dtype bt, const FieldView &g, void *rec32, void *rec64,
                             cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long total = (long long)g.nx * g.ny * g.nz;
    long long blocks = (total + 255) / 256;
    const long long cap = (long long)sms * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (g.rect) {
        // stretched grid: FP64 stencils for every record precision
        if (bt == FQSL_F32)
            k_curl_pack_rect<float><<<(unsigned)blocks, 256, 0, s>>>((const float *)B, g, (float4 *)rec32,
                                                                    (double2 *)rec64);
        else
            k_curl_pack_rect<double><<<(unsigned)blocks, 256, 0, s>>>((const double *)B, g, (float4 *)rec32,
                                                                     (double2 *)rec64);
        return cudaGetLastError();
    }
    if (bt == FQSL_F32 && rec32) {
        // FP32 records from an FP32 cube: float stencils (the FP64 records, if
        // also wanted, come from the FP64 stencils below)
        k_curl_pack32<<<(unsigned)blocks, 256, 0, s>>>((const float *)B, g.nx, g.ny, g.nz, (float)(1.0 / g.d[0]),
                                                       (float)(1.0 / g.d[1]), (float)(1.0 / g.d[2]),
                                                       (float4 *)rec32);
        if (rec64)
            k_curl_pack<float><<<(unsigned)blocks, 256, 0, s>>>((const float *)B, g.nx, g.ny, g.nz, g.d[0], g.d[1],
                                                               g.d[2], nullptr, (double2 *)rec64);
    } else if (bt == FQSL_F32)
        k_curl_pack<float><<<(unsigned)blocks, 256, 0, s>>>((const float *)B, g.nx, g.ny, g.nz, g.d[0], g.d[1],
                                                           g.d[2], (float4 *)rec32, (double2 *)rec64);
    else
        k_curl_pack<double><<<(unsigned)blocks, 256, 0, s>>>((const double *)B, g.nx, g.ny, g.nz, g.d[0], g.d[1],
                                                            g.d[2], (float4 *)rec32, (double2 *)rec64);
    return cudaGetLastError();
}

}  // namespace fqsl
