// sm_103a kernels of the flow diagnostics of the results section (arXiv 2108.08919, §5): fields on
// an M x M grid by Shepard interpolation with the method's kernel (Eq. 18), the kinetic-energy
// spectrum of Eq. 31 by a radix-4 FFT, the vorticity correlation of Eq. 32 along the centre line,
// topological defects as winding numbers of the gridded Q, the mixing of coloured particles, and
// unwrapped positions for pathlines.  None of these run inside a step.
#include "ann_device.cuh"

#include <cmath>

namespace ann {
namespace {

// ------------------------------------------------------------------------------------------------
// Shepard gridding.  Nodes (ix L/M, iy L/M).  Each node gathers from the particles of the 3 x 3 or
// 5 x 5 cells around its own cell in the cell order of the last re-sort: a particle has moved far less
// than one cell since then (a re-sort comes once anything moves half the 0.02 x 3h skin), so every
// particle within 3h of the node is in reach, and the sum runs in a fixed order.
// ------------------------------------------------------------------------------------------------

// Per slot: position relative to the corner of the slot's cell (FP32), and the four fields.
// out: how far any particle lies outside its cell, over both axes (FP32 bits, zeroed by the caller;
// 0 right after a re-sort): the gridding skips the cells this says no particle reaches.
__global__ void __launch_bounds__(256) k_grid_prep(DevParams P, Bufs b, DiagSrc src, float2 *off, float4 *fld,
                                                   unsigned *out)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    float e = 0.f;
    if (s < P.n) {
        uint32_t key = b.mkey[s];
        int cx = (int)(key % (uint32_t)P.nc), cy = (int)(key / (uint32_t)P.nc);
        const double ox = src.x[s] - b.origin[cx], oy = src.y[s] - b.origin[cy];
        float fx = (float)ox, fy = (float)oy;
        const float cell = (float)P.cell, hL = (float)(0.5 * P.L);
        // crossed a face since the re-sort (an offset is near 0 or near L: FP32 decides it)
        if (fabsf(fx) > hL) fx = (float)(fx > 0.f ? ox - P.L : ox + P.L);
        if (fabsf(fy) > hL) fy = (float)(fy > 0.f ? oy - P.L : oy + P.L);
        off[s] = make_float2(fx, fy);
        fld[s] = src.u4 ? src.u4[s] : make_float4(src.ux[s], src.uy[s], src.q11[s], src.q12[s]);
        e = fmaxf(fmaxf(fmaxf(-fx, fx - cell), fmaxf(-fy, fy - cell)), 0.f);
    }
    unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(e));   // e >= 0: bits order as values
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned *)out) atomicMax(out, m);
}

constexpr int GRID_TILE = 16;   // a block covers 16 x 16 nodes

// A node sums its particles in cell order (rows of cells, then cells, then slots), whatever cells are
// skipped: a skipped cell holds no particle within 3h, so the sum is the same to the last bit.  With
// e the excursion of k_grid_prep, cells two away are out of reach while e < cell - 3h (a re-sort comes
// before that in all but extreme steps), and a cell is skipped when its box, grown by e, lies
// beyond 3h.  The test carries a 1e-5 margin against FP32 rounding.  1M nodes on 1M particles: 244 us,
// where testing all 25 cells took 521 (380 distance tests a node for 44 hits).
__global__ void __launch_bounds__(256) k_grid(DevParams P, Bufs b, int M, const float2 *off, const float4 *fld,
                                              const unsigned *out, double *grid)
{
    int ix = blockIdx.x * GRID_TILE + (threadIdx.x % GRID_TILE);
    int iy = blockIdx.y * GRID_TILE + (threadIdx.x / GRID_TILE);
    if (ix >= M || iy >= M) return;
    const double im = 1.0 / M;   // exact: M is a power of two
    double gx = (double)ix * P.L * im, gy = (double)iy * P.L * im;
    int cx = min((int)(gx * P.inv_cell), P.nc - 1), cy = min((int)(gy * P.inv_cell), P.nc - 1);
    float rx0 = (float)(gx - b.origin[cx]), ry0 = (float)(gy - b.origin[cy]);
    float cellf = (float)P.cell;
    float R2 = (float)P.R2;   // (3h)^2: W vanishes there, so the FP32 test is enough
    const float e = __uint_as_float(*out), far = cellf + e, R2skip = R2 * (1.f + 1e-5f);
    const int reach = e < (cellf - sqrtf(R2)) - 1e-5f * cellf ? 1 : 2;
    // distance from the coordinate r (relative to a cell's corner) to the cell grown by e
    auto gap = [&](float r) { return fmaxf(fmaxf(r - far, -e - r), 0.f); };
    float sw = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int oy = -reach; oy <= reach; oy++) {
        int ccy = cy + oy;
        ccy = ccy < 0 ? ccy + P.nc : (ccy >= P.nc ? ccy - P.nc : ccy);
        float ry = ry0 - (float)oy * cellf;
        const float gy2 = gap(ry) * gap(ry);
        for (int ox = -reach; ox <= reach; ox++) {
            int ccx = cx + ox;
            ccx = ccx < 0 ? ccx + P.nc : (ccx >= P.nc ? ccx - P.nc : ccx);
            float rx = rx0 - (float)ox * cellf;
            if (gap(rx) * gap(rx) + gy2 > R2skip) continue;
            int c = ccy * P.nc + ccx;
            uint32_t s0 = b.cell_start[c], s1 = b.cell_start[c + 1];
            for (uint32_t s = s0; s < s1; s++) {
                float2 o = off[s];
                float2 d = make_float2(rx - o.x, ry - o.y);
                float r2 = len2(d);
                if (r2 < R2) {
                    float W = kernel_w<true>(r2, P);
                    float4 f = fld[s];
                    sw += W;
                    acc.x = fmaf(W, f.x, acc.x);
                    acc.y = fmaf(W, f.y, acc.y);
                    acc.z = fmaf(W, f.z, acc.z);
                    acc.w = fmaf(W, f.w, acc.w);
                }
            }
        }
    }
    size_t MM = (size_t)M * M, g = (size_t)iy * M + ix;
    bool any = sw > 0.f;
    grid[g] = any ? (double)acc.x / sw : 0.0;
    grid[MM + g] = any ? (double)acc.y / sw : 0.0;
    grid[2 * MM + g] = any ? (double)acc.z / sw : 0.0;
    grid[3 * MM + g] = any ? (double)acc.w / sw : 0.0;
    grid[4 * MM + g] = (double)sw;
}

// ------------------------------------------------------------------------------------------------
// FFT (FP64, radix 4, M a power of two).  z = ux + i uy is transformed along rows, transposed and
// transformed along rows again; |Z|^2 is symmetric under the transposition as far as the shells
// are concerned (|k| depends on kx^2 + ky^2).  E_n = 1/2 sum_{|k| -> n} |Z(k)|^2 / M^4 equals
// 1/2 sum (|ux_hat|^2 + |uy_hat|^2) with u_hat = fft2(u) / M^2, because Z(k) = Ux(k) + i Uy(k)
// for real ux, uy gives |Z(k)|^2 + |Z(-k)|^2 = 2 (|Ux(k)|^2 + |Uy(k)|^2) and every shell holds
// -k with k.
// ------------------------------------------------------------------------------------------------

__global__ void k_twiddles(int M, double2 *tw)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M / 2) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)M, &s, &c);   // exp(-2 pi i k / M)
    tw[k] = make_double2(c, s);
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// p = a + w b, m = a - w b (six operations: m = 2a - p)
__device__ __forceinline__ void butterfly(double2 a, double2 b, double2 w, double2 &p, double2 &m)
{
    p.x = fma(w.x, b.x, fma(-w.y, b.y, a.x));
    p.y = fma(w.x, b.y, fma(w.y, b.x, a.y));
    m.x = fma(2.0, a.x, -p.x);
    m.y = fma(2.0, a.y, -p.y);
}

// One row per block of M/4 threads: radix-4 passes of the self-sorting (Stockham) FFT, four points
// a thread in registers, one exchange through shared memory between passes; a last radix-2 pass when
// log2 M is odd.  Pass with sub-transforms of L points: thread j takes points j + r M/4, multiplies by
// exp(-2 pi i r k / 4L), k = j mod L, and writes 4 (j - k) + k + r L.  The first pass reads and the
// last writes global memory (coalesced).  The work is FP64 issue (2 a cycle and SM): 112 operations
// a thread of M = 1024 (16 in the first pass, whose factors are 1, and 24 in each other) against the
// 160 a thread would have in radix-2 passes; M = 1024: 79 us a dimension (ncu,
// cold caches), radix 2 took 92.  The
// exchange buffer is padded by an element in four, which keeps the stride-4 writes of the first pass
// free of bank conflicts.  PACK: the input is the real grid pair (ux, uy) packed as ux + i uy.
__host__ __device__ constexpr int fft_pad(int i) { return i + (i >> 2); }

template <bool PACK>
__global__ void __launch_bounds__(512) k_fft_rows(int M, const double2 *in, const double *gx, const double *gy,
                                                  double2 *out, const double2 *tw)
{
    extern __shared__ double2 sm[];
    const size_t base = (size_t)blockIdx.x * M;
    const int Q = M / 4, j = threadIdx.x;
    double2 *buf = sm;
    double2 x[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const size_t i = base + j + r * Q;
        x[r] = PACK ? make_double2(gx[i], gy[i]) : in[i];
    }
    int L = 1;
    for (; 4 * L <= M; L *= 4) {
        const int k = j & (L - 1), st = Q / L;   // factor r is exp(-2 pi i r k st / M)
        double2 a, b, c, d;   // a, b = x0 +- w2 x2, c, d = w1 x1 +- w3 x3
        if (L == 1) {
            a = cadd(x[0], x[2]);
            b = csub(x[0], x[2]);
            c = cadd(x[1], x[3]);
            d = csub(x[1], x[3]);
        } else {
            const int i3 = 3 * k * st;   // up to 3/4 M: the table holds half a turn
            double2 w3 = tw[i3 < M / 2 ? i3 : i3 - M / 2];
            if (i3 >= M / 2) w3 = make_double2(-w3.x, -w3.y);
            butterfly(x[0], x[2], tw[2 * k * st], a, b);
            butterfly(cmul(x[1], tw[k * st]), x[3], w3, c, d);
        }
        x[0] = cadd(a, c);
        x[2] = csub(a, c);
        x[1] = make_double2(b.x + d.y, b.y - d.x);   // b - i d
        x[3] = make_double2(b.x - d.y, b.y + d.x);
        const int o = 4 * (j - k) + k;
        if (4 * L == M) {   // done: o = j
#pragma unroll
            for (int r = 0; r < 4; r++) out[base + j + r * Q] = x[r];
            return;
        }
#pragma unroll
        for (int r = 0; r < 4; r++) buf[fft_pad(o + r * L)] = x[r];
        __syncthreads();
        if (8 * L == M) break;   // a radix-2 pass is left
#pragma unroll
        for (int r = 0; r < 4; r++) x[r] = buf[fft_pad(j + r * Q)];
        buf = buf == sm ? sm + fft_pad(M) : sm;   // the next pass writes the other buffer: one barrier a pass
    }
#pragma unroll
    for (int r = 0; r < 2; r++) {   // L = M/2: two of the M/2 pairs a thread
        const int i = j + r * Q;
        double2 p, m;
        butterfly(buf[fft_pad(i)], buf[fft_pad(i + M / 2)], tw[i], p, m);
        out[base + i] = p;
        out[base + i + M / 2] = m;
    }
}

__global__ void k_transpose(int M, const double2 *in, double2 *out)
{
    __shared__ double2 tile[32][33];
    int x = blockIdx.x * 32 + threadIdx.x, y0 = blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y)
        if (x < M && y0 + k < M) tile[k][threadIdx.x] = in[(size_t)(y0 + k) * M + x];
    __syncthreads();
    int xo = blockIdx.y * 32 + threadIdx.x, yo0 = blockIdx.x * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y)
        if (xo < M && yo0 + k < M) out[(size_t)(yo0 + k) * M + xo] = tile[threadIdx.x][k];
}

// One block per shell: its modes in increasing index order, a fixed-order tree over the threads.
__global__ void __launch_bounds__(256) k_shell_sum(int M, const double2 *Z, const int *off, const int *modes,
                                                   double *E)
{
    __shared__ double red[256];
    int n = blockIdx.x;
    double acc = 0.0;
    for (int t = off[n] + threadIdx.x; t < off[n + 1]; t += blockDim.x) {
        double2 z = Z[modes[t]];
        acc += z.x * z.x + z.y * z.y;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double m2 = (double)M * (double)M;
        E[n] = 0.5 * red[0] / (m2 * m2);
    }
}

// ------------------------------------------------------------------------------------------------
// Vorticity on the centre row by periodic central differences, and its correlation (Eq. 32).
// ------------------------------------------------------------------------------------------------

__device__ __forceinline__ double vorticity(int M, double L, const double *grid, int i)
{
    const size_t MM = (size_t)M * M;
    const double *ux = grid, *uy = grid + MM;
    const int j0 = M / 2, jm = j0 - 1, jp = (j0 + 1) % M, ip = (i + 1) % M, im = (i + M - 1) % M;
    const double D2 = 2.0 * (L / M);
    const double dvx = (uy[(size_t)j0 * M + ip] - uy[(size_t)j0 * M + im]) / D2;
    const double duy = (ux[(size_t)jp * M + i] - ux[(size_t)jm * M + i]) / D2;
    return dvx - duy;
}

__global__ void __launch_bounds__(256) k_vorticity_row(int M, double L, const double *grid, double *om)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) om[i] = vorticity(M, L, grid, i);
}

// One warp per lag k: lane l sums the origins l, l + 32, ... and a fixed tree joins the lanes.  The
// 2 M (M/2 + 1) multiply-adds are FP64 (2 a cycle and SM), so they are spread over the whole GPU: at
// M = 1024 this takes 9 us and the row kernel 4 us, where one block with a thread per lag took 283 us.
// ONE: where there is little to sum (one origin, or a row of at most 64 nodes) one block takes the row too: a
// second launch would cost more than it saves (a call 30.4 us with one kernel, 31.7 with two).
constexpr int CORR_WARPS = 4, CORR_ONE = 64;

template <bool ONE>
__global__ void __launch_bounds__(ONE ? 1024 : 32 * CORR_WARPS)
    k_correlation(int M, double L, const double *grid, const double *row, int all_origins, double *C)
{
    extern __shared__ double om[];
    for (int i = threadIdx.x; i < M; i += blockDim.x) om[i] = ONE ? vorticity(M, L, grid, i) : row[i];
    __syncthreads();
    if (ONE && !all_origins) {
        const int i0 = M / 2;
        for (int k = threadIdx.x; k <= M / 2; k += blockDim.x) C[k] = om[(i0 + k) & (M - 1)] * om[i0] / (om[i0] * om[i0]);
        return;
    }
    const int warps = blockDim.x >> 5, lane = threadIdx.x & 31;
    for (int k = blockIdx.x * warps + (threadIdx.x >> 5); k <= M / 2; k += ONE ? warps : M) {
        double num = 0.0, den = 0.0;
        for (int i = lane; i < M; i += 32) {
            num += om[(i + k) & (M - 1)] * om[i];   // M is a power of two
            den += om[i] * om[i];
        }
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        if (lane == 0) C[k] = num / den;
    }
}

// ------------------------------------------------------------------------------------------------
// Defects: winding number m of (Q11, Q12) around the plaquette with lower-left node (ix, iy), by
// signed crossings of the positive Q11 axis; cross products without fused operations so that the
// integer decision is the plain FP64 one.
// ------------------------------------------------------------------------------------------------

__device__ __forceinline__ int crossing(double a1, double a2, double b1, double b2)
{
    // the comparisons with zero on the bit patterns (FP64 issues at 1/64 of the integer rate):
    // v > 0 and v <= 0, both false for a NaN
    const long long a = __double_as_longlong(a2), b = __double_as_longlong(b2), inf = 0x7ff0000000000000ll;
    auto above = [&](long long v) { return v > 0 && v <= inf; };
    auto below = [&](long long v) { return v == 0 || (v < 0 && (v & 0x7fffffffffffffffll) <= inf); };
    const bool up = below(a) && above(b), down = below(b) && above(a);
    if (!(up || down)) return 0;
    const long long cr = __double_as_longlong(__dsub_rn(__dmul_rn(a1, b2), __dmul_rn(a2, b1)));
    if (up) return above(cr);                                   // cr > 0
    return cr < 0 && above(cr & 0x7fffffffffffffffll) ? -1 : 0;   // cr < 0
}

// A plaquette's winding is the sum of the crossings of its four edges, and an edge belongs to two
// plaquettes with opposite signs (the cross product changes sign exactly): a block of DEF_ROWS rows
// takes each edge once, through shared memory.  The kernel is bound by FP64 issue (2 a cycle and
// SM); the counts are summed per block.  M = 1024: 32 us, where taking four edges a
// plaquette with an atomic per defect took 74.
// Grids below 256 nodes a side, whose blocks would be too few or too narrow to hide a column's eight
// rows, take a row a block (a call at M = 8: 20.5 us with four edges a plaquette, 28.8 with eight rows a block).
constexpr int DEF_ROWS = 8, DEF_FEW = 256;

template <int ROWS>
__global__ void __launch_bounds__(256) k_defects(int M, const double *grid, signed char *map, unsigned long long *counts)
{
    __shared__ signed char up[ROWS][257];   // edge (ix, iy) -> (ix, iy + 1)
    __shared__ int sum[3];
    const size_t MM = (size_t)M * M;
    const double *q1 = grid + 2 * MM, *q2 = grid + 3 * MM;
    const int W = blockDim.x, x0 = blockIdx.x * W, ix = x0 + threadIdx.x, xp = (ix + 1) & (M - 1);
    const int y0 = blockIdx.y * ROWS, xe = (x0 + W) & (M - 1);   // M is a power of two, at least 8
    if (threadIdx.x < 3) sum[threadIdx.x] = 0;
    int right[ROWS + 1];   // edge (ix, iy) -> (ix + 1, iy)
    double a1 = q1[(size_t)y0 * M + ix], a2 = q2[(size_t)y0 * M + ix];
#pragma unroll
    for (int r = 0; r <= ROWS; r++) {
        const size_t row = (size_t)((y0 + r) & (M - 1)) * M;
        right[r] = crossing(a1, a2, q1[row + xp], q2[row + xp]);
        if (r == ROWS) break;
        const size_t nxt = (size_t)((y0 + r + 1) & (M - 1)) * M + ix;
        const double b1 = q1[nxt], b2 = q2[nxt];
        up[r][threadIdx.x] = (signed char)crossing(a1, a2, b1, b2);
        a1 = b1;
        a2 = b2;
    }
    if (threadIdx.x < ROWS) {   // the column past the block's last
        const size_t g = (size_t)(y0 + threadIdx.x) * M + xe;
        const size_t h = (size_t)((y0 + threadIdx.x + 1) & (M - 1)) * M + xe;
        up[threadIdx.x][W] = (signed char)crossing(q1[g], q2[g], q1[h], q2[h]);
    }
    __syncthreads();
    int plus = 0, minus = 0, more = 0;
#pragma unroll
    for (int r = 0; r < ROWS; r++) {
        const int m = right[r] + up[r][threadIdx.x + 1] - right[r + 1] - up[r][threadIdx.x];
        map[(size_t)(y0 + r) * M + ix] = (signed char)m;
        plus += m == 1;
        minus += m == -1;
        more += m < -1 || m > 1;
    }
    atomicAdd(&sum[0], plus);
    atomicAdd(&sum[1], minus);
    atomicAdd(&sum[2], more);
    __syncthreads();
    if (threadIdx.x < 3 && sum[threadIdx.x]) atomicAdd(&counts[threadIdx.x], (unsigned long long)sum[threadIdx.x]);
}

// ------------------------------------------------------------------------------------------------
// Mixing: particles per (bin, colour), bins floor(x G / L) clamped to G - 1 (integer counts, exact).
// Pathlines: unwrapped positions of chosen particle IDs.
// ------------------------------------------------------------------------------------------------

__global__ void k_mix_bins(DevParams P, Bufs b, const unsigned char *colors, int G, int S, unsigned *cnt)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= P.n) return;
    int bx = min((int)floor(__ddiv_rn(__dmul_rn(b.sx[s], (double)G), P.L)), G - 1);
    int by = min((int)floor(__ddiv_rn(__dmul_rn(b.sy[s], (double)G), P.L)), G - 1);
    int col = colors[b.sid[s]];
    atomicAdd(&cnt[((size_t)by * G + bx) * S + col], 1u);
}

__global__ void k_inverse(int n, const int *sid, int *inv)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) inv[sid[s]] = s;
}

__global__ void k_unwrap(DevParams P, Bufs b, const int *inv, const long long *ids, int k, double *xy)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= k) return;
    long long id = ids[t];
    int s = inv[id];
    int2 im = b.img[id];
    xy[2 * t] = b.sx[s] + (double)im.x * P.L;
    xy[2 * t + 1] = b.sy[s] + (double)im.y * P.L;
}

inline unsigned blocks(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t enqueue_grid(const DevParams &P, const Bufs &b, DiagSrc src, int M, float2 *off, float4 *fld,
                         unsigned *out, double *grid, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned), s);
    if (e) return e;
    k_grid_prep<<<blocks(P.n, 256), 256, 0, s>>>(P, b, src, off, fld, out);
    dim3 g((M + GRID_TILE - 1) / GRID_TILE, (M + GRID_TILE - 1) / GRID_TILE);
    k_grid<<<g, 256, 0, s>>>(P, b, M, off, fld, out, grid);
    return cudaGetLastError();
}

cudaError_t enqueue_twiddles(int M, double2 *tw, cudaStream_t s)
{
    k_twiddles<<<blocks(M / 2, 256), 256, 0, s>>>(M, tw);
    return cudaGetLastError();
}

cudaError_t enqueue_spectrum(int M, const double *grid, double2 *z, double2 *zt, const double2 *tw,
                             const int *shell_off, const int *shell_modes, int nshell, double *E, cudaStream_t s)
{
    const int th = M / 4;   // 2 (M = 8) to 512
    size_t smem = sizeof(double2) * 2 * (size_t)fft_pad(M);
    cudaError_t e = cudaFuncSetAttribute(k_fft_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (!e) e = cudaFuncSetAttribute(k_fft_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    size_t MM = (size_t)M * M;
    k_fft_rows<true><<<M, th, smem, s>>>(M, nullptr, grid, grid + MM, z, tw);
    dim3 tb(32, 8), tg((M + 31) / 32, (M + 31) / 32);
    k_transpose<<<tg, tb, 0, s>>>(M, z, zt);
    k_fft_rows<false><<<M, th, smem, s>>>(M, zt, nullptr, nullptr, z, tw);
    k_shell_sum<<<nshell, 256, 0, s>>>(M, z, shell_off, shell_modes, E);
    return cudaGetLastError();
}

cudaError_t enqueue_correlation(int M, double L, const double *grid, int all_origins, double *C, double *om,
                                cudaStream_t s)
{
    size_t smem = sizeof(double) * (size_t)M;
    if (!all_origins || M <= CORR_ONE) {
        k_correlation<true><<<1, 1024, smem, s>>>(M, L, grid, om, all_origins, C);
    } else {
        k_vorticity_row<<<blocks(M, 256), 256, 0, s>>>(M, L, grid, om);
        k_correlation<false><<<blocks(M / 2 + 1, CORR_WARPS), 32 * CORR_WARPS, smem, s>>>(M, L, grid, om, all_origins, C);
    }
    return cudaGetLastError();
}

cudaError_t enqueue_defects(int M, const double *grid, signed char *map, unsigned long long *counts, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, 3 * sizeof(unsigned long long), s);
    if (e) return e;
    const int w = M < 256 ? M : 256;
    if (M < DEF_FEW) k_defects<1><<<dim3(M / w, M), w, 0, s>>>(M, grid, map, counts);
    else k_defects<DEF_ROWS><<<dim3(M / w, M / DEF_ROWS), w, 0, s>>>(M, grid, map, counts);
    return cudaGetLastError();
}

cudaError_t enqueue_mixing(const DevParams &P, const Bufs &b, const unsigned char *colors, int G, int S,
                           unsigned *cnt, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(unsigned) * (size_t)G * G * S, s);
    if (e) return e;
    k_mix_bins<<<blocks(P.n, 256), 256, 0, s>>>(P, b, colors, G, S, cnt);
    return cudaGetLastError();
}

cudaError_t enqueue_unwrapped(const DevParams &P, const Bufs &b, int *inv, const long long *ids, int k, double *xy,
                              cudaStream_t s)
{
    k_inverse<<<blocks(P.n, 256), 256, 0, s>>>(P.n, b.sid, inv);
    if (k > 0) k_unwrap<<<blocks(k, 256), 256, 0, s>>>(P, b, inv, ids, k, xy);
    return cudaGetLastError();
}

}  // namespace ann
