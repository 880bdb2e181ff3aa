// Three-dimensional variant of the SPH active-nematic step (the paper's equations for d = 3):
// a periodic cube, Q as the symmetric traceless 3x3 tensor (Q11, Q12, Q13, Q22, Q23), the corrected
// SPH operators with a 3x3 correction tensor, the viscous term with 2 (d + 2) nu = 10 nu.
//
// One step (modified Euler, §3.1), one CUDA graph launch:
//   predict     u += dt/2 a, r += dt/2 u (wrap), max |u|; the re-sort test (a particle has moved
//               half the skin since the last re-sort)
//   re-sort only (a conditional graph node): cell keys and counts, scan (one block), scatter, each
//               cell's slots ordered by particle ID (deterministic) and the state gathered, the tile
//               lists and candidate lists below
//   filter      neighbour bits (|r_i - r_j| < 3h among the candidates; FP32 test, FP64 in a band
//               around 3h), sum W, V = 1 / sum W (Eq. 19)
//   pass 1      alpha (Eq. 22) and B = alpha^-1, continuity k (Eq. 25), rho_half, corrected
//               velocity gradient (Eq. 20): one walk of the candidates, B applied to the sums afterwards
//   pass 2      density filter (Eq. 28), equation of state (Eq. 26) with c0 = max(10 max|u|, c0_min),
//               corrected Laplacian of Q (Eq. 21), Q rate m (Eqs. 2, 7, 24), Q^{n+1}
//   pass 3      momentum (Eq. 23), artificial displacement (Eq. 29), corrector
//
// Tiles.  A pair kernel runs one block per non-empty cell (side >= 3h (1 + 0.05), ~70 particles on a
// lattice at h = 1.3 dx; wider where that would hold few, see cells3).  The re-sort lists, for each cell, the particles of the 27 surrounding cells that come
// within the candidate radius of the box around the cell's own particles (~1,300 of ~1,900); a
// pair kernel stages these "slots" in shared memory, with positions relative to the cell's centre,
// and the candidate lists name slots: 16-bit byte offsets of 16-byte records, whose free bit 0 says
// whether the candidate is a neighbour in this step.  Beyond the support the clamped kernel gives
// W = F = 0, so the passes sum over candidates; only the displacement's sums use the bit.
// Four lanes share a particle, lane l taking candidates l, l + 4, ...: consecutive candidates are
// mostly consecutive slots, so a load of the 32 lanes meets few bank conflicts, and a small
// box has four times the threads to hide latency with.  A cell whose slots exceed the staging
// capacity (dense clusters, boxes of 14 to 16 spacings) reads its candidates from global memory through
// 32-bit lists instead, in the same kernels.
//
// What bounds it (GB300, 64^3, ~250 neighbours): FP32 and issue (filter, pass 1, 2, 3: the FMA pipe is busy in 40, 47, 52 and
// 54 % of cycles, issue in 72, 54, 62 and 62 %), and the shared-memory loads (62, 69, 78 and 70 % of the LSU's data
// cycles; consecutive particles' lists drift apart, so a load takes about twice its least wavefronts).  They take
// 140, 190, 211 and 306 us; one thread per particle gathering through L1, with lists of the exact neighbours and the
// Laplacian as six sums per component in pass 1, took 305, 351, 194 and 335 (predictor: 55, now 18).
//
// The state lives in S between steps, in the cell order of the last re-sort.  Errors are sticky bits
// set by the kernels' own checks (neighbour overflow, non-finite state, singular alpha).
#include "../../include/ann.h"
#include "ann_device.cuh"

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

namespace {

using ann::add2;
using ann::bc;
using ann::f2;
using ann::fma2;
using ann::in_box;
using ann::mul2;
using ann::sub2;

constexpr int MAXN3 = ANN3_MAX_NEIGHBORS;
constexpr int MAXC3 = 576;          // candidates: neighbours within 3h (1 + SKIN3) at the last re-sort
constexpr double CELL3 = 0.05;      // cells are at least 3h (1 + CELL3) wide
constexpr double SPARSE3 = 50.0, GROW3 = 3.0;   // and wider, up to GROW3 times, where they would hold fewer than SPARSE3 particles: see cells3
// Candidate lists stay valid while no particle moves SKIN3 3h / 2.  A skin of 0.02 keeps ~6 % more
// candidates than neighbours (0.05: 16 %); a re-sort costs about one step and a half.  us a step of 64^3 in a
// box-scale flow with a re-sort in 180 / 36 / 13 / 4 steps at 0.02: 865 / 885 / 919 / 1,047; with 0.05 (half as many or fewer)
// 921 / 932 / 943 / 1,004: the smaller skin loses only where every fourth step re-sorts.
constexpr double SKIN3 = 0.02;
constexpr uint32_t E3_NBR = 4u, E3_NONFINITE = 8u, E3_ALPHA = 16u;

// Staged slots of a tile, with one empty slot at the end that pads the lists.  52 bytes a slot
// (pass 3, the widest) leave room for two blocks per SM.
constexpr int CAP3 = 2200;
constexpr int T3 = 256;             // threads of the list kernel's block
constexpr int LP = 4;               // lanes per particle
constexpr int GRP = 4 * LP;         // candidates per list group: LP lanes x 4 entries
constexpr int NGRP = MAXC3 / GRP;
// Threads and resident blocks per SM of the pair kernels.  The staged slots limit pass 2 and pass 3 to
// two blocks, which leaves the registers (pass 3: 94 a thread) to set the threads; 64^3 / 32^3, us:
// filter 256 x 6: 136 / 30 (320 x 5: 175 / 43); pass 1 384 x 2: 180 / 41 (256 x 3: 200 / 39, 320 x 3:
// 204 / 42); pass 2 512 x 2: 213 / 48 (384 x 2: 220 / 50, 320 x 2: 254 / 55); pass 3 320 x 2: 314 / 66
// (256 x 2: 352 / 63, 288 x 2: 366 / 75, 352 x 2: 344 / 70).
constexpr int TF3 = 256, BF3 = 6, T13 = 384, B13 = 2, T23 = 512, B23 = 2, T33 = 320, B33 = 2;
static_assert(MAXC3 % GRP == 0 && CAP3 * 16 <= 0x10000, "lists are whole groups of 16-bit offsets");
constexpr uint32_t ID_BITS = 26, G_MASK = (1u << ID_BITS) - 1;   // a slot entry: particle | halo cell << 26
constexpr uint32_t NOENTRY = 0xffffffffu;

struct P3 {
    int n, nc, ncell, nblk;      // nblk: blocks of a pair kernel, at least the non-empty cells
    double L, inv_cell, R2d, half_dt_d;
    long long bitsL;
    float inv_h, ad, kw6, kw15, kf5, kf30, kf75, W0, dt, half_dt, cell_f, cell_lo, hL, R2lo, R2hi, R2c, far;   // hL: L / 2; far: beyond any tile and its support
    float skin_max2;
    float rho0, nu, Gamma, lambda, A, B, C, K, zeta, gamma_eos, beta, c0_min, c_shift;
    int apd;
};

struct Set3 {   // the state, sorted by cell
    double *x, *y, *z;
    float4 *ua;   // (u, Q11)
    float4 *qb;   // (Q12, Q13, Q22, Q23)
    float4 *aa;   // (a, dr): dr the density deviation rho / rho0 - 1 (FP32 keeps its digits)
    int *id;
};

// A tile: cell, first entry and number of its slots in Work3::slot, slot of its first own particle
// (count > CAP3 - 1: not staged, candidates in cand32).
struct Tile3 {
    int cell, base, count, self;
};

// Candidate lists.  Candidate k of particle i: group k / 16, lane k mod 4, entry (k / 4) mod 4 of the
// lane's word cand16[(group n + i) 4 + lane] (or cand32), so the four lanes of a particle read 32
// consecutive bytes, and consecutive particles consecutive words.
struct Work3 {
    int *key, *rank, *perm, *count, *start, *nnbr, *ncand, *cell_of;   // cell_of: cx | cy << 10 | cz << 20
    Tile3 *tile;
    int *ntile, *slots_used;
    uint32_t *slot;             // 27 n: the tiles' slots, particle | halo cell << 26
    uint2 *cand16;
    uint4 *cand32;
    const double *centre;       // centre of cell c along an axis
    float4 *xi, *xi_ref;        // position relative to the centre of the particle's cell; at the last re-sort
    unsigned *flag;             // non-zero: this step re-sorts and rebuilds the lists
    unsigned *rebuilds;
    float *sumW, *p, *k, *dhat, *gu, *lap, *m, *qn4;
    float4 *xv;    // (xi, V)                                   written by the filter
    float4 *dq;    // (density deviation at the half step, Q11, Q12, Q13)  written by pass 1
    float2 *q2;    // (Q22, Q23) of the midpoint state          written by pass 1
    float4 *qn;    // Q^{n+1}: (Q11, Q12, Q13, Q22), qn4: Q23   written by pass 2
    float4 *b0;    // B: (11, 12, 13, 22)                       written by pass 1
    float2 *b1;    // B: (23, 33)                               written by pass 1
    float4 *pu;    // (p / rho_hat^2, u)                        written by pass 2
    unsigned *umax, *err;
};

__device__ __forceinline__ double wrap(double v, double L)
{
    double w = v - L * floor(v / L);
    if (w >= L) w -= L;
    if (w < 0.0) w = 0.0;
    return w;
}

__device__ __forceinline__ double min_image(double d, double L)
{
    if (d > 0.5 * L) d -= L;
    else if (d < -0.5 * L) d += L;
    return d;
}

// Offset of a coordinate from the centre c of its cell, across the periodic face if need be (an
// offset is within a cell of 0 or of +-L: FP32 tells which).
__device__ __forceinline__ float offset3(double x, double c, const P3 &P)
{
    const double d = x - c;
    const float f = (float)d;
    return fabsf(f) > P.hL ? (float)(f > 0.f ? d - P.L : d + P.L) : f;
}

__device__ __forceinline__ float4 offsets3(const P3 &P, const Work3 &w, double x, double y, double z, int cc)
{
    return make_float4(offset3(x, __ldg(w.centre + (cc & 1023)), P), offset3(y, __ldg(w.centre + ((cc >> 10) & 1023)), P),
                       offset3(z, __ldg(w.centre + (cc >> 20)), P), 0.f);
}

__device__ __forceinline__ bool resorting(const Work3 &w) { return *(volatile unsigned *)w.flag != 0u; }

// ---- predictor -------------------------------------------------------------------------------------

// Predictor on S, in place, and the offsets to the particles' cells (the cells of the last re-sort); a
// particle that has moved SKIN3 3h / 2 since then makes this step re-sort.
__global__ void __launch_bounds__(256) k3_predict(P3 P, Set3 S, Work3 w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float sp = 0.f;
    int moved = 0;
    const bool rs = resorting(w);
    if (i < P.n) {
        float4 ua = S.ua[i];
        const float4 aa = S.aa[i];
        ua.x += P.half_dt * aa.x;
        ua.y += P.half_dt * aa.y;
        ua.z += P.half_dt * aa.z;
        S.ua[i] = ua;
        double x = S.x[i] + P.half_dt_d * (double)ua.x, y = S.y[i] + P.half_dt_d * (double)ua.y,
               z = S.z[i] + P.half_dt_d * (double)ua.z;
        if (!(in_box(x, P.bitsL) && in_box(y, P.bitsL) && in_box(z, P.bitsL))) {   // rare: crossed a face
            x = wrap(x, P.L);
            y = wrap(y, P.L);
            z = wrap(z, P.L);
        }
        if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(ua.x) && isfinite(ua.y) && isfinite(ua.z))) {
            atomicOr(w.err, E3_NONFINITE);
            x = y = z = 0.0;
        }
        S.x[i] = x;
        S.y[i] = y;
        S.z[i] = z;
        sp = sqrtf(ua.x * ua.x + ua.y * ua.y + ua.z * ua.z);
        if (!isfinite(sp)) sp = 0.f;
        if (!rs) {
            const float4 xi = offsets3(P, w, x, y, z, w.cell_of[i]), rf = w.xi_ref[i];
            const float ex = xi.x - rf.x, ey = xi.y - rf.y, ez = xi.z - rf.z;
            moved = ex * ex + ey * ey + ez * ez > P.skin_max2;
            w.xi[i] = xi;
        }
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(sp));   // sp >= 0: bits order as values
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned *)w.umax) atomicMax(w.umax, m);
    if (__syncthreads_or(moved) && threadIdx.x == 0) *(volatile unsigned *)w.flag = 1u;
}

__global__ void k3_set_condition(Work3 w, cudaGraphConditionalHandle h)
{
    cudaGraphSetConditional(h, resorting(w) ? 1u : 0u);
}

// ---- re-sort (a conditional node: these run only when the flag is set) ------------------------------

__device__ __forceinline__ int cell_coord(const P3 &P, double x)
{
    return max(min((int)(x * P.inv_cell), P.nc - 1), 0);
}

__global__ void __launch_bounds__(256) k3_keys(P3 P, const Set3 S, Work3 w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    int key = -1;
    if (i < P.n) {
        key = (cell_coord(P, S.z[i]) * P.nc + cell_coord(P, S.y[i])) * P.nc + cell_coord(P, S.x[i]);
        w.key[i] = key;
    }
    // particles arrive in the previous cell order: one atomic per run of equal keys in a warp
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(grp) - 1;
    int base = 0;
    if (lane == leader && key >= 0) base = atomicAdd(&w.count[key], __popc(grp));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (i < P.n) w.rank[i] = base + __popc(grp & ((1u << lane) - 1u));
}

// Exclusive scan of the cell counts (low words) and of the non-empty cells (high words) by one block
// of 1024 threads, four cells a thread; lists the non-empty cells and clears the counts.
__global__ void __launch_bounds__(1024) k3_scan(P3 P, Work3 w)
{
    __shared__ unsigned long long part[32];
    __shared__ unsigned long long carry;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    if (t == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < P.ncell; base += 4096) {
        const int c0 = base + 4 * t;
        int v[4];
        unsigned long long sum = 0;
        for (int k = 0; k < 4; k++) {
            v[k] = c0 + k < P.ncell ? w.count[c0 + k] : 0;
            sum += (unsigned long long)v[k] | (v[k] > 0 ? 1ull << 32 : 0ull);
        }
        unsigned long long inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) part[wp] = inc;
        __syncthreads();
        if (wp == 0) {
            const unsigned long long x = part[lane];
            unsigned long long xi = x;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long u = __shfl_up_sync(0xffffffffu, xi, o);
                if (lane >= o) xi += u;
            }
            part[lane] = xi - x;
        }
        __syncthreads();
        unsigned long long run = carry + part[wp] + inc - sum;
        for (int k = 0; k < 4; k++) {
            if (c0 + k >= P.ncell) break;
            w.start[c0 + k] = (int)(run & 0xffffffffu);
            if (v[k] > 0) {
                w.tile[run >> 32].cell = c0 + k;
                run += (unsigned long long)v[k] | 1ull << 32;
            }
            w.count[c0 + k] = 0;
        }
        __syncthreads();
        if (t == 1023) carry = run;
        __syncthreads();
    }
    if (t == 0) {
        w.start[P.ncell] = (int)(carry & 0xffffffffu);
        *w.ntile = (int)(carry >> 32);
        *w.slots_used = 0;
        atomicAdd(w.rebuilds, 1u);
    }
}

__global__ void __launch_bounds__(256) k3_scatter(P3 P, Work3 w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < P.n) w.perm[w.start[w.key[i]] + w.rank[i]] = i;
}

// Adds up, over the particles, how many particles share each one's cell (w.key and w.count of k3_keys).
__global__ void __launch_bounds__(256) k3_crowd(int n, Work3 w, unsigned long long *sum)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned v = __reduce_add_sync(0xffffffffu, i < n ? (unsigned)w.count[w.key[i]] : 0u);
    if ((threadIdx.x & 31) == 0) atomicAdd(sum, (unsigned long long)v);
}

// The slots of each cell in particle-ID order: a warp per cell ranks each particle among the cell's by
// comparing IDs (all distinct), and moves its state to its place in T.
__global__ void __launch_bounds__(256) k3_order(P3 P, const Set3 S, Set3 T, Work3 w)
{
    const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= *w.ntile) return;
    const int c = w.tile[b].cell, s0 = w.start[c], cnt = w.start[c + 1] - s0;
    for (int e0 = 0; e0 < cnt; e0 += 32) {
        const bool live = e0 + lane < cnt;
        const int i = live ? w.perm[s0 + e0 + lane] : 0, id = live ? S.id[i] : 0;
        int rank = 0;
        for (int f0 = 0; f0 < cnt; f0 += 32) {
            const int other = f0 + lane < cnt ? S.id[w.perm[s0 + f0 + lane]] : 0x7fffffff;
            for (int k = 0; k < 32; k++) rank += __shfl_sync(0xffffffffu, other, k) < id;
        }
        if (live) {
            const int g = s0 + rank;
            T.x[g] = S.x[i];
            T.y[g] = S.y[i];
            T.z[g] = S.z[i];
            T.ua[g] = S.ua[i];
            T.qb[g] = S.qb[i];
            T.aa[g] = S.aa[i];
            T.id[g] = id;
            w.cell_of[g] = c % P.nc | (c / P.nc) % P.nc << 10 | c / (P.nc * P.nc) << 20;
        }
    }
}

// T back into S (the order now), with the offsets to the cells.
__global__ void __launch_bounds__(256) k3_copy_back(P3 P, Set3 S, const Set3 T, Work3 w)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    const double x = T.x[g], y = T.y[g], z = T.z[g];
    S.x[g] = x;
    S.y[g] = y;
    S.z[g] = z;
    S.ua[g] = T.ua[g];
    S.qb[g] = T.qb[g];
    S.aa[g] = T.aa[g];
    S.id[g] = T.id[g];
    const float4 xi = offsets3(P, w, x, y, z, w.cell_of[g]);
    w.xi[g] = xi;
    w.xi_ref[g] = xi;
}

// Cell of halo cell o (0..26) around (cx, cy, cz).
__device__ __forceinline__ int halo_cell(const P3 &P, int cx, int cy, int cz, int o)
{
    int qx = cx + o % 3 - 1, qy = cy + o / 3 % 3 - 1, qz = cz + o / 9 - 1;
    qx += qx < 0 ? P.nc : (qx >= P.nc ? -P.nc : 0);
    qy += qy < 0 ? P.nc : (qy >= P.nc ? -P.nc : 0);
    qz += qz < 0 ? P.nc : (qz >= P.nc ? -P.nc : 0);
    return (qz * P.nc + qy) * P.nc + qx;
}

// Position relative to the tile's centre of a particle with offsets xi in halo cell o (cell_lo: what FP32 drops of
// the cell's side).
__device__ __forceinline__ float4 tile_pos(const P3 &P, float4 xi, int o)
{
    auto at = [&](int k, float x) { return fmaf((float)k, P.cell_f, fmaf((float)k, P.cell_lo, x)); };
    return make_float4(at(o % 3 - 1, xi.x), at(o / 3 % 3 - 1, xi.y), at(o / 9 - 1, xi.z), xi.w);
}

__device__ __forceinline__ float dist2(float4 a, float4 b)
{
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// One block per tile: its slots (halo particles within the candidate radius of the box around its own
// particles, in cell order), then the candidate lists of its particles.  Four lanes test four
// consecutive slots of one particle, a vote places the hits.
__global__ void __launch_bounds__(T3) k3_lists(P3 P, Work3 w)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    float4 *pos = reinterpret_cast<float4 *>(dsm);
    __shared__ int off[28], start[27], wcnt[T3 / 32];
    __shared__ float box[6][T3 / 32];
    __shared__ int s_base, s_self;
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, wp = t >> 5;
    if (b >= *w.ntile) return;
    const int c = w.tile[b].cell, cx = c % P.nc, cy = (c / P.nc) % P.nc, cz = c / (P.nc * P.nc);
    const int i0 = w.start[c], ni = w.start[c + 1] - i0;
    if (t < 27) {
        const int q = halo_cell(P, cx, cy, cz, t);
        start[t] = w.start[q];
        off[t + 1] = w.start[q + 1] - w.start[q];
    }
    float lo[3] = {3e38f, 3e38f, 3e38f}, hi[3] = {-3e38f, -3e38f, -3e38f};
    for (int q = t; q < ni; q += T3) {
        const float4 x = w.xi[i0 + q];
        const float v[3] = {x.x, x.y, x.z};
        for (int k = 0; k < 3; k++) {
            lo[k] = fminf(lo[k], v[k]);
            hi[k] = fmaxf(hi[k], v[k]);
        }
    }
    for (int k = 0; k < 3; k++) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) {
            box[k][wp] = lo[k];
            box[3 + k][wp] = hi[k];
        }
    }
    __syncthreads();
    if (t == 0) {
        off[0] = 0;
        for (int o = 0; o < 27; o++) off[o + 1] += off[o];
        s_base = atomicAdd(w.slots_used, off[27]);   // 27 n over all tiles: each particle is in 27 halos
    }
    for (int k = 0; k < 3; k++)
        for (int v = 0; v < T3 / 32; v++) {
            lo[k] = fminf(lo[k], box[k][v]);
            hi[k] = fmaxf(hi[k], box[3 + k][v]);
        }
    __syncthreads();
    const int all = off[27], base = s_base;
    int kept = 0;
    for (int e0 = 0; e0 < all; e0 += T3) {
        const int e = e0 + t;
        bool keep = false;
        int o = 0, g = 0;
        float4 x;
        if (e < all) {
            int a = 0, z = 26;   // halo cell of entry e: the largest with off <= e
            while (a < z) {
                const int mid = (a + z + 1) >> 1;
                if (off[mid] <= e) a = mid;
                else z = mid - 1;
            }
            o = a;
            g = start[o] + (e - off[o]);
            x = tile_pos(P, w.xi[g], o);
            const float dx = fmaxf(fmaxf(lo[0] - x.x, x.x - hi[0]), 0.f), dy = fmaxf(fmaxf(lo[1] - x.y, x.y - hi[1]), 0.f),
                        dz = fmaxf(fmaxf(lo[2] - x.z, x.z - hi[2]), 0.f);
            keep = dx * dx + dy * dy + dz * dz < P.R2c * (1.f + 1e-5f);
        }
        const unsigned vote = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wcnt[wp] = __popc(vote);
        __syncthreads();
        int before = kept, total = kept;
        for (int v = 0; v < T3 / 32; v++) {
            if (v < wp) before += wcnt[v];
            total += wcnt[v];
        }
        if (keep) {
            const int s = before + __popc(vote & ((1u << lane) - 1u));
            w.slot[base + s] = (uint32_t)g | (uint32_t)o << ID_BITS;
            if (s < CAP3 - 1) pos[s] = x;
            if (g == i0) s_self = s;   // the tile's own particles are all kept: their slots follow each other
        }
        kept = total;
        __syncthreads();
    }
    if (t == 0) {
        w.tile[b].base = base;
        w.tile[b].count = kept;
        w.tile[b].self = s_self;
    }
    const bool staged = kept <= CAP3 - 1;
    const int self = s_self, l = lane & (LP - 1), shift = lane & ~(LP - 1);
    const size_t n4 = (size_t)P.n * LP;
    for (int q0 = wp * (32 / LP); q0 < ni; q0 += T3 / LP) {
        const int q = q0 + lane / LP;
        const bool live = q < ni;
        const int i = i0 + (live ? q : 0), si = self + (live ? q : 0);
        const float4 xi = staged ? pos[si] : w.xi[i];
        int cnt = 0;
        for (int s0 = 0; s0 < kept; s0 += LP) {
            const int s = s0 + l;
            bool in = live && s < kept && s != si;
            uint32_t entry = 0;
            if (in) {
                if (staged) {
                    in = dist2(xi, pos[s]) < P.R2c;
                    entry = (uint32_t)s << 4;
                } else {
                    const uint32_t ge = w.slot[base + s];
                    entry = ge & G_MASK;
                    in = dist2(xi, tile_pos(P, w.xi[entry], (int)(ge >> ID_BITS))) < P.R2c;
                }
            }
            const unsigned mine = __ballot_sync(0xffffffffu, in) >> shift & ((1u << LP) - 1u);
            const int k = cnt + __popc(mine & ((1u << l) - 1u));
            if (in && k < MAXC3) {
                const size_t word = (size_t)(k / GRP) * n4 + (size_t)i * LP + (k & (LP - 1));
                if (staged) reinterpret_cast<uint16_t *>(w.cand16 + word)[(k / LP) & 3] = (uint16_t)entry;
                else reinterpret_cast<uint32_t *>(w.cand32 + word)[(k / LP) & 3] = entry;
            }
            cnt += __popc(mine);
        }
        if (!live) continue;
        if (cnt > MAXC3) {
            if (l == 0) atomicOr(w.err, E3_NBR);
            cnt = MAXC3;
        }
        for (int k = (cnt & ~(LP - 1)) + l; k < (cnt + GRP - 1) / GRP * GRP; k += LP) {   // pad the last group
            if (k < cnt) continue;
            const size_t word = (size_t)(k / GRP) * n4 + (size_t)i * LP + (k & (LP - 1));
            if (staged) reinterpret_cast<uint16_t *>(w.cand16 + word)[(k / LP) & 3] = (uint16_t)(kept << 4);
            else reinterpret_cast<uint32_t *>(w.cand32 + word)[(k / LP) & 3] = NOENTRY;
        }
        if (l == 0) w.ncand[i] = cnt;
    }
}

// ---- the pair kernels' frame -------------------------------------------------------------------------

// A tile as its block sees it.
struct Here3 {
    Tile3 t;
    int i0, ni, cx, cy, cz;
    bool staged;
};

__device__ __forceinline__ bool begin3(const P3 &P, const Work3 &w, Here3 &h)
{
    if ((int)blockIdx.x >= *w.ntile) return false;
    const int4 v = *reinterpret_cast<const int4 *>(w.tile + blockIdx.x);
    h.t = Tile3{v.x, v.y, v.z, v.w};
    h.i0 = w.start[v.x];
    h.ni = w.start[v.x + 1] - h.i0;
    h.cx = v.x % P.nc;
    h.cy = (v.x / P.nc) % P.nc;
    h.cz = v.x / (P.nc * P.nc);
    h.staged = v.z <= CAP3 - 1;
    return true;
}

// Stages record x (positions first) of the tile's slots: fn(slot, particle, halo cell), and the empty slot.
template <typename Fn>
__device__ __forceinline__ void stage3(const P3 &P, const Work3 &w, const Here3 &h, float4 *pos, Fn &&fn)
{
#pragma unroll 2
    for (int s = threadIdx.x; s < h.t.count; s += blockDim.x) {
        const uint32_t e = __ldg(w.slot + h.t.base + s);
        fn(s, (int)(e & G_MASK), (int)(e >> ID_BITS));
    }
    if (threadIdx.x == 0) pos[h.t.count] = make_float4(P.far, P.far, P.far, 0.f);   // outside any support, V = 0
}

// The halo cell of particle j seen from tile h (tiles that are not staged).
__device__ __forceinline__ int halo_of(const P3 &P, const Work3 &w, const Here3 &h, int j)
{
    const int cc = w.cell_of[j];
    auto step = [&](int d) { return d > 1 ? d - P.nc : (d < -1 ? d + P.nc : d); };
    return (step((cc >> 20) - h.cz) + 1) * 9 + (step(((cc >> 10) & 1023) - h.cy) + 1) * 3 + step((cc & 1023) - h.cx) + 1;
}

// Element of a staged array of T at the byte offset of a 16-byte record.
template <typename T>
__device__ __forceinline__ const T &at3(const T *a, uint32_t o)
{
    return *reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(a) + o / (16 / sizeof(T)));
}

// Visits this lane's candidates of particle i, fn(entry): of a staged tile the byte offset of the slot |
// neighbour bit, else the particle | bit 31.  The next word is in flight while one is processed.
template <bool ST, typename Fn>
__device__ __forceinline__ void walk3(const P3 &P, const Work3 &w, int i, int l, int ncand, Fn &&fn)
{
    const size_t n4 = (size_t)P.n * LP;
    const int ng = (ncand + GRP - 1) / GRP;
    if (ST) {
        const uint2 *p = w.cand16 + (size_t)i * LP + l;
        uint2 nxt = ng > 0 ? __ldg(p) : make_uint2(0u, 0u);
        for (int g = 0; g < ng; g++) {
            const uint2 e = nxt;
            p += n4;
            if (g + 1 < ng) nxt = __ldg(p);
            fn(e.x & 0xffffu);
            fn(e.x >> 16);
            fn(e.y & 0xffffu);
            fn(e.y >> 16);
        }
    } else {
        const uint4 *p = w.cand32 + (size_t)i * LP + l;
        for (int g = 0; g < ng; g++, p += n4) {
            const uint4 e = __ldg(p);
            if (e.x != NOENTRY) fn(e.x);
            if (e.y != NOENTRY) fn(e.y);
            if (e.z != NOENTRY) fn(e.z);
            if (e.w != NOENTRY) fn(e.w);
        }
    }
}

__device__ __forceinline__ float quad_sum(float v)
{
#pragma unroll
    for (int o = 1; o < LP; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float2 quad_sum(float2 v) { return f2(quad_sum(v.x), quad_sum(v.y)); }

// s + e += the other lane's (two-sum: the rounding of the sum goes into e)
__device__ __forceinline__ void quad_two_sum(float &s, float &e)
{
#pragma unroll
    for (int o = 1; o < LP; o <<= 1) {
        const float t = __shfl_xor_sync(0xffffffffu, s, o), f = __shfl_xor_sync(0xffffffffu, e, o);
        const float r = s + t, bb = r - s;
        e += f + ((s - (r - bb)) + (t - bb));
        s = r;
    }
}

// Pair geometry d = x_i - x_j (xy as one two-lane value), |d|^2, 1/|d|, |d|, and the kernel's powers
// t_k = max(k - r/h, 0) and t_k^4 of the quintic kernel (Eq. 18): (t3, t2) travel together.
struct Pair3 {
    float2 dxy, t, q;
    float dz, r2, rinv, r, t1, q1;
};

__device__ __forceinline__ Pair3 pair3(const P3 &P, float4 a, float4 b)
{
    Pair3 g;
    g.dxy = sub2(f2(a.x, a.y), f2(b.x, b.y));
    g.dz = a.z - b.z;
    g.r2 = fmaf(g.dxy.x, g.dxy.x, fmaf(g.dxy.y, g.dxy.y, g.dz * g.dz));
    g.rinv = ann::rsqrt_approx(g.r2);
    g.r = g.r2 * g.rinv;
    const float bq = g.r * P.inv_h;
    g.t = add2(f2(3.f, 2.f), bc(-bq));
    g.t = f2(fmaxf(g.t.x, 0.f), fmaxf(g.t.y, 0.f));
    g.t1 = fmaxf(1.f - bq, 0.f);
    const float2 s = mul2(g.t, g.t);
    const float s1 = g.t1 * g.t1;
    g.q = mul2(s, s);
    g.q1 = s1 * s1;
    return g;
}

// W(r), and F with grad_i W = F d.
__device__ __forceinline__ float w_of(const P3 &P, const Pair3 &g)
{
    const float2 v = mul2(g.q, g.t);
    return fmaf(P.ad, v.x, fmaf(P.kw6, v.y, P.kw15 * (g.q1 * g.t1)));
}
__device__ __forceinline__ float f_of(const P3 &P, const Pair3 &g)
{
    return fmaf(P.kf75, g.q1, fmaf(P.kf30, g.q.y, P.kf5 * g.q.x)) * g.rinv;
}

// A warp's particles: 8 at a time, all lanes in step (lanes past the last particle repeat it).
#define FOR_PARTICLES3(h)                                                                                             \
    for (int q0 = (int)(threadIdx.x >> 5) * (32 / LP); q0 < (h).ni; q0 += (int)blockDim.x / LP)

struct Own3 {
    int i, s, l;   // particle, its slot, lane
    bool store;    // lane 0 of a particle writes its results
};

__device__ __forceinline__ Own3 own3(const Here3 &h, int q0)
{
    const int lane = threadIdx.x & 31, q = q0 + lane / LP, r = min(q, h.ni - 1);
    return Own3{h.i0 + r, h.t.self + r, lane & (LP - 1), q < h.ni && (lane & (LP - 1)) == 0};
}

// ---- filter: neighbour bits, volumes ------------------------------------------------------------------

__device__ __noinline__ bool support3(const P3 &P, const Set3 &S, int i, int j)
{
    const double ex = min_image(S.x[i] - S.x[j], P.L), ey = min_image(S.y[i] - S.y[j], P.L),
                 ez = min_image(S.z[i] - S.z[j], P.L);
    return ex * ex + ey * ey + ez * ez < P.R2d;
}

template <bool ST>
__device__ __forceinline__ void filter_tile(const P3 &P, const Set3 &S, const Work3 &w, const Here3 &h, const float4 *pos)
{
    FOR_PARTICLES3(h)
    {
        const Own3 o = own3(h, q0);
        const float4 xi = ST ? pos[o.s] : w.xi[o.i];
        float s = 0.f;
        int nn = 0;
        auto test = [&](int j, float4 xj) {   // j: for a pair in the band, decided in FP64
            const Pair3 g = pair3(P, xi, xj);
            s += w_of(P, g);
            bool in = g.r2 < P.R2lo;
            if (!in && g.r2 < P.R2hi) in = support3(P, S, o.i, ST ? (int)(w.slot[h.t.base + j] & G_MASK) : j);
            nn += in;
            return (uint32_t)in;
        };
        const size_t n4 = (size_t)P.n * LP;
        const int ng = (w.ncand[o.i] + GRP - 1) / GRP;
        if (ST) {   // plain loads: this kernel writes the words; a word is stored only when a bit changed
            uint2 *p = w.cand16 + (size_t)o.i * LP + o.l;
            uint2 nxt = ng > 0 ? *p : make_uint2(0u, 0u);
            for (int g = 0; g < ng; g++, p += n4) {
                const uint2 e = nxt;
                if (g + 1 < ng) nxt = p[n4];
                auto bit = [&](uint32_t v) { return (v & 0xfff0u) | test((int)(v >> 4), at3(pos, v & 0xfff0u)); };
                const uint32_t e0 = bit(e.x & 0xffffu), e1 = bit(e.x >> 16), e2 = bit(e.y & 0xffffu), e3 = bit(e.y >> 16);
                const uint2 v = make_uint2(e0 | e1 << 16, e2 | e3 << 16);
                if (v.x != e.x || v.y != e.y) *p = v;
            }
        } else {
            uint4 *p = w.cand32 + (size_t)o.i * LP + o.l;
            for (int g = 0; g < ng; g++, p += n4) {
                uint4 e = *p;
                auto bit = [&](uint32_t v) {
                    if (v == NOENTRY) return v;
                    const int j = (int)(v & G_MASK);
                    return (uint32_t)j | test(j, tile_pos(P, w.xi[j], halo_of(P, w, h, j))) << 31;
                };
                e.x = bit(e.x);
                e.y = bit(e.y);
                e.z = bit(e.z);
                e.w = bit(e.w);
                *p = e;
            }
        }
        __syncwarp();
        s = P.W0 + quad_sum(s);
#pragma unroll
        for (int v = 1; v < LP; v <<= 1) nn += __shfl_xor_sync(0xffffffffu, nn, v);
        if (o.store) {
            if (nn > MAXN3) atomicOr(w.err, E3_NBR);
            w.nnbr[o.i] = nn;
            w.sumW[o.i] = s;
            w.xv[o.i] = make_float4(xi.x, xi.y, xi.z, 1.f / s);
        }
    }
}

__global__ void __launch_bounds__(TF3, BF3) k3_filter(P3 P, const Set3 S, Work3 w)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    float4 *pos = reinterpret_cast<float4 *>(dsm);
    if (blockIdx.x == 0 && threadIdx.x == 0) *(volatile unsigned *)w.flag = 0u;   // the re-sort kernels have run
    Here3 h;
    if (!begin3(P, w, h)) return;
    if (h.staged) {
        stage3(P, w, h, pos, [&](int s, int g, int o) { pos[s] = tile_pos(P, w.xi[g], o); });
        __syncthreads();
        filter_tile<true>(P, S, w, h, pos);
    } else {
        filter_tile<false>(P, S, w, h, pos);
    }
}

// B = alpha^-1 of a symmetric alpha (Eq. 22); flags a non-positive determinant.
__device__ __forceinline__ void invert_alpha(const float a[3][3], float *B, unsigned *err)
{
    float det = a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0]) +
                a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]);
    if (!(det > 0.f)) atomicOr(err, E3_ALPHA);
    float id = 1.f / det;
    B[0] = (a[1][1] * a[2][2] - a[1][2] * a[2][1]) * id;
    B[1] = (a[0][2] * a[2][1] - a[0][1] * a[2][2]) * id;
    B[2] = (a[0][1] * a[1][2] - a[0][2] * a[1][1]) * id;
    B[3] = (a[1][2] * a[2][0] - a[1][0] * a[2][2]) * id;
    B[4] = (a[0][0] * a[2][2] - a[0][2] * a[2][0]) * id;
    B[5] = (a[0][2] * a[1][0] - a[0][0] * a[1][2]) * id;
    B[6] = (a[1][0] * a[2][1] - a[1][1] * a[2][0]) * id;
    B[7] = (a[0][1] * a[2][0] - a[0][0] * a[2][1]) * id;
    B[8] = (a[0][0] * a[1][1] - a[0][1] * a[1][0]) * id;
}

// Q in full.
__device__ __forceinline__ void full_q(const float *q, float Q[3][3])
{
    Q[0][0] = q[0]; Q[0][1] = q[1]; Q[0][2] = q[2];
    Q[1][0] = q[1]; Q[1][1] = q[3]; Q[1][2] = q[4];
    Q[2][0] = q[2]; Q[2][1] = q[4]; Q[2][2] = -q[0] - q[3];
}

// Eq. (24) with Eqs. (2) and (7): m = S + Gamma H, projected onto the symmetric traceless part.
__device__ void q_rate3(const P3 &P, const float *q, const float D[3][3], const float *lq, float *m5)
{
    float Q[3][3], LQ[3][3], M[3][3], E[3][3], Om[3][3];
    full_q(q, Q);
    full_q(lq, LQ);
    float QD = 0.f;
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) {
            E[a][b] = 0.5f * (D[a][b] + D[b][a]);
            Om[a][b] = 0.5f * (D[a][b] - D[b][a]);
            M[a][b] = Q[a][b] + (a == b ? P.c_shift : 0.f);
            QD += Q[a][b] * D[a][b];
        }
    float trQ2 = 0.f, Q2[3][3];
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) {
            Q2[a][b] = Q[a][0] * Q[0][b] + Q[a][1] * Q[1][b] + Q[a][2] * Q[2][b];
        }
    trQ2 = Q2[0][0] + Q2[1][1] + Q2[2][2];
    float m[3][3];
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) {
            // (lambda E + Omega) M + M (lambda E - Omega) - 2 lambda M (Q : grad u)
            float s = 0.f;
            for (int c = 0; c < 3; c++)
                s += (P.lambda * E[a][c] + Om[a][c]) * M[c][b] + M[a][c] * (P.lambda * E[c][b] - Om[c][b]);
            s -= 2.f * P.lambda * M[a][b] * QD;
            float H = -P.A * Q[a][b] + P.B * (Q2[a][b] - (a == b ? trQ2 / 3.f : 0.f)) - P.C * Q[a][b] * trQ2 +
                      P.K * LQ[a][b];
            m[a][b] = s + P.Gamma * H;
        }
    float tr = m[0][0] + m[1][1] + m[2][2];
    m5[0] = m[0][0] - tr / 3.f;
    m5[1] = 0.5f * (m[0][1] + m[1][0]);
    m5[2] = 0.5f * (m[0][2] + m[2][0]);
    m5[3] = m[1][1] - tr / 3.f;
    m5[4] = 0.5f * (m[1][2] + m[2][1]);
}

// ---- pass 1: correction tensor, velocity gradient, continuity ------------------------------------------

// One walk gives alpha and the raw sums of the velocity gradient; B enters after the walk, since the
// corrected quantities are contractions of B with sums that do not involve it:
//   alpha_ab = -sum_j V_j F d_a d_b                                                   (Eq. 22)
//   grad u   = rhs B,  rhs_cl = sum_j V_j (u_j - u_i)_c F d_l                         (Eq. 20)
//   k / rho  = sum_j V_j F (u_i - u_j) . B d = -sum_ab B_ab rhs_ab                    (Eq. 25)
// The symmetric products d_a d_b travel as the two-lane values (00, 01), (02, 12), (11, 22).
// (The Laplacian of Q could be summed here the same way, as six sums per component: 30 more
// accumulators, which left 16 warps an SM; in pass 2, with B known, it is one sum per component.)
template <bool ST>
__device__ __forceinline__ void pass1_tile(const P3 &P, const Set3 &S, const Work3 &w, const Here3 &h, const float4 *xs,
                                           const float4 *us)
{
    FOR_PARTICLES3(h)
    {
        const Own3 o = own3(h, q0);
        const float4 xi = ST ? xs[o.s] : w.xv[o.i], ui = ST ? us[o.s] : S.ua[o.i];
        float2 al0 = f2(0.f, 0.f), al1 = al0, al2 = al0, ra0 = al0, ra1 = al0, ra2 = al0;   // ra_c: (rhs_c0, rhs_c1)
        float rz0 = 0.f, rz1 = 0.f, rz2 = 0.f;                                             // rhs_c2
        walk3<ST>(P, w, o.i, o.l, w.ncand[o.i], [&](uint32_t e) {
            float4 xj, uj;
            if (ST) {
                xj = at3(xs, e & 0xfff0u);
                uj = at3(us, e & 0xfff0u);
            } else {
                const int j = (int)(e & G_MASK);
                xj = tile_pos(P, w.xv[j], halo_of(P, w, h, j));
                uj = S.ua[j];
            }
            const Pair3 g = pair3(P, xi, xj);
            const float vf = xj.w * f_of(P, g);   // V_j F
            const float2 exy = mul2(bc(vf), g.dxy);
            const float ez = vf * g.dz;
            al0 = fma2(bc(exy.x), g.dxy, al0);
            al1 = fma2(bc(g.dz), exy, al1);
            al2 = f2(fmaf(exy.y, g.dxy.y, al2.x), fmaf(ez, g.dz, al2.y));
            const float2 duxy = sub2(f2(uj.x, uj.y), f2(ui.x, ui.y));   // u_j - u_i
            const float duz = uj.z - ui.z;
            ra0 = fma2(bc(duxy.x), exy, ra0);
            ra1 = fma2(bc(duxy.y), exy, ra1);
            ra2 = fma2(bc(duz), exy, ra2);
            rz0 = fmaf(duxy.x, ez, rz0);
            rz1 = fmaf(duxy.y, ez, rz1);
            rz2 = fmaf(duz, ez, rz2);
        });
        __syncwarp();
        al0 = quad_sum(al0);
        al1 = quad_sum(al1);
        al2 = quad_sum(al2);
        ra0 = quad_sum(ra0);
        ra1 = quad_sum(ra1);
        ra2 = quad_sum(ra2);
        rz0 = quad_sum(rz0);
        rz1 = quad_sum(rz1);
        rz2 = quad_sum(rz2);
        if (!o.store) continue;
        const int i = o.i;
        const float a[3][3] = {{-al0.x, -al0.y, -al1.x}, {-al0.y, -al2.x, -al1.y}, {-al1.x, -al1.y, -al2.y}};
        float B[9];   // symmetric, as alpha is
        invert_alpha(a, B, w.err);
        const float rhs[3][3] = {{ra0.x, ra0.y, rz0}, {ra1.x, ra1.y, rz1}, {ra2.x, ra2.y, rz2}};
        float kc = 0.f;
        for (int c = 0; c < 3; c++)
            for (int b = 0; b < 3; b++) {
                w.gu[(size_t)(3 * c + b) * P.n + i] = rhs[c][0] * B[b] + rhs[c][1] * B[3 + b] + rhs[c][2] * B[6 + b];
                kc -= B[3 * c + b] * rhs[c][b];
            }
        const float4 qb = S.qb[i];
        const float dr = S.aa[i].w, k_i = P.rho0 * (1.f + dr) * kc;
        w.b0[i] = make_float4(B[0], B[1], B[2], B[4]);
        w.b1[i] = make_float2(B[5], B[8]);
        w.dq[i] = make_float4(dr + P.half_dt * k_i / P.rho0, ui.w, qb.x, qb.y);
        w.q2[i] = make_float2(qb.z, qb.w);
        w.k[i] = k_i;
    }
}

__global__ void __launch_bounds__(T13, B13) k3_pass1(P3 P, const Set3 S, Work3 w)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    float4 *xs = reinterpret_cast<float4 *>(dsm), *us = xs + CAP3;
    Here3 h;
    if (!begin3(P, w, h)) return;
    if (h.staged) {
        stage3(P, w, h, xs, [&](int s, int g, int o) {
            xs[s] = tile_pos(P, w.xv[g], o);
            us[s] = S.ua[g];
        });
        if (threadIdx.x == 32) us[h.t.count] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        pass1_tile<true>(P, S, w, h, xs, us);
    } else {
        pass1_tile<false>(P, S, w, h, xs, us);
    }
}

// ---- pass 2: density filter, equation of state, Laplacian of Q, Q rate ------------------------------------

// lap Q_c = 2 sum_j V_j F (Q_i - Q_j)_c (d . B d) / r^2                                (Eq. 21)
template <bool ST>
__device__ __forceinline__ void pass2_tile(const P3 &P, const Set3 &S, const Work3 &w, const Here3 &h, const float4 *xs,
                                           const float4 *ds, const float2 *qs)
{
    const float c0 = fmaxf(10.f * __uint_as_float(*w.umax), P.c0_min);
    FOR_PARTICLES3(h)
    {
        const Own3 o = own3(h, q0);
        const int i = o.i;
        const float4 xi = ST ? xs[o.s] : w.xv[i], di = ST ? ds[o.s] : w.dq[i], b0 = w.b0[i];
        const float2 qi = ST ? qs[o.s] : w.q2[i], b1 = w.b1[i];
        // (d . B d) = d_x (B d)_x + ...; the off-diagonal entries count twice
        const float2 bx = f2(b0.x, b0.w);   // (B11, B22)
        const float b12 = 2.f * b0.y;
        const float2 bz = f2(2.f * b0.z, 2.f * b1.x);   // (2 B13, 2 B23)
        float num = 0.f;   // Eq. (28) on the deviations (rho0 factors out of the filter)
        float2 L0 = f2(0.f, 0.f), L1 = L0;
        float L4 = 0.f;
        walk3<ST>(P, w, i, o.l, w.ncand[i], [&](uint32_t e) {
            float4 xj, dj;
            float2 qj;
            if (ST) {
                xj = at3(xs, e & 0xfff0u);
                dj = at3(ds, e & 0xfff0u);
                qj = at3(qs, e & 0xfff0u);
            } else {
                const int j = (int)(e & G_MASK);
                xj = tile_pos(P, w.xv[j], halo_of(P, w, h, j));
                dj = w.dq[j];
                qj = w.q2[j];
            }
            const Pair3 g = pair3(P, xi, xj);
            num = fmaf(di.x - dj.x, w_of(P, g), num);
            const float2 t = fma2(bz, bc(g.dz), mul2(bx, g.dxy));
            const float dBd = fmaf(g.dxy.x, fmaf(b12, g.dxy.y, t.x), fmaf(g.dxy.y, t.y, b1.y * g.dz * g.dz));
            const float wt = xj.w * f_of(P, g) * (g.rinv * g.rinv) * dBd;
            L0 = fma2(bc(wt), sub2(f2(di.z, di.w), f2(dj.z, dj.w)), L0);
            L1 = fma2(bc(wt), sub2(qi, qj), L1);
            L4 = fmaf(wt, di.y - dj.y, L4);
        });
        __syncwarp();
        num = quad_sum(num);
        L0 = quad_sum(L0);
        L1 = quad_sum(L1);
        L4 = quad_sum(L4);
        if (!o.store) continue;
        const float q[5] = {di.y, di.z, di.w, qi.x, qi.y};
        const float lap[5] = {2.f * L4, 2.f * L0.x, 2.f * L0.y, 2.f * L1.x, 2.f * L1.y};
        const size_t n = (size_t)P.n;
        float D[3][3];
        for (int c = 0; c < 9; c++) D[c / 3][c % 3] = w.gu[c * n + i];
        float m5[5], qn[5];
        q_rate3(P, q, D, lap, m5);
        for (int c = 0; c < 5; c++) {
            qn[c] = q[c] + P.dt * m5[c];
            w.m[c * n + i] = m5[c];
            w.lap[c * n + i] = lap[c];
        }
        w.qn[i] = make_float4(qn[0], qn[1], qn[2], qn[3]);
        w.qn4[i] = qn[4];
        const float dhat = di.x - P.beta * num / w.sumW[i];
        w.dhat[i] = dhat;
        // Eq. (26): (rho / rho0)^gamma - 1 = expm1(gamma log1p(delta)), accurate for small delta
        const float p = P.rho0 * c0 * c0 / P.gamma_eos * expm1f(P.gamma_eos * log1pf(dhat));
        const float rho = P.rho0 * (1.f + dhat);
        const float4 ua = S.ua[i];
        w.p[i] = p;
        w.pu[i] = make_float4(p / (rho * rho), ua.x, ua.y, ua.z);
    }
}

__global__ void __launch_bounds__(T23, B23) k3_pass2(P3 P, const Set3 S, Work3 w)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    float4 *xs = reinterpret_cast<float4 *>(dsm), *ds = xs + CAP3;
    float2 *qs = reinterpret_cast<float2 *>(ds + CAP3);
    Here3 h;
    if (!begin3(P, w, h)) return;
    if (h.staged) {
        stage3(P, w, h, xs, [&](int s, int g, int o) {
            xs[s] = tile_pos(P, w.xv[g], o);
            ds[s] = w.dq[g];
            qs[s] = w.q2[g];
        });
        if (threadIdx.x == 32) {
            ds[h.t.count] = make_float4(0.f, 0.f, 0.f, 0.f);
            qs[h.t.count] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        pass2_tile<true>(P, S, w, h, xs, ds, qs);
    } else {
        pass2_tile<false>(P, S, w, h, xs, ds, qs);
    }
}

// ---- pass 3: momentum, artificial displacement, corrector ------------------------------------------------

// As in pass 1 the sums are raw and B is applied after the walk:
//   pressure and viscous terms  B sum_j V_j F [ -rho_i (p_i/rho_i^2 + p_j/rho_j^2) + kv (u_ij . d) / r^2 ] d,
//                               kv = 10 nu rho0 / rho_i
//   div Q^{n+1}                 sum_b B_bl R_cb,l,  R_cb,l = sum_j V_j F (Q_j - Q_i)_cb d_l
template <bool ST>
__device__ __forceinline__ void pass3_tile(const P3 &P, const Set3 &S, const Work3 &w, const Here3 &h, const float4 *xs,
                                           const float4 *ps, const float4 *qs, const float *q4)
{
    FOR_PARTICLES3(h)
    {
        const Own3 o = own3(h, q0);
        const int i = o.i;
        const float4 xi = ST ? xs[o.s] : w.xv[i], pi = ST ? ps[o.s] : w.pu[i], qi = ST ? qs[o.s] : w.qn[i];
        const float qi4 = ST ? q4[o.s] : w.qn4[i], dhat = w.dhat[i], ri = P.rho0 * (1.f + dhat);
        const float kv = 10.f * P.nu * P.rho0 / ri, nri = -ri, pci = nri * pi.x;
        float2 fw = f2(0.f, 0.f), su = fw, sd = fw, sc = fw, R[5] = {};
        float fz = 0.f, suz = 0.f, sr = 0.f, sdz = 0.f, scz = 0.f, Rz[5] = {};
        auto add = [&](float4 xj, float4 pj, float4 qj, float qj4, bool in) {
            const Pair3 g = pair3(P, xi, xj);
            const float W = w_of(P, g), vf = xj.w * f_of(P, g);
            const float2 du = sub2(f2(pi.y, pi.z), f2(pj.y, pj.z));   // u_i - u_j
            const float duz = pi.w - pj.w;
            const float ud = fmaf(du.x, g.dxy.x, fmaf(du.y, g.dxy.y, duz * g.dz));
            const float rinv2 = g.rinv * g.rinv;
            const float coef = fmaf(kv, ud * rinv2, fmaf(nri, pj.x, pci));
            const float2 exy = mul2(bc(vf), g.dxy);
            const float ez = vf * g.dz;
            fw = fma2(bc(coef), exy, fw);
            fz = fmaf(coef, ez, fz);
            const float2 dqa = sub2(f2(qj.x, qj.y), f2(qi.x, qi.y)), dqb = sub2(f2(qj.z, qj.w), f2(qi.z, qi.w));
            const float dq[5] = {dqa.x, dqa.y, dqb.x, dqb.y, qj4 - qi4};
#pragma unroll
            for (int c = 0; c < 5; c++) {
                R[c] = fma2(bc(dq[c]), exy, R[c]);
                Rz[c] = fmaf(dq[c], ez, Rz[c]);
            }
            su = fma2(bc(W), du, su);
            suz = fmaf(W, duz, suz);
            // Eq. (29) sums over the neighbours only.  sum_j d / r^3 nearly cancels (terms ~1/r^2, sum ~
            // their imbalance): compensated (Kahan) summation keeps it to FP32 rounding of the sum
            // (a candidate that is no neighbour adds 0 and the pending compensation).  sc holds y - (t - sd).
            const float rinv3 = in ? rinv2 * g.rinv : 0.f;
            const float2 y = fma2(bc(rinv3), g.dxy, sc), t = add2(sd, y);
            sc = sub2(y, sub2(t, sd));
            sd = t;
            const float yz = fmaf(rinv3, g.dz, scz), tz = sdz + yz;
            scz = yz - (tz - sdz);
            sdz = tz;
            sr += in ? g.r : 0.f;
        };
        walk3<ST>(P, w, i, o.l, w.ncand[i], [&](uint32_t e) {
            if (ST) {
                const uint32_t off = e & 0xfff0u;
                add(at3(xs, off), at3(ps, off), at3(qs, off), at3(q4, off), e & 1u);
            } else {
                const int j = (int)(e & G_MASK);
                add(tile_pos(P, w.xv[j], halo_of(P, w, h, j)), w.pu[j], w.qn[j], w.qn4[j], e >> 31);
            }
        });
        __syncwarp();
        fw = quad_sum(fw);
        fz = quad_sum(fz);
        su = quad_sum(su);
        suz = quad_sum(suz);
        sr = quad_sum(sr);
#pragma unroll
        for (int c = 0; c < 5; c++) {
            R[c] = quad_sum(R[c]);
            Rz[c] = quad_sum(Rz[c]);
        }
        float ex = sc.x, ey = sc.y, ez = scz;   // the lanes' sums join without losing their compensation
        quad_two_sum(sd.x, ex);
        quad_two_sum(sd.y, ey);
        quad_two_sum(sdz, ez);
        if (!o.store) continue;
        const float4 b0 = w.b0[i];
        const float2 b1 = w.b1[i];
        const float B[3][3] = {{b0.x, b0.y, b0.z}, {b0.y, b0.w, b1.x}, {b0.z, b1.x, b1.y}};
        float BR[6][3];   // [component][b] = sum_l B_bl R_l; component 5 is Q33 = -Q11 - Q22
        for (int c = 0; c < 5; c++)
            for (int b = 0; b < 3; b++) BR[c][b] = B[b][0] * R[c].x + B[b][1] * R[c].y + B[b][2] * Rz[c];
        for (int b = 0; b < 3; b++) BR[5][b] = -BR[0][b] - BR[3][b];
        const float dv[3] = {BR[0][0] + BR[1][1] + BR[2][2], BR[1][0] + BR[3][1] + BR[4][2], BR[2][0] + BR[4][1] + BR[5][2]};
        const float ui[3] = {pi.y, pi.z, pi.w};
        const float sdv[3] = {sd.x + ex, sd.y + ey, sdz + ez};
        const int m = w.nnbr[i];
        float an[3], un[3], apd[3] = {0.f, 0.f, 0.f};
        for (int c = 0; c < 3; c++) an[c] = B[c][0] * fw.x + B[c][1] * fw.y + B[c][2] * fz - P.zeta / ri * dv[c];
        if (P.apd) {
            const float uv = sqrtf(su.x * su.x + su.y * su.y + suz * suz) / w.sumW[i];
            const float r0 = m > 0 ? sr / (float)m : 0.f;
            for (int c = 0; c < 3; c++) apd[c] = sdv[c] * r0 * r0 * uv * P.dt;
        }
        for (int c = 0; c < 3; c++) un[c] = ui[c] + P.half_dt * an[c];
        double x = S.x[i] + P.half_dt_d * (double)un[0] + (double)apd[0];
        double y = S.y[i] + P.half_dt_d * (double)un[1] + (double)apd[1];
        double z = S.z[i] + P.half_dt_d * (double)un[2] + (double)apd[2];
        if (!(in_box(x, P.bitsL) && in_box(y, P.bitsL) && in_box(z, P.bitsL))) {
            x = wrap(x, P.L);
            y = wrap(y, P.L);
            z = wrap(z, P.L);
        }
        const float dr = dhat + P.half_dt * w.k[i] / P.rho0;
        const bool ok = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(un[0]) && isfinite(un[1]) && isfinite(un[2]) &&
                        isfinite(dr) && isfinite(qi.x) && isfinite(qi.y) && isfinite(qi.z) && isfinite(qi.w) && isfinite(qi4);
        if (!ok) {
            atomicOr(w.err, E3_NONFINITE);
            x = y = z = 0.0;
        }
        S.x[i] = x;
        S.y[i] = y;
        S.z[i] = z;
        S.ua[i] = make_float4(un[0], un[1], un[2], qi.x);
        S.qb[i] = make_float4(qi.y, qi.z, qi.w, qi4);
        S.aa[i] = make_float4(an[0], an[1], an[2], dr);
    }
}

__global__ void __launch_bounds__(T33, B33) k3_pass3(P3 P, Set3 S, Work3 w)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    float4 *xs = reinterpret_cast<float4 *>(dsm), *ps = xs + CAP3, *qs = ps + CAP3;
    float *q4 = reinterpret_cast<float *>(qs + CAP3);
    if (blockIdx.x == 0 && threadIdx.x == 0) *w.umax = 0u;   // pass 2 has consumed it
    Here3 h;
    if (!begin3(P, w, h)) return;
    if (h.staged) {
        stage3(P, w, h, xs, [&](int s, int g, int o) {
            xs[s] = tile_pos(P, w.xv[g], o);
            ps[s] = w.pu[g];
            qs[s] = w.qn[g];
            q4[s] = w.qn4[g];
        });
        if (threadIdx.x == 32) {
            ps[h.t.count] = qs[h.t.count] = make_float4(0.f, 0.f, 0.f, 0.f);
            q4[h.t.count] = 0.f;
        }
        __syncthreads();
        pass3_tile<true>(P, S, w, h, xs, ps, qs, q4);
    } else {
        pass3_tile<false>(P, S, w, h, xs, ps, qs, q4);
    }
}

constexpr int SMEM3_POS = CAP3 * 16, SMEM3_1 = CAP3 * 32, SMEM3_2 = CAP3 * 40, SMEM3_3 = CAP3 * 52;

// ---- fields ------------------------------------------------------------------------------------------------

struct Planes3 {
    const float *p[9];
    int stride[9];   // floats from one particle to the next
};

// dst[id[g] * ncomp + c] = component c of slot g (ID order, interleaved, FP64)
__global__ void k3_to_id(int n, int ncomp, Planes3 pl, const int *id, double *dst)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
#pragma unroll
    for (int c = 0; c < 9; c++)
        if (c < ncomp) dst[(size_t)id[g] * ncomp + c] = (double)pl.p[c][(size_t)g * pl.stride[c]];
}

__global__ void k3_pos_to_id(int n, const double *x, const double *y, const double *z, const int *id, double *dst)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    dst[3 * (size_t)id[g]] = x[g];
    dst[3 * (size_t)id[g] + 1] = y[g];
    dst[3 * (size_t)id[g] + 2] = z[g];
}

__global__ void k3_int_to_id(int n, const int *v, const int *id, double *dst)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) dst[id[g]] = (double)v[g];
}

inline unsigned nb3(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// A named NVTX range for the lifetime of the object (profilers show the library's calls).
struct Range3 {
    explicit Range3(const char *name) { nvtxRangePushA(name); }
    ~Range3() { nvtxRangePop(); }
    Range3(const Range3 &) = delete;
    Range3 &operator=(const Range3 &) = delete;
};

}  // namespace

struct ann3_ctx {
    ann3_params prm;
    P3 P;
    Set3 S, T;
    Work3 w;
    std::vector<void *> allocs;
    cudaStream_t s = nullptr, aux = nullptr;   // aux captures the body of the step graph's conditional node
    cudaGraphExec_t exec = nullptr;
    bool have = false;
    int64_t steps = 0;
    std::string last_err;
    double *tmp = nullptr;         // device staging for ann3_get_field (9n doubles)
    int nc_fine = 0;               // cells a side at their least width
    double *centre = nullptr;      // Work3::centre, nc_fine values
};

namespace {

template <typename T>
cudaError_t alloc3(ann3_ctx *c, T *&p, size_t count)
{
    void *v = nullptr;
    cudaError_t e = cudaMalloc(&v, std::max<size_t>(count, 1) * sizeof(T));
    if (e) return e;
    c->allocs.push_back(v);
    p = static_cast<T *>(v);
    return cudaMemsetAsync(v, 0, std::max<size_t>(count, 1) * sizeof(T), c->s);
}

cudaError_t alloc_set(ann3_ctx *c, Set3 &S, size_t n)
{
    cudaError_t e = alloc3(c, S.x, n);
    if (!e) e = alloc3(c, S.y, n);
    if (!e) e = alloc3(c, S.z, n);
    if (!e) e = alloc3(c, S.ua, n);
    if (!e) e = alloc3(c, S.qb, n);
    if (!e) e = alloc3(c, S.aa, n);
    if (!e) e = alloc3(c, S.id, n);
    return e;
}

// The step graph: predictor -> set the condition -> IF (re-sort flag) { sort, tile and candidate lists }
// -> filter, passes 1 to 3.
cudaError_t capture3(ann3_ctx *c)
{
    const P3 &P = c->P;
    const Set3 &S = c->S;
    const Work3 &w = c->w;
    const unsigned g = nb3((size_t)P.n), nt = (unsigned)P.nblk;
    cudaGraph_t gr = nullptr;
    cudaError_t e = cudaGraphCreate(&gr, 0);
    if (e) return e;
    e = cudaStreamBeginCaptureToGraph(c->s, gr, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e) {
        cudaGraphDestroy(gr);
        return e;
    }
    cudaGraphConditionalHandle h = 0;
    cudaError_t ec = cudaGraphConditionalHandleCreate(&h, gr, 0, cudaGraphCondAssignDefault);
    if (!ec) {
        k3_predict<<<g, 256, 0, c->s>>>(P, S, w);
        k3_set_condition<<<1, 1, 0, c->s>>>(w, h);
        ec = cudaGetLastError();
    }
    cudaGraph_t body = nullptr;
    if (!ec) {
        cudaStreamCaptureStatus st;
        const cudaGraphNode_t *deps = nullptr;
        size_t nd = 0;
        cudaGraph_t capg = nullptr;
        ec = cudaStreamGetCaptureInfo(c->s, &st, nullptr, &capg, &deps, nullptr, &nd);
        cudaGraphNode_t cn = nullptr;
        if (!ec) {
            // zeroed storage: the parameter struct's union has no default constructor
            alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)] = {};
            cudaGraphNodeParams &cp = *reinterpret_cast<cudaGraphNodeParams *>(raw);
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = h;
            cp.conditional.type = cudaGraphCondTypeIf;
            cp.conditional.size = 1;
            ec = cudaGraphAddNode(&cn, capg, deps, nullptr, nd, &cp);
            if (!ec) body = cp.conditional.phGraph_out[0];
        }
        if (!ec) ec = cudaStreamUpdateCaptureDependencies(c->s, &cn, nullptr, 1, cudaStreamSetCaptureDependencies);
    }
    if (!ec) ec = cudaStreamBeginCaptureToGraph(c->aux, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (!ec) {
        k3_keys<<<g, 256, 0, c->aux>>>(P, S, w);
        k3_scan<<<1, 1024, 0, c->aux>>>(P, w);
        k3_scatter<<<g, 256, 0, c->aux>>>(P, w);
        k3_order<<<nb3(nt, 8), 256, 0, c->aux>>>(P, S, c->T, w);
        k3_copy_back<<<g, 256, 0, c->aux>>>(P, S, c->T, w);
        k3_lists<<<nt, T3, SMEM3_POS, c->aux>>>(P, w);
        const cudaError_t el = cudaGetLastError();
        cudaGraph_t got = body;
        ec = cudaStreamEndCapture(c->aux, &got);
        if (!ec) ec = el;
    }
    if (!ec) {
        k3_filter<<<nt, TF3, SMEM3_POS, c->s>>>(P, S, w);
        k3_pass1<<<nt, T13, SMEM3_1, c->s>>>(P, S, w);
        k3_pass2<<<nt, T23, SMEM3_2, c->s>>>(P, S, w);
        k3_pass3<<<nt, T33, SMEM3_3, c->s>>>(P, S, w);
        ec = cudaGetLastError();
    }
    e = cudaStreamEndCapture(c->s, &gr);
    if (!ec && !e) e = cudaGraphInstantiate(&c->exec, gr, 0);
    if (gr) cudaGraphDestroy(gr);
    return ec ? ec : e;
}

// Cells a side for n particles that share a cell of the least width with m particles on average, themselves included.
// A pair kernel's block pays for its launch and for staging a cell's halo whatever the cell holds, so with cells
// of few particles (h below ~1.15 dx) a step got dearer the fewer neighbours there were.  There the cells are
// widened until they hold 50 particles, or up to 216 where that leaves 700 tiles (a tile then stages at most
// ~1,900 of the 2,199 slots).  us a step with cells of the least width / these / one thread a particle and no tiles:
// 80^3 at h = 0.5 dx 6,759 / 536 / 433, 0.6 4,152 / 474 / 501, 0.8 2,262 / 672 / 818, 1.0 1,629 / 885 / 1,214, 1.1 1,580 /
// 1,088 / 1,589; 48^3 at 0.5 993 / 123 / 131, 0.8 384 / 176 / 227, 1.0 299 / 232 / 328; 24^3 at 0.5 148 / 44 / 84, 0.9 62 / 56 /
// 146.  From m = 50 on (1.15 dx) nothing changes.  m is an average over the particles, not over the box: a
// dense patch in an empty box keeps the cells that fit it.  At most GROW3 times the least width: positions are FP32
// offsets within a tile, up to 4.7 h with the least cells and 7.8 h with these, which leaves the fields' errors against
// FP64 at 0.7 to 1.4 times (~3e-7 of the field) and r^2 of a pair good to 2.1e-6, inside the band that FP64 decides.
int cells3(int nc_fine, int64_t n, double m)
{
    if (m >= SPARSE3) return nc_fine;
    const double want = std::min(std::max((double)n / 700.0, SPARSE3), 216.0);
    const int nc = std::max(3, (int)std::lround(nc_fine / std::min(GROW3, std::cbrt(want / m))));
    return nc == 7 ? 6 : nc;   // 343 tiles: a second wave of 39 on the 304 blocks that run at once
}

// nc cells a side: the parameters that depend on it, and the cells' centres.
cudaError_t set_cells3(ann3_ctx *c, int nc)
{
    P3 &P = c->P;
    const double cell = c->prm.L / nc;
    P.nc = nc;
    P.ncell = nc * nc * nc;
    P.nblk = std::min(P.ncell, P.n);
    P.inv_cell = nc / c->prm.L;
    P.cell_f = (float)cell;
    P.cell_lo = (float)(cell - (double)P.cell_f);
    P.far = (float)(64.0 * cell);
    std::vector<double> centre((size_t)nc);
    for (int k = 0; k < nc; k++) centre[(size_t)k] = (k + 0.5) * cell;
    const cudaError_t e =
        cudaMemcpyAsync(c->centre, centre.data(), sizeof(double) * (size_t)nc, cudaMemcpyHostToDevice, c->s);
    return e ? e : cudaStreamSynchronize(c->s);
}

// Gives the box nc cells a side and captures the step anew if that is not what it has.
cudaError_t regrid3(ann3_ctx *c, int nc)
{
    if (nc == c->P.nc) return cudaSuccess;
    const int was = c->P.nc;
    cudaGraphExec_t old = c->exec;
    cudaError_t e = set_cells3(c, nc);
    if (!e) e = capture3(c);
    if (e) {   // as it was
        c->exec = old;
        set_cells3(c, was);
        return e;
    }
    return cudaGraphExecDestroy(old);
}

// Sizes the cells for the state loaded in S: counts it into cells of the least width, unless these hold SPARSE3 over
// the whole box and so, or more, over the particles.
cudaError_t fit_cells3(ann3_ctx *c)
{
    P3 fine = c->P;
    fine.nc = c->nc_fine;
    fine.inv_cell = c->nc_fine / c->prm.L;
    const size_t n = (size_t)fine.n, ncell = (size_t)fine.nc * fine.nc * fine.nc;
    if ((double)n / (double)ncell >= SPARSE3) return regrid3(c, fine.nc);
    unsigned long long crowd = 0, *sum = reinterpret_cast<unsigned long long *>(c->tmp);
    cudaError_t e = cudaMemsetAsync(sum, 0, sizeof crowd, c->s);
    if (e) return e;
    k3_keys<<<nb3(n), 256, 0, c->s>>>(fine, c->S, c->w);
    k3_crowd<<<nb3(n), 256, 0, c->s>>>(fine.n, c->w, sum);
    e = cudaGetLastError();
    if (!e) e = cudaMemcpyAsync(&crowd, sum, sizeof crowd, cudaMemcpyDeviceToHost, c->s);
    if (!e) e = cudaMemsetAsync(c->w.count, 0, sizeof(int) * ncell, c->s);   // as the re-sort leaves them
    if (!e) e = cudaStreamSynchronize(c->s);
    return e ? e : regrid3(c, cells3(c->nc_fine, fine.n, (double)crowd / (double)n));
}

int fail3(ann3_ctx *c, int code, const std::string &m)
{
    if (c) c->last_err = m;
    return code;
}

int cuda3(ann3_ctx *c, cudaError_t e, const char *where)
{
    return fail3(c, e == cudaErrorMemoryAllocation ? ANN_ERR_OOM : ANN_ERR_CUDA, std::string(where) + ": " +
                                                                                  cudaGetErrorString(e));
}

// The first cause wins: truncated neighbour lists can make alpha singular and the state non-finite.
int status_of_bits(uint32_t b)
{
    if (b & E3_NBR) return ANN_ERR_NBR_OVERFLOW;
    if (b & E3_ALPHA) return ANN_ERR_SINGULAR_ALPHA;
    if (b & E3_NONFINITE) return ANN_ERR_NONFINITE;
    return ANN_OK;
}

}  // namespace

extern "C" {

int ann3_default_params(ann3_params *p)
{
    if (!p) return ANN_ERR_INVALID_ARG;
    std::memset(p, 0, sizeof *p);
    p->n = 32 * 32 * 32;
    p->L = 1.0;
    p->h = 1.3 / 32;
    p->dt = 1e-4;
    p->rho0 = 1.0;
    p->eta = 1.0;
    p->Gamma = 0.34;
    p->lambda_ = 0.7;
    p->A = 0.0;
    p->B = 0.0;
    p->C = 1.0;
    p->K = 0.04;
    p->zeta = 0.05;
    p->gamma_eos = 7.0;
    p->beta = 1.0;
    p->c0_min = 0.0;
    p->c_shift = 1.0 / 3.0;
    p->apd = 1;
    return ANN_OK;
}

int ann3_create(const ann3_params *p, ann3_ctx **out)
{
    if (!p || !out) return ANN_ERR_INVALID_ARG;
    *out = nullptr;
    if (p->n < 1 || p->n > (1ll << 26) || !(p->L > 0.0) || !(p->h > 0.0) || !(p->dt > 0.0) || !(p->rho0 > 0.0) ||
        !(p->gamma_eos > 0.0))
        return ANN_ERR_INVALID_ARG;
    int nc = (int)std::floor(p->L / (3.0 * p->h * (1.0 + CELL3)));
    if (nc < 3 || (int64_t)nc * nc * nc > (1ll << 28)) return ANN_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDeviceCount(&dev) != cudaSuccess || dev == 0) return ANN_ERR_NOT_AVAILABLE;
    ann3_ctx *c = new (std::nothrow) ann3_ctx();
    if (!c) return ANN_ERR_OOM;
    c->prm = *p;
    P3 &P = c->P;
    c->nc_fine = nc;
    const size_t ncell = (size_t)nc * nc * nc;
    P.n = (int)p->n;
    P.L = p->L;
    std::memcpy(&P.bitsL, &p->L, sizeof P.bitsL);
    P.hL = (float)(0.5 * p->L);
    P.R2d = 9.0 * p->h * p->h;
    P.R2lo = (float)(P.R2d * (1.0 - 4e-6));   // FP32 r^2 of a pair is good to ~1e-6 relative
    P.R2hi = (float)(P.R2d * (1.0 + 4e-6));
    P.R2c = (float)(P.R2d * (1.0 + SKIN3) * (1.0 + SKIN3) * (1.0 + 1e-5));   // padded for FP32 rounding
    P.skin_max2 = (float)((0.5 * SKIN3 * 3.0 * p->h) * (0.5 * SKIN3 * 3.0 * p->h));
    P.half_dt_d = 0.5 * p->dt;
    P.inv_h = (float)(1.0 / p->h);
    const double ad = 3.0 / (359.0 * 3.14159265358979323846 * p->h * p->h * p->h);   // Eq. (18), d = 3
    P.ad = (float)ad;
    P.kw6 = (float)(-6.0 * ad);
    P.kw15 = (float)(15.0 * ad);
    P.kf5 = (float)(-5.0 * ad / p->h);
    P.kf30 = (float)(30.0 * ad / p->h);
    P.kf75 = (float)(-75.0 * ad / p->h);
    P.W0 = (float)(66.0 * ad);                                    // W(0) = a_d (3^5 - 6 2^5 + 15)
    P.dt = (float)p->dt;
    P.half_dt = (float)(0.5 * p->dt);
    P.rho0 = (float)p->rho0;
    P.nu = (float)(p->eta / p->rho0);
    P.Gamma = (float)p->Gamma;
    P.lambda = (float)p->lambda_;
    P.A = (float)p->A;
    P.B = (float)p->B;
    P.C = (float)p->C;
    P.K = (float)p->K;
    P.zeta = (float)p->zeta;
    P.gamma_eos = (float)p->gamma_eos;
    P.beta = (float)p->beta;
    P.c0_min = (float)p->c0_min;
    P.c_shift = (float)p->c_shift;
    P.apd = p->apd;
    size_t n = (size_t)p->n;
    cudaError_t e = cudaStreamCreateWithFlags(&c->s, cudaStreamNonBlocking);
    if (!e) e = cudaStreamCreateWithFlags(&c->aux, cudaStreamNonBlocking);
    if (!e) e = alloc_set(c, c->S, n);
    if (!e) e = alloc_set(c, c->T, n);
    Work3 &w = c->w;
    if (!e) e = alloc3(c, w.key, n);
    if (!e) e = alloc3(c, w.rank, n);
    if (!e) e = alloc3(c, w.perm, n);
    if (!e) e = alloc3(c, w.count, ncell);
    if (!e) e = alloc3(c, w.start, ncell + 1);
    if (!e) e = alloc3(c, w.tile, std::min(ncell, n));
    if (!e) e = alloc3(c, w.ntile, 1);
    if (!e) e = alloc3(c, w.slots_used, 1);
    if (!e) e = alloc3(c, w.slot, 27 * n);
    if (!e) e = alloc3(c, w.cand16, (size_t)NGRP * LP * n);
    if (!e) e = alloc3(c, w.cand32, (size_t)NGRP * LP * n);
    if (!e) e = alloc3(c, w.ncand, n);
    if (!e) e = alloc3(c, w.nnbr, n);
    if (!e) e = alloc3(c, w.cell_of, n);
    if (!e) e = alloc3(c, w.xi, n);
    if (!e) e = alloc3(c, w.xi_ref, n);
    if (!e) e = alloc3(c, w.xv, n);
    if (!e) e = alloc3(c, w.dq, n);
    if (!e) e = alloc3(c, w.q2, n);
    if (!e) e = alloc3(c, w.qn, n);
    if (!e) e = alloc3(c, w.qn4, n);
    if (!e) e = alloc3(c, w.b0, n);
    if (!e) e = alloc3(c, w.b1, n);
    if (!e) e = alloc3(c, w.pu, n);
    if (!e) e = alloc3(c, w.flag, 1);
    if (!e) e = alloc3(c, w.rebuilds, 1);
    if (!e) e = alloc3(c, w.sumW, n);
    if (!e) e = alloc3(c, w.k, n);
    if (!e) e = alloc3(c, w.dhat, n);
    if (!e) e = alloc3(c, w.p, n);
    if (!e) e = alloc3(c, w.gu, 9 * n);
    if (!e) e = alloc3(c, w.lap, 5 * n);
    if (!e) e = alloc3(c, w.m, 5 * n);
    if (!e) e = alloc3(c, w.umax, 1);
    if (!e) e = alloc3(c, w.err, 1);
    if (!e) e = alloc3(c, c->tmp, 9 * n);
    if (!e) e = alloc3(c, c->centre, (size_t)nc);
    w.centre = c->centre;
    if (!e) e = set_cells3(c, nc);
    if (!e) e = cudaFuncSetAttribute(k3_pass1, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM3_1);
    if (!e) e = cudaFuncSetAttribute(k3_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM3_2);
    if (!e) e = cudaFuncSetAttribute(k3_pass3, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM3_3);
    if (!e) e = cudaStreamSynchronize(c->s);
    if (!e) e = capture3(c);
    if (!e) e = cudaStreamSynchronize(c->s);
    if (e) {
        int code = e == cudaErrorMemoryAllocation ? ANN_ERR_OOM : ANN_ERR_CUDA;
        ann3_destroy(c);
        return code;
    }
    *out = c;
    return ANN_OK;
}

void ann3_destroy(ann3_ctx *c)
{
    if (!c) return;
    if (c->s) cudaStreamSynchronize(c->s);
    if (c->exec) cudaGraphExecDestroy(c->exec);
    for (void *p : c->allocs) cudaFree(p);
    if (c->s) cudaStreamDestroy(c->s);
    if (c->aux) cudaStreamDestroy(c->aux);
    delete c;
}

int ann3_set_particles(ann3_ctx *c, int64_t n, const double *x, const double *y, const double *z, const double *u,
                       const double *q, const double *rho)
{
    if (!c) return ANN_ERR_INVALID_ARG;
    if (n != c->prm.n || !x || !y || !z || !u || !q) return fail3(c, ANN_ERR_INVALID_ARG, "bad arguments");
    const double L = c->prm.L;
    for (int64_t i = 0; i < n; i++) {
        const double r[3] = {x[i], y[i], z[i]};
        for (double v : r)
            if (!(v >= 0.0 && v < L)) return fail3(c, ANN_ERR_INVALID_ARG, "position outside [0, L)");
        for (int k = 0; k < 3; k++)
            if (!std::isfinite(u[3 * i + k])) return fail3(c, ANN_ERR_INVALID_ARG, "non-finite velocity");
        for (int k = 0; k < 5; k++)
            if (!std::isfinite(q[5 * i + k])) return fail3(c, ANN_ERR_INVALID_ARG, "non-finite Q");
        if (rho && !(std::isfinite(rho[i]) && rho[i] > 0.0)) return fail3(c, ANN_ERR_INVALID_ARG, "bad density");
    }
    size_t nn = (size_t)n;
    std::vector<float4> ua(nn), qb(nn), aa(nn);
    std::vector<int> id(nn);
    for (size_t i = 0; i < nn; i++) {
        const double *ui = u + 3 * i, *qi = q + 5 * i;
        ua[i] = make_float4((float)ui[0], (float)ui[1], (float)ui[2], (float)qi[0]);
        qb[i] = make_float4((float)qi[1], (float)qi[2], (float)qi[3], (float)qi[4]);
        // a = 0 and the density's deviation, taken in FP64
        aa[i] = make_float4(0.f, 0.f, 0.f, rho ? (float)(rho[i] / c->prm.rho0 - 1.0) : 0.f);
        id[i] = (int)i;
    }
    cudaError_t e = cudaMemcpyAsync(c->S.x, x, nn * 8, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.y, y, nn * 8, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.z, z, nn * 8, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.ua, ua.data(), nn * 16, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.qb, qb.data(), nn * 16, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.aa, aa.data(), nn * 16, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemcpyAsync(c->S.id, id.data(), nn * 4, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemsetAsync(c->w.umax, 0, 4, c->s);
    if (!e) e = cudaMemsetAsync(c->w.err, 0, 4, c->s);
    const unsigned one = 1u;   // the first step re-sorts
    if (!e) e = cudaMemcpyAsync(c->w.flag, &one, 4, cudaMemcpyHostToDevice, c->s);
    if (!e) e = cudaMemsetAsync(c->w.rebuilds, 0, 4, c->s);
    if (!e) e = cudaStreamSynchronize(c->s);
    if (!e) e = fit_cells3(c);
    if (e) return cuda3(c, e, "ann3_set_particles");
    c->have = true;
    c->steps = 0;
    return ANN_OK;
}

int ann3_step(ann3_ctx *c, int64_t nsteps)
{
    Range3 range("ann3_step");
    if (!c || nsteps < 0) return ANN_ERR_INVALID_ARG;
    if (!c->have) return fail3(c, ANN_ERR_STATE, "ann3_step before ann3_set_particles");
    cudaStream_t s = c->s;
    cudaError_t e = cudaSuccess;
    for (int64_t t = 0; t < nsteps && !e; t++) e = cudaGraphLaunch(c->exec, s);
    uint32_t bits = 0;
    if (!e) e = cudaMemcpyAsync(&bits, c->w.err, 4, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) return cuda3(c, e, "ann3_step");
    c->steps += nsteps;
    int st = status_of_bits(bits);
    if (st) return fail3(c, st, "ann3_step: device error bits " + std::to_string(bits));
    return ANN_OK;
}

int ann3_get_field(ann3_ctx *c, int32_t field, double *dst)
{
    if (!c || !dst || field < 0 || field >= ANN3_FIELD_COUNT) return ANN_ERR_INVALID_ARG;
    if (!c->have) return fail3(c, ANN_ERR_STATE, "no particles");
    const int n = c->P.n;
    const Work3 &w = c->w;
    const Set3 &S = c->S;
    Planes3 pl{};
    int nc = 0;
    cudaError_t e = cudaSuccess;
    auto put = [&](const void *p, int stride, int first, int count) {   // components first .. of packed records
        for (int k = 0; k < count; k++, nc++) {
            pl.p[nc] = static_cast<const float *>(p) + first + k;
            pl.stride[nc] = stride;
        }
    };
    auto planes = [&](const float *p, int count) {
        for (int k = 0; k < count; k++) put(p + (size_t)k * n, 1, 0, 1);
    };
    switch (field) {
    case ANN3_FIELD_POS:
        k3_pos_to_id<<<nb3(n), 256, 0, c->s>>>(n, S.x, S.y, S.z, S.id, c->tmp);
        nc = -3;
        break;
    case ANN3_FIELD_NNBR:
        k3_int_to_id<<<nb3(n), 256, 0, c->s>>>(n, w.nnbr, S.id, c->tmp);
        nc = -1;
        break;
    case ANN3_FIELD_U: put(S.ua, 4, 0, 3); break;
    case ANN3_FIELD_Q: put(S.ua, 4, 3, 1); put(S.qb, 4, 0, 4); break;
    case ANN3_FIELD_RHO: put(S.aa, 4, 3, 1); break;
    case ANN3_FIELD_A: put(S.aa, 4, 0, 3); break;
    case ANN3_FIELD_SUMW: planes(w.sumW, 1); break;
    case ANN3_FIELD_GRADU: planes(w.gu, 9); break;
    case ANN3_FIELD_LAPQ: planes(w.lap, 5); break;
    case ANN3_FIELD_QRATE: planes(w.m, 5); break;
    case ANN3_FIELD_P: planes(w.p, 1); break;
    default: return ANN_ERR_INVALID_ARG;
    }
    int comps = nc < 0 ? -nc : nc;
    if (nc > 0) k3_to_id<<<nb3(n), 256, 0, c->s>>>(n, nc, pl, S.id, c->tmp);
    e = cudaGetLastError();
    if (!e) e = cudaMemcpyAsync(dst, c->tmp, sizeof(double) * (size_t)n * comps, cudaMemcpyDeviceToHost, c->s);
    if (!e) e = cudaStreamSynchronize(c->s);
    if (e) return cuda3(c, e, "ann3_get_field");
    if (field == ANN3_FIELD_RHO)
        for (int i = 0; i < n; i++) dst[i] = c->prm.rho0 * (1.0 + dst[i]);
    return ANN_OK;
}

int ann3_get_status(ann3_ctx *c, int64_t *steps, uint32_t *error_bits, int64_t *resorts)
{
    if (!c) return ANN_ERR_INVALID_ARG;
    uint32_t b = 0, r = 0;
    cudaError_t e = cudaMemcpyAsync(&b, c->w.err, 4, cudaMemcpyDeviceToHost, c->s);
    if (!e) e = cudaMemcpyAsync(&r, c->w.rebuilds, 4, cudaMemcpyDeviceToHost, c->s);
    if (!e) e = cudaStreamSynchronize(c->s);
    if (e) return cuda3(c, e, "ann3_get_status");
    if (steps) *steps = c->steps;
    if (error_bits) *error_bits = b;
    if (resorts) *resorts = r;
    return ANN_OK;
}

const char *ann3_last_error(ann3_ctx *c) { return c ? c->last_err.c_str() : ""; }

}  // extern "C"
