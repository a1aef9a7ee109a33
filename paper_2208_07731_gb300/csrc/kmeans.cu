// Step 2: weighted Lloyd K-means on the real-space grid (Sec. 2.2,
// Eq. opt second form, Eq. r_k, Algorithm 1).
//
// Design (one CTA of 8 warps per 8 x 8 x 8 tile of the grid; each warp owns a
// 4 x 4 x 4 sub-cube, two points per lane):
//  * exact two-level pruning: the CTA bounds every centroid's squared
//    distance to its tile from below (LB) and above (UB) in FP32 with error
//    margins and keeps those with LB <= min UB (only they can be the nearest
//    centroid of a point in the tile); each warp prunes that list again
//    against its own sub-cube. The centroids that can pass the tile's test
//    while none of them has moved by more than some Delta are listed per tile
//    in memory (tens of n_mu), and later passes scan that list until the
//    largest moves since then add up to Delta; the test on what is listed is
//    the same, so the candidates are the same as from a scan of all centroids.
//    Tiles with more candidates than shared memory holds are left to a kernel
//    of their own (km_crowded);
//  * FP32 screen: each point evaluates its warp's candidates in FP32 in
//    tile-local coordinates and keeps the two smallest values; when their gap
//    exceeds a rigorous bound E on |d_fp32 - d_exact| (+ FP64 rounding) the
//    FP32 winner is the FP64 winner. Otherwise the point re-evaluates the close
//    candidates with the FP64 formula ((dx*dx + dy*dy) + dz*dz) and takes the
//    smallest (distance, mu) pair - exactly the brute-force FP64 decision. The
//    bound and the gap test are evaluated in FP32 with upward margins (a test
//    that errs sends a point to the FP64 path, never past it), and the grid
//    coordinates RN(i h) of a tile come from a per-CTA table: GB300 issues
//    FP64 at about 2 operations per clock per SM, so the pass keeps FP64 for
//    the decisions and the products w*x of the exact sums;
//  * exact update: each FP64 product w*x enters as the 128-bit integer
//    floor(w*x*2^s); sums are integer (associative, so the result does not
//    depend on thread or block order). They are kept from pass to pass: a point
//    that changes its cluster moves its four integers from the old sums to the
//    new ones, and a point that keeps it (nearly all, after a few passes) costs
//    neither FP64 products nor a reduction. The moves of a warp are added per
//    cluster by warp reductions over 26-bit limbs and once to memory; the update
//    kernel rounds each sum to FP64 and divides once.
// Measured against scanning all centroids and summing every point in every pass: 100 updates at 128^3, n_mu = 4096,
// 31.0 -> 14.2 ms, and 9.2 ms with four CTAs a SM (64 registers, four candidates in flight), fused FP64 terms of the
// objective, reductions by one instruction and the objective's partials summed by 256 threads (31 -> 7 us an
// update), and chained launches (9.6 -> 9.2).
// A late pass takes 75 us, 38 of them FP64 issue of the objective; one that writes new lists 115.
#include "common.cuh"

namespace {

constexpr int TX = 8, TY = 8, TZ = 8;    // CTA tile (smaller tiles repeat the per-tile centroid scan)
constexpr int kThreads = 256;            // 8 warps x (4 x 4 x 4 sub-cube, 2 points per lane)
constexpr int kWarpCap = 256;            // per-warp candidate list capacity (else the CTA list is used)
constexpr int kCand = 1024;              // tile candidates held in shared memory (more: km_crowded)
constexpr int kMaxMu = 8192;
constexpr double kCrowd = -1.0;          // mark of a tile with more than kCand candidates

struct KmCtl {
    unsigned long long wmax_bits;
    unsigned long long ties;
    unsigned long long refined;
    unsigned int moved[2];     // update t sets moved[t & 1] when any centroid changed
    int error;
    int converged;
    int n_iter;
    int pad;
    float left[2];             // pass t: moves that the tile lists still cover after update t - 1 (slot t & 1)
    unsigned int disp[2];      // update t: largest move of a centroid, rounded up (float bits, slot t & 1)
    unsigned int crowds[2];    // pass t: tiles left to km_crowded (slot t & 1)
};

struct KmArgs {
    const double *w;
    int nx, ny, nz;
    double hx, hy, hz;
    double tie_floor;     // hmin^2
    int n_mu;
    int s_base;           // 126 - bits(N_r) - e(max(L, 1))
    int ntx, nty, ntz;    // tiles per axis
    double *cent;         // n_mu x 3
    float4 *c32;          // n_mu: FP32 copies of the centroids for the conservative tile scan
    float scan_err;       // bound on the FP32 error of a tile-local centroid coordinate in the scan
    float h32[3], lmax32, tie_floor32;   // hx, hy, hz, max(Lx, Ly, Lz, 1), hmin^2 in FP32
    int want_obj;         // objective requested: FP64 distance of every winner
    unsigned long long *acc;  // n_mu x 8: (w, wx, wy, wz) x (lo, hi)
    int32_t *labels;
    double *dist;         // final pass: distances; before it, the tiles' lists (dist and the lists never live together)
    int list_cap;         // entries of a tile's list after its count
    float h_ref;          // mean grid spacing, the unit of the lists' Delta
    double *jpart;        // the tiles' parts of the objective; kCrowd: the tile is left to km_crowded
    unsigned long long *best;
    unsigned long long *idx_u;
    KmCtl *ctl;
    int early_stop;
};

struct U128 {
    unsigned long long lo, hi;
};

// floor(v * 2^s) for finite v >= 0 and 0 <= s, as an exact 128-bit integer
__device__ __forceinline__ U128 fixed_of(double v, int s)
{
    U128 r{0ull, 0ull};
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);   // +-0 gives m = 0 below
    const int e = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    int sh;
    if (e == 0) {
        sh = s - 1074;
    } else {
        m |= 1ull << 52;
        sh = e - 1075 + s;
    }
    if (sh >= 0) {
        if (sh == 0) {
            r.lo = m;
        } else if (sh < 64) {
            r.lo = m << sh;
            r.hi = m >> (64 - sh);
        } else if (sh < 128) {
            r.hi = m << (sh - 64);
        }
    } else if (sh > -64) {
        r.lo = m >> (-sh);
    }
    return r;
}

__device__ __forceinline__ void atomic_add_u128(unsigned long long *p, U128 v)
{
    if ((v.lo | v.hi) == 0ull) return;
    const unsigned long long old = atomicAdd(p, v.lo);
    const unsigned long long h = v.hi + ((old + v.lo < old) ? 1ull : 0ull);
    if (h) atomicAdd(p + 1, h);
}

// round-to-nearest-even conversion of an unsigned 128-bit integer
__device__ __forceinline__ double u128_to_double(unsigned long long lo, unsigned long long hi)
{
    if (hi == 0ull) return __ull2double_rn(lo);
    const int n = __clzll((long long)hi);
    unsigned long long top = n ? ((hi << n) | (lo >> (64 - n))) : hi;
    const unsigned long long rest = lo << n;
    if (rest) top |= 1ull;
    return ldexp(__ull2double_rn(top), 64 - n);
}

__device__ __forceinline__ double dist2_fp64(double x, double y, double z, double cx, double cy, double cz)
{
    const double dx = __dsub_rn(x, cx), dy = __dsub_rn(y, cy), dz = __dsub_rn(z, cz);
    double d = __dmul_rn(dx, dx);
    d = __dadd_rn(d, __dmul_rn(dy, dy));
    d = __dadd_rn(d, __dmul_rn(dz, dz));
    return d;
}

__device__ __forceinline__ int fixed_scale(const KmArgs &a)
{
    const double wmax = __longlong_as_double((long long)a.ctl->wmax_bits);
    int e = 0;
    if (wmax > 0.0) frexp(wmax, &e);
    return a.s_base - e;
}

// deterministic block sum (fixed shuffle pattern, fixed warp order)
__device__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s = __dadd_rn(s, red[i]);
    return s;  // valid in thread 0
}

__global__ void km_init(KmArgs a, const int64_t *__restrict__ init_idx, int64_t n_r)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        a.ctl->wmax_bits = 0ull;
        a.ctl->ties = 0ull;
        a.ctl->refined = 0ull;
        a.ctl->moved[0] = 0u;
        a.ctl->moved[1] = 0u;
        a.ctl->error = 0;
        a.ctl->converged = 0;
        a.ctl->n_iter = 0;
        a.ctl->left[0] = a.ctl->left[1] = 0.f;
        a.ctl->disp[0] = a.ctl->disp[1] = 0u;
        a.ctl->crowds[0] = a.ctl->crowds[1] = 0u;
    }
    if (i < a.n_mu) {
        int64_t r = init_idx[i];
        if (r < 0 || r >= n_r) {
            atomicExch(&a.ctl->error, 2);
            r = 0;
        }
        const int64_t ix = r / ((int64_t)a.ny * a.nz), iy = (r / a.nz) % a.ny, iz = r % a.nz;
        a.cent[3 * i + 0] = __dmul_rn((double)ix, a.hx);
        a.cent[3 * i + 1] = __dmul_rn((double)iy, a.hy);
        a.cent[3 * i + 2] = __dmul_rn((double)iz, a.hz);
        a.c32[i] = make_float4((float)a.cent[3 * i], (float)a.cent[3 * i + 1], (float)a.cent[3 * i + 2], 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) a.acc[8 * i + k] = 0ull;
        a.best[i] = ~0ull;
        a.idx_u[i] = ~0ull;
    }
    for (int64_t b = i; b < (int64_t)a.ntx * a.nty * a.ntz; b += (int64_t)gridDim.x * blockDim.x) a.jpart[b] = 0.0;
    for (int64_t r = i; r < n_r; r += (int64_t)gridDim.x * blockDim.x) a.labels[r] = -1;
}

__global__ void km_wmax(KmArgs a, int64_t n_r)
{
    unsigned long long m = 0ull;
    int bad = 0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_r; r += (int64_t)gridDim.x * blockDim.x) {
        const double v = a.w[r];
        if (!(v >= 0.0) || isinf(v)) bad = 1;
        else if (v > 0.0) m = max(m, (unsigned long long)__double_as_longlong(v));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = max(m, __shfl_down_sync(0xffffffffu, m, o));
        bad |= __shfl_down_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (m) atomicMax(&a.ctl->wmax_bits, m);
        if (bad) atomicExch(&a.ctl->error, 1);
    }
}

__global__ void km_check_scale(KmArgs a)
{
    if (threadIdx.x == 0 && fixed_scale(a) < 0) atomicExch(&a.ctl->error, 1);
}

__device__ __forceinline__ U128 add_u128(U128 a, U128 b)
{
    U128 r;
    r.lo = a.lo + b.lo;
    r.hi = a.hi + b.hi + (r.lo < a.lo ? 1ull : 0ull);
    return r;
}

__device__ __forceinline__ U128 sub_u128(U128 a, U128 b)
{
    U128 r;
    r.lo = a.lo - b.lo;
    r.hi = a.hi - b.hi - (a.lo < b.lo ? 1ull : 0ull);
    return r;
}

// min / max over the warp of non-negative floats (their bits order like integers): one warp reduction each
__device__ __forceinline__ float warp_min_pos(float v)
{
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

__device__ __forceinline__ float warp_max_pos(float v)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// the sum of v over the warp (mod 2^128), valid in every lane: five 26-bit limbs, each summed by one warp reduction
__device__ __forceinline__ U128 warp_sum_u128(U128 v)
{
    constexpr unsigned int m = (1u << 26) - 1u;
    const unsigned long long l0 = __reduce_add_sync(0xffffffffu, (unsigned int)v.lo & m);
    const unsigned long long l1 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.lo >> 26) & m);
    const unsigned long long l2 = __reduce_add_sync(0xffffffffu, (unsigned int)((v.lo >> 52) | (v.hi << 12)) & m);
    const unsigned long long l3 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.hi >> 14) & m);
    const unsigned long long l4 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.hi >> 40) & m);   // 24 bits
    U128 r = add_u128(U128{l0, 0ull}, U128{l1 << 26, l1 >> 38});
    r = add_u128(r, U128{l2 << 52, l2 >> 12});
    r.hi += (l3 << 14) + (l4 << 40);
    return r;
}

// Move the integers (w, wx, wy, wz) of this lane's points h = 0, 1 with from[h] != to[h] from the sums of cluster
// from[h] (-1: none yet) to those of to[h]: one distinct cluster of the warp at a time, added once (lane q adds sum q).
__device__ __forceinline__ void warp_move(const int (&from)[2], const int (&to)[2], const U128 (&v)[2][4],
                                          unsigned long long *acc, int lane)
{
    // pending entries of this lane: bit 2 h is the arrival of point h, bit 2 h + 1 its departure
    unsigned pend = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (from[h] != to[h]) pend |= (1u << (2 * h)) | (from[h] >= 0 ? 2u << (2 * h) : 0u);
    for (;;) {
        const unsigned lanes = __ballot_sync(0xffffffffu, pend != 0u);
        if (!lanes) return;
        const int mine = (pend & 1u) ? to[0] : (pend & 2u) ? from[0] : (pend & 4u) ? to[1] : from[1];
        const int k = __shfl_sync(0xffffffffu, mine, __ffs(lanes) - 1);
        U128 s[4] = {{0ull, 0ull}, {0ull, 0ull}, {0ull, 0ull}, {0ull, 0ull}};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if ((pend >> (2 * h) & 1u) && to[h] == k) {
                pend &= ~(1u << (2 * h));
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = add_u128(s[q], v[h][q]);
            }
            if ((pend >> (2 * h) & 2u) && from[h] == k) {
                pend &= ~(2u << (2 * h));
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = sub_u128(s[q], v[h][q]);
            }
        }
        U128 mysum{0ull, 0ull};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const U128 r = warp_sum_u128(s[q]);
            if (lane == q) mysum = r;
        }
        if (lane < 4) atomic_add_u128(acc + 8 * (int64_t)k + 2 * lane, mysum);
    }
}

// Bound on |d_fp32 - d_exact| (+ FP64 rounding) of a warp: the point coordinates
// (integer offset x FP32 spacing) carry <= 2.01 u32 |p|, the candidates <= 1.0001 u32 |q|,
// their difference one more rounding, then three FP32 products and two FP32 additions
// It is evaluated in FP32: every quantity is positive, so each operation adds at most a relative
// 2^-24 (a fused multiply-add one rounding); the factor 1 + 2^-16 covers the dozen roundings, and the
// formula's 1 % slack the rounding of its decimal constants and of L. Pm, Qm: the largest coordinates of the tile's
// points and of the candidates.
constexpr float kUp = 1.f + 1.52587890625e-5f;   // 1 + 2^-16
__device__ __forceinline__ float screen_error(float Pm, float Qm, float L)
{
    constexpr float u32 = 5.9604644775390625e-8f;   // 2^-24
    const float Tm = (Pm + Qm) * (1.f + 4.f * u32);
    const float del = 1.01f * u32 * (2.01f * Pm + 1.0001f * Qm + (Pm + Qm)) + 8e-16f * L;
    return 1.01f * (3.f * del * (2.f * Tm + del) + 9.001f * u32 * Tm * Tm + 1.6e-15f * 3.f * Tm * Tm) * kUp;
}

// The FP32 winner is the FP64 winner when the runner-up is further than the gap; the test is
// conservative in FP32 (gap rounded up by 1 + 2^-16, the difference scaled down by 1 - 2^-22)
__device__ __forceinline__ float screen_gap(float d1, float E, float floor32)
{
    return (2.f * E + 2.0e-12f * fmaxf(d1 + E, floor32) + 1.0e-14f * (d1 + E)) * kUp;
}
__device__ __forceinline__ bool screen_clear(float d1, float d2, float gap)
{
    return (d2 - d1) * (1.f - 2.384185791015625e-7f) > gap;
}

// The cut of a warp's candidates from the smallest of their largest squared distances: tile-local coordinates are
// accurate to ~1e-7 relative; the margin covers them and the float sums
__device__ __forceinline__ float warp_cut(float wub, float Tmx)
{
    return wub * 1.0001f + 4e-6f * (Tmx * Tmx + wub) + 1e-30f;
}

// FP64 decision among the candidates that can still win: the smallest (distance, centroid) pair, the runner-up's
// distance
struct Decision {
    double b1, b2;
    int mu;
    __device__ __forceinline__ void see(double e, int m)
    {
        if (e < b1 || (e == b1 && m < mu)) {
            b2 = b1;
            b1 = e;
            mu = m;
        } else if (e < b2) {
            b2 = e;
        }
    }
};

// The largest and the smallest squared distance of q to a box in tile-local FP32 coordinates
__device__ __forceinline__ float box_upper(float qx, float qy, float qz, float x0, float y0, float z0, float x1, float y1,
                                           float z1)
{
    const float ux = fmaxf(fabsf(qx - x0), fabsf(x1 - qx));
    const float uy = fmaxf(fabsf(qy - y0), fabsf(y1 - qy));
    const float uz = fmaxf(fabsf(qz - z0), fabsf(z1 - qz));
    return ux * ux + uy * uy + uz * uz;
}
__device__ __forceinline__ float box_lower(float qx, float qy, float qz, float x0, float y0, float z0, float x1, float y1,
                                           float z1)
{
    const float lx = fmaxf(0.f, fmaxf(x0 - qx, qx - x1));
    const float ly = fmaxf(0.f, fmaxf(y0 - qy, qy - y1));
    const float lz = fmaxf(0.f, fmaxf(z0 - qz, qz - z1));
    return lx * lx + ly * ly + lz * lz;
}
// the smallest squared distance of a centroid q from the origin of a tile of extents P to the tile
__device__ __forceinline__ float tile_lower(float qx, float qy, float qz, float Px, float Py, float Pz)
{
    const float lx = fmaxf(0.f, fmaxf(-qx, qx - Px));
    const float ly = fmaxf(0.f, fmaxf(-qy, qy - Py));
    const float lz = fmaxf(0.f, fmaxf(-qz, qz - Pz));
    return lx * lx + ly * ly + lz * lz;
}
// keep every centroid whose smallest squared distance to the tile can reach min UB: each
// coordinate carries an error <= dq, so LB and UB move by <= dq (2 sqrt(3) sqrt(.) + 3 dq)
__device__ __forceinline__ bool tile_reaches(float lb, float minub, float sminub, float dq)
{
    const float margin = dq * (3.5f * (sqrtf(lb) + sminub) + 6.f * dq) + 1e-6f * (lb + minub) + 1e-30f;
    return lb <= minub + margin;
}

// Shared memory of a CTA: separate arrays (in one struct the compiler cannot tell their accesses apart: a pass took 7 %
// longer) and a view of them
template <int NW>
struct TileShared {
    float4 *cand;             // kCand + 1 (qx, qy, qz, mu bits), tile-local FP32 coordinates; the last one is at infinity
    unsigned short (*wlist)[kWarpCap + 4];
    unsigned int *counts;     // candidates, listed centroids
    float *minub;
    double *jterm;            // 32 NW
    // grid coordinates of the tile (xs[i] = RN((ix0 + i) hx), ...) and its FP32 extents, formed once per CTA:
    // the FP64 pipe (about 2 operations per clock per SM) is the scarce unit of this kernel
    double *xs, *ys, *zs;
    float *hdr32;             // hx, hy, hz, Px, Py, Pz (tile extents), ox, oy, oz (origin), L, hmin^2 in FP32
};
#define TILE_SHARED(sh)                                                                                  \
    __shared__ float4 cand_[kCand + 1];                                                                  \
    __shared__ __align__(8) unsigned short wlist_[NW][kWarpCap + 4];                                     \
    __shared__ unsigned int counts_[2];                                                                  \
    __shared__ float minub_[NW], hdr32_[11];                                                             \
    __shared__ double jterm_[32 * NW], xs_[NW == 8 ? TX : TX / 2], ys_[TY], zs_[TZ];                     \
    const TileShared<NW> sh{cand_, wlist_, counts_, minub_, jterm_, xs_, ys_, zs_, hdr32_}

// Tables of tile b, by threads 0 .. 32 of the CTA (a barrier follows)
template <int NW>
__device__ __forceinline__ void tile_tables(const KmArgs &a, TileShared<NW> sh, int b)
{
    constexpr int TXE = NW == 8 ? TX : TX / 2;
    const int tid = threadIdx.x, tz = b % a.ntz, ty = (b / a.ntz) % a.nty, tx = b / (a.ntz * a.nty);
    const int ix0 = tx * TXE, iy0 = ty * TY, iz0 = tz * TZ;
    if (tid < TXE) sh.xs[tid] = __dmul_rn((double)(ix0 + tid), a.hx);
    else if (tid < TXE + TY) sh.ys[tid - TXE] = __dmul_rn((double)(iy0 + tid - TXE), a.hy);
    else if (tid < TXE + TY + TZ) sh.zs[tid - TXE - TY] = __dmul_rn((double)(iz0 + tid - TXE - TY), a.hz);
    else if (tid == 32) {
        sh.hdr32[0] = a.h32[0];
        sh.hdr32[1] = a.h32[1];
        sh.hdr32[2] = a.h32[2];
        sh.hdr32[3] = (float)((min(TXE, a.nx - ix0) - 1) * a.hx);
        sh.hdr32[4] = (float)((min(TY, a.ny - iy0) - 1) * a.hy);
        sh.hdr32[5] = (float)((min(TZ, a.nz - iz0) - 1) * a.hz);
        sh.hdr32[6] = (float)__dmul_rn((double)ix0, a.hx);   // = (float)xs[0], ...
        sh.hdr32[7] = (float)__dmul_rn((double)iy0, a.hy);
        sh.hdr32[8] = (float)__dmul_rn((double)iz0, a.hz);
        sh.hdr32[9] = a.lmax32;
        sh.hdr32[10] = a.tie_floor32;
        sh.counts[0] = 0u;
        sh.counts[1] = 0u;
        sh.cand[kCand] = make_float4(INFINITY, 0.f, 0.f, 0.f);
    }
}

// The smallest of the scanned centroids' largest squared distances to the tile (FP32), in every thread: min UB
template <int NW>
__device__ __forceinline__ float tile_min_upper(const KmArgs &a, TileShared<NW> sh, const unsigned short *list, int n_scan)
{
    const float Px = sh.hdr32[3], Py = sh.hdr32[4], Pz = sh.hdr32[5], ox = sh.hdr32[6], oy = sh.hdr32[7], oz = sh.hdr32[8];
    float mub = INFINITY;
    for (int i = threadIdx.x; i < n_scan; i += 32 * NW) {
        const float4 c = a.c32[list ? (int)list[i] : i];
        const float qx = c.x - ox, qy = c.y - oy, qz = c.z - oz;
        const float ux = fmaxf(fabsf(qx), fabsf(Px - qx));
        const float uy = fmaxf(fabsf(qy), fabsf(Py - qy));
        const float uz = fmaxf(fabsf(qz), fabsf(Pz - qz));
        mub = fminf(mub, ux * ux + uy * uy + uz * uz);
    }
    mub = warp_min_pos(mub);
    if ((threadIdx.x & 31) == 0) sh.minub[threadIdx.x >> 5] = mub;
    __syncthreads();
    float minub = sh.minub[0];
    for (int i = 1; i < NW; ++i) minub = fminf(minub, sh.minub[i]);
    return minub;
}

// accurate tile-local coordinates of a kept centroid (one FP64 subtraction each)
template <int NW>
__device__ __forceinline__ float4 tile_local(const KmArgs &a, TileShared<NW> sh, int m)
{
    return make_float4((float)__dsub_rn(a.cent[3 * m + 0], sh.xs[0]), (float)__dsub_rn(a.cent[3 * m + 1], sh.ys[0]),
                       (float)__dsub_rn(a.cent[3 * m + 2], sh.zs[0]), __int_as_float(m));
}

// The two points of a lane: (bx + lx2 + 2 h, by + ly, bz + lz) of the tile for h = 0, 1
struct Points {
    int x, y, z;          // of point 0
    int64_t r0, step;     // grid index of point 0, from point 0 to point 1
    bool valid[2];
    int from[2], to[2];   // clusters
    double wr[2];
    double jv;            // objective of both
    unsigned ties, refined;
};

template <bool FINAL, int NW>
__device__ __forceinline__ Points tile_points(const KmArgs &a, int b, int warp, int lane)
{
    constexpr int TXE = NW == 8 ? TX : TX / 2;
    const int tz = b % a.ntz, ty = (b / a.ntz) % a.nty, tx = b / (a.ntz * a.nty);
    Points p;
    p.x = 4 * ((warp >> 2) & 1) + (lane >> 4);
    p.y = 4 * ((warp >> 1) & 1) + ((lane >> 2) & 3);
    p.z = 4 * (warp & 1) + (lane & 3);
    const int ix = tx * TXE + p.x, iy = ty * TY + p.y, iz = tz * TZ + p.z;
    p.r0 = ((int64_t)ix * a.ny + iy) * a.nz + iz;
    p.step = (int64_t)2 * a.ny * a.nz;
    p.jv = 0.0;
    p.ties = p.refined = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        p.valid[h] = ix + 2 * h < a.nx && iy < a.ny && iz < a.nz;
        p.from[h] = p.to[h] = -1;
        p.wr[h] = 0.0;
        if (p.valid[h]) {   // loaded ahead of the scan that hides their latency
            p.wr[h] = a.w[p.r0 + h * p.step];
            if (!FINAL) p.from[h] = a.labels[p.r0 + h * p.step];
        }
    }
    return p;
}

// The outcome for point h: `clear` if the screen has settled that mu is its centroid, else the FP64 decision `best`
template <bool FINAL, int NW>
__device__ __forceinline__ void settle_point(const KmArgs &a, TileShared<NW> sh, Points &p, int h, bool clear, int mu,
                                             const Decision &best)
{
    const double x = sh.xs[p.x + 2 * h], y = sh.ys[p.y], z = sh.zs[p.z];   // RN(ix hx), ...
    int win_mu = mu;
    double win_d = 0.0;
    if (clear) {
        if (FINAL) {
            win_d = dist2_fp64(x, y, z, a.cent[3 * win_mu], a.cent[3 * win_mu + 1], a.cent[3 * win_mu + 2]);
        } else if (a.want_obj) {   // for the objective only: fused, one rounding and one FP64 issue less per term
            const double dx = x - a.cent[3 * win_mu], dy = y - a.cent[3 * win_mu + 1], dz = z - a.cent[3 * win_mu + 2];
            win_d = fma(dz, dz, fma(dy, dy, dx * dx));
        }
    } else {
        p.refined += 1;
        win_mu = best.mu;
        win_d = best.b1;
        if (a.n_mu > 1 && __dsub_rn(best.b2, best.b1) <= 1e-12 * fmax(best.b1, a.tie_floor)) p.ties += 1;
    }
    if (FINAL || a.want_obj) p.jv = fma(p.wr[h], win_d, p.jv);
    p.to[h] = win_mu;
    const int64_t r = p.r0 + h * p.step;
    if (FINAL) {
        a.labels[r] = win_mu;
        a.dist[r] = win_d;
        atomicMin(&a.best[win_mu], (unsigned long long)__double_as_longlong(win_d));
    } else if (p.from[h] != win_mu) {
        a.labels[r] = win_mu;
    }
}

// Sums of the clusters that points left and joined, counts and the tile's part of the objective. By all threads
template <bool FINAL, int NW>
__device__ __forceinline__ void settle_tile(const KmArgs &a, TileShared<NW> sh, const Points &p, int b)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (!FINAL && __any_sync(0xffffffffu, p.from[0] != p.to[0] || p.from[1] != p.to[1])) {
        const int s_fix = fixed_scale(a);
        U128 v[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int q = 0; q < 4; ++q) v[h][q] = U128{0ull, 0ull};
            if (p.from[h] != p.to[h]) {
                v[h][0] = fixed_of(p.wr[h], s_fix);
                v[h][1] = fixed_of(__dmul_rn(p.wr[h], sh.xs[p.x + 2 * h]), s_fix);
                v[h][2] = fixed_of(__dmul_rn(p.wr[h], sh.ys[p.y]), s_fix);
                v[h][3] = fixed_of(__dmul_rn(p.wr[h], sh.zs[p.z]), s_fix);
            }
        }
        warp_move(p.from, p.to, v, a.acc, lane);
    }
    // the objective partial (fixed order: deterministic) and the two counts, reduced together with one barrier. One
    // warp sums the CTA's terms: NW - 1 + 5 FP64 instructions instead of 5 in each of NW warps.
    const bool want_j = FINAL || a.want_obj;
    if (want_j) sh.jterm[tid] = p.jv;
    const unsigned ties = __reduce_add_sync(0xffffffffu, p.ties), refined = __reduce_add_sync(0xffffffffu, p.refined);
    if (lane == 0) {
        if (ties) atomicAdd(&a.ctl->ties, (unsigned long long)ties);
        if (refined) atomicAdd(&a.ctl->refined, (unsigned long long)refined);
    }
    grid_release();
    if (!want_j) return;
    __syncthreads();
    if (warp == 0) {
        double s = sh.jterm[lane];
#pragma unroll
        for (int i = 1; i < NW; ++i) s = __dadd_rn(s, sh.jterm[32 * i + lane]);
        for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_down_sync(0xffffffffu, s, o));
        if (lane == 0) a.jpart[b] = s;
    }
}

// NW = 8: an 8 x 8 x 8 tile per CTA (warps = its eight 4 x 4 x 4 sub-cubes); NW = 4: a 4 x 8 x 8 half
// tile (the four sub-cubes of one x half), which doubles the CTAs on grids with few tiles per SM
template <bool FINAL, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? 4 : 8) km_assign(KmArgs a, int t)
{
    constexpr int NT = 32 * NW, TXE = NW == 8 ? TX : TX / 2;
    grid_wait();
    if (a.ctl->error) return;
    if (!FINAL && a.ctl->converged) return;
    if (!FINAL && a.early_stop && t >= 2 && a.ctl->moved[(t - 1) & 1] == 0u) {
        // update t-1 left every centroid bit-identical, so this and every later pass would
        // repeat the labels and sums of pass t-1: the loop has converged. The labels first
        // repeated at pass t-1 (labels repeat, so the sums and then the centroids repeat one
        // update later), which is the count reported; objective entries and near-tie counts
        // of passes 0 .. t-1 are complete. (Points of zero weight can change cluster without
        // moving a centroid; then the count is one below the first pass whose labels repeat.)
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.ctl->n_iter = t - 1;
            a.ctl->converged = 1;
        }
        return;
    }
    // Do the tiles' lists still hold every possible candidate? Pass t reads what pass t-1 left (slot (t-1) & 1) and
    // the largest move of update t-1, and writes the other slots.
    bool full = true;
    float cover = 0.f;   // Delta of the lists written by this pass, or what is left of the present ones
    if (!FINAL && t > 0) {
        const float move = __uint_as_float(a.ctl->disp[(t - 1) & 1]);
        cover = __fsub_rd(a.ctl->left[(t - 1) & 1], move);
        full = !(cover >= 0.f);
        // a Delta of twelve of the last moves lasts for many passes (moves shrink); 2 h keeps the lists short
        if (full) cover = fminf(fmaxf(12.f * move, 0.5f * a.h_ref), 2.f * a.h_ref);
    }
    if (!FINAL && blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->left[t & 1] = cover;
        a.ctl->disp[t & 1] = 0u;
        a.ctl->crowds[(t + 1) & 1] = 0u;
    }

    TILE_SHARED(sh);
    float4 *const cand = sh.cand;
    double *const xs = sh.xs, *const ys = sh.ys, *const zs = sh.zs;
    float *const hdr32 = sh.hdr32;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const int tz = b % a.ntz, ty = (b / a.ntz) % a.nty, tx = b / (a.ntz * a.nty);
    const int ix0 = tx * TXE, iy0 = ty * TY, iz0 = tz * TZ;
    const int ex = min(TXE, a.nx - ix0), ey = min(TY, a.ny - iy0), ez = min(TZ, a.nz - iz0);
    tile_tables(a, sh, b);
    unsigned short *list = reinterpret_cast<unsigned short *>(a.dist) + (int64_t)b * (a.list_cap + 1);
    int n_scan = a.n_mu;   // centroids to scan: all of them, or the tile's list
    if (!full) {
        const int n = list[0];
        if (n <= a.list_cap) n_scan = n;
        else full = true;   // the list did not fit
    }
    const bool write_list = !FINAL && full && n_scan == a.n_mu && a.list_cap > 0;
    __syncthreads();
    const float hx = hdr32[0], hy = hdr32[1], hz = hdr32[2];
    const float Px = hdr32[3], Py = hdr32[4], Pz = hdr32[5];

    // ---- tile scan (FP32, conservative): min over centroids of the largest squared distance to the tile
    const float ox32 = hdr32[6], oy32 = hdr32[7], oz32 = hdr32[8];
    const float dq = a.scan_err;
    const float minub = tile_min_upper(a, sh, full ? nullptr : list + 1, n_scan);
    const float sminub = sqrtf(minub);
    // The list for later passes: once every centroid has moved by at most Delta, sqrt(LB) has shrunk and sqrt(min UB)
    // grown by at most Delta each, so who may pass the test above then has sqrt(LB) <= sqrt(min UB) + 2 Delta now, but
    // for the margin: a > b (1 + 1e-4) + 16 dq gives a^2 - b^2 > margin for a = sqrt(LB), b = sqrt(min UB).
    const float reach = (sminub + 2.f * cover) * 1.0001f + 16.f * dq;
    for (int i = tid; i < n_scan; i += NT) {
        const int m = full ? i : (int)list[1 + i];
        const float4 c = a.c32[m];
        const float lb = tile_lower(c.x - ox32, c.y - oy32, c.z - oz32, Px, Py, Pz);
        if (tile_reaches(lb, minub, sminub, dq)) {
            const unsigned j = atomicAdd(&sh.counts[0], 1u);
            if (j < kCand) cand[j] = tile_local(a, sh, m);
        }
        if (write_list && sqrtf(lb) <= reach) {
            const unsigned j = atomicAdd(&sh.counts[1], 1u);
            if (j < (unsigned)a.list_cap) list[1 + j] = (unsigned short)m;
        }
    }
    __syncthreads();
    if (write_list && tid == 0) list[0] = (unsigned short)min(sh.counts[1], (unsigned)a.list_cap + 1u);
    const int nc = (int)sh.counts[0];
    if (nc > kCand) {   // km_crowded's
        if (tid == 0) {
            a.jpart[b] = kCrowd;
            atomicAdd(&a.ctl->crowds[t & 1], 1u);
        }
        return;
    }

    // ---- this warp's 4 x 4 x 4 sub-cube and its candidate list
    const int sx = (warp >> 2) & 1, sy = (warp >> 1) & 1, sz = warp & 1;
    const int bx = 4 * sx, by = 4 * sy, bz = 4 * sz;
    const int wex = min(4, ex - bx), wey = min(4, ey - by), wez = min(4, ez - bz);
    const float Sx0 = bx * hx, Sy0 = by * hy, Sz0 = bz * hz;
    const float Sx1 = Sx0 + (wex - 1) * hx, Sy1 = Sy0 + (wey - 1) * hy, Sz1 = Sz0 + (wez - 1) * hz;
    unsigned short *const wlist = sh.wlist[warp];
    float wub = INFINITY;
    for (int j = lane; j < nc; j += 32) {
        const float4 q = cand[j];
        wub = fminf(wub, box_upper(q.x, q.y, q.z, Sx0, Sy0, Sz0, Sx1, Sy1, Sz1));
    }
    const float Tmx = fmaxf(Px, fmaxf(Py, Pz)), wcut = warp_cut(warp_min_pos(wub), Tmx);
    int wn = 0;
    float wq = 0.f;
    for (int base = 0; base < nc; base += 32) {
        const int j = base + lane;
        bool keep = false;
        if (j < nc) {
            const float4 q = cand[j];
            keep = box_lower(q.x, q.y, q.z, Sx0, Sy0, Sz0, Sx1, Sy1, Sz1) * 0.9999f <= wcut;
            if (keep) wq = fmaxf(wq, fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z))));
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        const int pos = wn + __popc(bal & ((1u << lane) - 1u));
        if (keep && pos < kWarpCap) wlist[pos] = (unsigned short)j;
        wn += __popc(bal);
    }
    const bool use_w = wn <= kWarpCap;          // overflow: scan the whole tile list instead
    const int cnt = use_w ? wn : nc;
    if (!use_w) {
        wq = 0.f;
        for (int j = lane; j < nc; j += 32) {
            const float4 q = cand[j];
            wq = fmaxf(wq, fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z))));
        }
    }
    wq = warp_max_pos(wq);
    if (use_w && lane < 4) wlist[wn + lane] = (unsigned short)kCand;   // pads the list to a multiple of 4
    __syncwarp();
    const float E = screen_error(Tmx, wq, hdr32[9]);

    // ---- the two points of this lane
    Points p = tile_points<FINAL, NW>(a, b, warp, lane);
    float px[2], py, pz, d1[2], d2[2], m1[2];
    py = (float)p.y * hy;
    pz = (float)p.z * hz;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        px[h] = (float)(p.x + 2 * h) * hx;
        d1[h] = INFINITY;
        d2[h] = INFINITY;
        m1[h] = 0.f;
    }
    auto nearer = [&](const float4 &q) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float dx = px[h] - q.x, dy = py - q.y, dz = pz - q.z;
            const float d = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
            if (d < d1[h]) {
                d2[h] = d1[h];
                d1[h] = d;
                m1[h] = q.w;
            } else if (d < d2[h]) {
                d2[h] = d;
            }
        }
    };
    if (use_w) {
        for (int i = 0; i < cnt; i += 4) {   // four candidates in flight
            const ushort4 j = *reinterpret_cast<const ushort4 *>(&wlist[i]);
            const float4 q0 = cand[j.x], q1 = cand[j.y], q2 = cand[j.z], q3 = cand[j.w];
            nearer(q0);
            nearer(q1);
            nearer(q2);
            nearer(q3);
        }
    } else {
        for (int i = 0; i < cnt; ++i) nearer(cand[i]);
    }

#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!p.valid[h]) continue;
        const float gap = screen_gap(d1[h], E, hdr32[10]);
        const bool clear = screen_clear(d1[h], d2[h], gap);
        Decision best{INFINITY, INFINITY, 0x7fffffff};
        if (!clear) {   // the candidates that can still win
            const double lim = (double)d1[h] + (double)gap;
            for (int i = 0; i < cnt; ++i) {
                const float4 q = cand[use_w ? (int)wlist[i] : i];
                const float dx = px[h] - q.x, dy = py - q.y, dz = pz - q.z;
                const float d = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                if ((double)d > lim) continue;
                const int m = __float_as_int(q.w);
                const double *c = a.cent + 3 * m;
                best.see(dist2_fp64(xs[p.x + 2 * h], ys[p.y], zs[p.z], c[0], c[1], c[2]), m);
            }
        }
        settle_point<FINAL, NW>(a, sh, p, h, clear, __float_as_int(m1[h]), best);
    }
    settle_tile<FINAL, NW>(a, sh, p, b);
}

// The tiles of pass t with more candidates than shared memory holds (centroids crowded in a part of a large cell),
// which km_assign has marked. Every use of the candidates takes the scanned centroids (the tile's list, or all) in
// chunks of kCand whose candidates are put into shared memory anew: a coordinate's FP64 subtraction is made once a
// chunk and CTA. Lists, bounds, decisions and counts of the warps are those of km_assign. A launch of its own after
// each pass with n_mu > kCand: as a branch or a function of km_assign it cost 2 to 7 % of every pass (registers); a
// launch that finds no tile costs 1.3 us. 20 passes at 128^3 of 4,096 centroids started in a ball of 14 spacings and of
// 8,192 in one of 20: 445 and 475 ms when every use of a candidate formed its coordinates, 66 and 82 with room for all
// centroids in each CTA's shared memory (one or three CTAs a SM), now 48 and 43.
template <bool FINAL, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? 4 : 8) km_crowded(KmArgs a, int t)
{
    constexpr int NT = 32 * NW;
    grid_wait();
    if (a.ctl->error || a.ctl->crowds[t & 1] == 0u || (!FINAL && a.ctl->converged)) return;
    TILE_SHARED(sh);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_tiles = a.ntx * a.nty * a.ntz;
#pragma unroll 1
    for (int b = blockIdx.x; b < n_tiles; b += gridDim.x) {
        if (a.jpart[b] != kCrowd) continue;
        __syncthreads();   // shared memory is free, and every thread has read the mark
        tile_tables(a, sh, b);
        // the list, if it fits: of this pass or one that still holds (km_assign); the final pass has none
        const unsigned short *list = reinterpret_cast<const unsigned short *>(a.dist) + (int64_t)b * (a.list_cap + 1);
        int n_scan = a.n_mu;
        if (!FINAL && a.list_cap > 0 && list[0] <= a.list_cap) n_scan = *list++;
        else list = nullptr;
        __syncthreads();
        const float minub = tile_min_upper(a, sh, list, n_scan), sminub = sqrtf(minub);
        const float hx = sh.hdr32[0], hy = sh.hdr32[1], hz = sh.hdr32[2];
        const float Px = sh.hdr32[3], Py = sh.hdr32[4], Pz = sh.hdr32[5];
        Points p = tile_points<FINAL, NW>(a, b, warp, lane);
        float4 *cand = sh.cand;
        unsigned short *wlist = sh.wlist[warp];
        // by all threads: use(n) for every chunk, its n candidates in cand
        auto chunks = [&](auto &&use) {
#pragma unroll 1
            for (int base = 0; base < n_scan; base += kCand) {
                __syncthreads();
                if (tid == 0) sh.counts[0] = 0u;
                __syncthreads();
                for (int i = base + tid; i < min(n_scan, base + kCand); i += NT) {
                    const int m = list ? (int)list[i] : i;
                    const float4 c = a.c32[m];
                    const float lb = tile_lower(c.x - sh.hdr32[6], c.y - sh.hdr32[7], c.z - sh.hdr32[8], Px, Py, Pz);
                    if (tile_reaches(lb, minub, sminub, a.scan_err))
                        cand[atomicAdd(&sh.counts[0], 1u)] = tile_local(a, sh, m);
                }
                __syncthreads();
                use((int)sh.counts[0]);
            }
            __syncthreads();
        };
        // this warp's sub-cube
        const int bx = p.x & 4, by = p.y & 4, bz = p.z & 4;
        const int ex = min(NW == 8 ? TX : TX / 2, a.nx - b / (a.ntz * a.nty) * (NW == 8 ? TX : TX / 2));
        const int ey = min(TY, a.ny - (b / a.ntz) % a.nty * TY), ez = min(TZ, a.nz - b % a.ntz * TZ);
        const float Sx0 = bx * hx, Sy0 = by * hy, Sz0 = bz * hz;
        const float Sx1 = Sx0 + (min(4, ex - bx) - 1) * hx, Sy1 = Sy0 + (min(4, ey - by) - 1) * hy;
        const float Sz1 = Sz0 + (min(4, ez - bz) - 1) * hz;
        float wub = INFINITY;
        chunks([&](int n) {
            for (int j = lane; j < n; j += 32)
                wub = fminf(wub, box_upper(cand[j].x, cand[j].y, cand[j].z, Sx0, Sy0, Sz0, Sx1, Sy1, Sz1));
        });
        const float Tmx = fmaxf(Px, fmaxf(Py, Pz)), wcut = warp_cut(warp_min_pos(wub), Tmx);
        int wn = 0;
        float wq = 0.f, tq = 0.f;   // largest coordinates of the warp's and of the tile's candidates
        chunks([&](int n) {
            for (int base = 0; base < n; base += 32) {
                const int j = base + lane;
                bool keep = false;
                float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                if (j < n) {
                    q = cand[j];
                    const float qq = fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z)));
                    keep = box_lower(q.x, q.y, q.z, Sx0, Sy0, Sz0, Sx1, Sy1, Sz1) * 0.9999f <= wcut;
                    tq = fmaxf(tq, qq);
                    if (keep) wq = fmaxf(wq, qq);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                const int pos = wn + __popc(bal & ((1u << lane) - 1u));
                if (keep && pos < kWarpCap) wlist[pos] = (unsigned short)__float_as_int(q.w);
                wn += __popc(bal);
            }
        });
        const bool use_w = wn <= kWarpCap;   // else all of the tile's candidates
        const float E = screen_error(Tmx, warp_max_pos(use_w ? wq : tq), sh.hdr32[9]);
        // by all threads: see(q) for each of the warp's candidates if the warp wants them, the listed ones through the
        // warp's share of cand
        auto walk = [&](bool want, auto &&see) {
            if (__syncthreads_or(want && !use_w))
                chunks([&](int n) {
                    if (want && !use_w)
                        for (int i = 0; i < n; ++i) see(cand[i]);
                });
            if (want && use_w) {
                constexpr int share = kCand / NW;
                float4 *own = cand + warp * share;
#pragma unroll 1
                for (int base = 0; base < wn; base += share) {
                    const int n = min(share, wn - base);
                    __syncwarp();
                    for (int i = lane; i < n; i += 32) own[i] = tile_local(a, sh, (int)wlist[base + i]);
                    __syncwarp();
                    for (int i = 0; i < n; ++i) see(own[i]);
                }
            }
            __syncthreads();
        };
        float px[2], d1[2], d2[2], m1[2];
        const float py = (float)p.y * hy, pz = (float)p.z * hz;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            px[h] = (float)(p.x + 2 * h) * hx;
            d1[h] = d2[h] = INFINITY;
            m1[h] = 0.f;
        }
        walk(true, [&](const float4 &q) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float dx = px[h] - q.x, dy = py - q.y, dz = pz - q.z;
                const float d = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                if (d < d1[h]) {
                    d2[h] = d1[h];
                    d1[h] = d;
                    m1[h] = q.w;
                } else if (d < d2[h]) {
                    d2[h] = d;
                }
            }
        });
        float lim[2];   // who is beyond cannot win (rounded up: one candidate more changes nothing)
        bool close[2];
        Decision best[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float gap = screen_gap(d1[h], E, sh.hdr32[10]);
            close[h] = p.valid[h] && !screen_clear(d1[h], d2[h], gap);
            lim[h] = __fadd_ru(d1[h], gap);
            best[h] = Decision{INFINITY, INFINITY, 0x7fffffff};
        }
        walk(__any_sync(0xffffffffu, close[0] || close[1]), [&](const float4 &q) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float dx = px[h] - q.x, dy = py - q.y, dz = pz - q.z;
                if (!close[h] || fmaf(dz, dz, fmaf(dy, dy, dx * dx)) > lim[h]) continue;
                const int m = __float_as_int(q.w);
                const double *at = a.cent + 3 * m;
                best[h].see(dist2_fp64(sh.xs[p.x + 2 * h], sh.ys[p.y], sh.zs[p.z], at[0], at[1], at[2]), m);
            }
        });
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (p.valid[h]) settle_point<FINAL, NW>(a, sh, p, h, !close[h], __float_as_int(m1[h]), best[h]);
        settle_tile<FINAL, NW>(a, sh, p, b);
        if (!FINAL && !a.want_obj && tid == 0) a.jpart[b] = 0.0;
    }
}

// deterministic sum of the per-tile objective partials (one CTA)
__device__ double sum_partials(const double *p, int n, double *red)
{
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 16 * (int)blockDim.x) {
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = i + k * (int)blockDim.x < n ? p[i + k * (int)blockDim.x] : 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = __dadd_rn(x[k], x[k + 8]);
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = __dadd_rn(x[k], x[k + 4]);
        v = __dadd_rn(v, __dadd_rn(__dadd_rn(x[0], x[2]), __dadd_rn(x[1], x[3])));
    }
    return block_sum(v, red);
}

// Centroids of update t from the running sums; the last block adds the objective's partials instead, with 256 threads
// and 16 loads in flight (64 threads took 31 us for 4,096 partials). The largest
// move of a centroid (rounded up) decides whether the next pass may use the tiles' lists.
constexpr int kUpd = 64;        // centroids of an update block: the FP64 divisions spread over many SMs
__global__ void __launch_bounds__(256) km_update(KmArgs a, int t, int n_tiles, double *objective)
{
    __shared__ double red[32];
    grid_wait();
    grid_release();
    if (a.ctl->error || a.ctl->converged) return;
    if (blockIdx.x == gridDim.x - 1) {
        if (objective) {
            const double J = sum_partials(a.jpart, n_tiles, red);
            if (threadIdx.x == 0) objective[t] = J;
        }
        if (threadIdx.x == 0) {
            a.ctl->moved[(t + 1) & 1] = 0u;   // read by pass t (done), next written by update t + 1
            a.ctl->n_iter = t + 1;
        }
        return;
    }
    if (threadIdx.x >= kUpd) return;
    const int m = blockIdx.x * kUpd + threadIdx.x;
    float move = 0.f;
    if (m < a.n_mu) {
        const unsigned long long *q = &a.acc[8 * (int64_t)m];
        if ((q[0] | q[1]) != 0ull) {
            const double sw = u128_to_double(q[0], q[1]);
            const double cx = __ddiv_rn(u128_to_double(q[2], q[3]), sw);
            const double cy = __ddiv_rn(u128_to_double(q[4], q[5]), sw);
            const double cz = __ddiv_rn(u128_to_double(q[6], q[7]), sw);
            const double px = a.cent[3 * m], py = a.cent[3 * m + 1], pz = a.cent[3 * m + 2];
            const bool same = __double_as_longlong(cx) == __double_as_longlong(px) &&
                              __double_as_longlong(cy) == __double_as_longlong(py) &&
                              __double_as_longlong(cz) == __double_as_longlong(pz);
            if (!same) {
                if (a.early_stop) atomicOr(&a.ctl->moved[t & 1], 1u);
                a.cent[3 * m + 0] = cx;
                a.cent[3 * m + 1] = cy;
                a.cent[3 * m + 2] = cz;
                const float4 c = make_float4((float)cx, (float)cy, (float)cz, 0.f);
                a.c32[m] = c;
                // the FP32 difference of each coordinate is off by 2^-23 L at most
                const float dx = c.x - (float)px, dy = c.y - (float)py, dz = c.z - (float)pz;
                move = sqrtf(dx * dx + dy * dy + dz * dz) * 1.00001f + a.scan_err;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) move = fmaxf(move, __shfl_xor_sync(0xffffffffu, move, o));
    if ((threadIdx.x & 31) == 0 && move > 0.f) atomicMax(&a.ctl->disp[t & 1], __float_as_uint(move));
}

__global__ void km_snap(KmArgs a, int64_t n_r)
{
    if (a.ctl->error) return;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_r; r += (int64_t)gridDim.x * blockDim.x) {
        const int m = a.labels[r];
        if (m < 0) continue;
        if ((unsigned long long)__double_as_longlong(a.dist[r]) == a.best[m]) atomicMin(&a.idx_u[m], (unsigned long long)r);
    }
}

__global__ void km_finish(KmArgs a, int max_iter, int n_tiles, int64_t *idx, double *centroids, double *objective,
                          int64_t *stats)
{
    __shared__ double red[32];
    __shared__ int empty_sh;
    if (threadIdx.x == 0) empty_sh = 0;
    __syncthreads();
    const int err = a.ctl->error;
    const double J = sum_partials(a.jpart, n_tiles, red);
    int empty = 0;
    for (int m = threadIdx.x; m < a.n_mu; m += blockDim.x) {
        const unsigned long long u = a.idx_u[m];
        const bool e = err || u == ~0ull;
        idx[m] = e ? -1 : (int64_t)u;
        empty += e ? 1 : 0;
        if (centroids) {
            centroids[3 * m + 0] = a.cent[3 * m + 0];
            centroids[3 * m + 1] = a.cent[3 * m + 1];
            centroids[3 * m + 2] = a.cent[3 * m + 2];
        }
    }
    atomicAdd(&empty_sh, empty);
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nit = a.ctl->converged ? a.ctl->n_iter : max_iter;
        if (objective) {
            objective[max_iter] = J;
            for (int p = nit + 1; p < max_iter; ++p) objective[p] = objective[nit];
        }
        if (stats) {
            stats[0] = nit;
            stats[1] = (int64_t)a.ctl->ties;
            stats[2] = err == 2 ? -2 : (err ? -1 : empty_sh);
            stats[3] = (int64_t)a.ctl->refined;
        }
    }
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

struct WsLayout {
    size_t cent, c32, acc, labels, dist, jpart, best, idx_u, ctl, total;
};

WsLayout ws_layout(int64_t n_r, int n_mu, int n_tiles)
{
    WsLayout L;
    size_t o = 0;
    L.cent = o; o = align256(o + sizeof(double) * 3 * n_mu);
    L.c32 = o; o = align256(o + sizeof(float4) * n_mu);
    L.acc = o; o = align256(o + sizeof(unsigned long long) * 8 * n_mu);
    L.labels = o; o = align256(o + sizeof(int32_t) * n_r);
    L.dist = o; o = align256(o + sizeof(double) * n_r);
    L.jpart = o; o = align256(o + sizeof(double) * n_tiles);
    L.best = o; o = align256(o + sizeof(unsigned long long) * n_mu);
    L.idx_u = o; o = align256(o + sizeof(unsigned long long) * n_mu);
    L.ctl = o; o = align256(o + sizeof(KmCtl));
    L.total = o;
    return L;
}

int bits_of(uint64_t v)
{
    int b = 0;
    while (v) {
        ++b;
        v >>= 1;
    }
    return b;
}

// CTA tiles of the assignment: 8 x 8 x 8, or 4 x 8 x 8 halves when the grid has fewer than two full
// tiles per SM of the 152 (the halves' own candidate scans cost less than the idle SMs)
struct TilePlan {
    int half, ntx, nty, ntz, n_tiles;
};

TilePlan tile_plan(int nx, int ny, int nz)
{
    TilePlan p;
    p.nty = (ny + TY - 1) / TY;
    p.ntz = (nz + TZ - 1) / TZ;
    const int full = ((nx + TX - 1) / TX) * p.nty * p.ntz;
    p.half = full < 2 * 152 ? 1 : 0;
    const int tx = p.half ? TX / 2 : TX;
    p.ntx = (nx + tx - 1) / tx;
    p.n_tiles = p.ntx * p.nty * p.ntz;
    return p;
}

}  // namespace

extern "C" isdf_status isdf_kmeans_workspace(int32_t nx, int32_t ny, int32_t nz, int32_t n_mu, size_t *ws_bytes)
{
    if (nx < 1 || ny < 1 || nz < 1 || n_mu < 1 || !ws_bytes) return ISDF_ERR_INVALID_ARG;
    const int64_t n_r = (int64_t)nx * ny * nz;
    *ws_bytes = ws_layout(n_r, n_mu, tile_plan(nx, ny, nz).n_tiles).total;
    return ISDF_OK;
}

extern "C" isdf_status isdf_kmeans(const double *w, int32_t nx, int32_t ny, int32_t nz, const double *cell,
                                   int32_t n_mu, const int64_t *init_idx, int32_t max_iter, int32_t flags,
                                   int64_t *idx, double *centroids, double *objective, int32_t *labels,
                                   int64_t *stats, void *ws, size_t ws_bytes, void *stream)
{
    if (nx < 1 || ny < 1 || nz < 1 || !cell || !w || !init_idx || !idx) return ISDF_ERR_INVALID_ARG;
    const int64_t n_r = (int64_t)nx * ny * nz;
    if (n_r >= ((int64_t)1 << 31)) return ISDF_ERR_UNSUPPORTED;
    if (n_mu < 1 || n_mu > n_r || max_iter < 0 || (flags & ~ISDF_KMEANS_EARLY_STOP)) return ISDF_ERR_INVALID_ARG;
    if (n_mu > kMaxMu) return ISDF_ERR_UNSUPPORTED;
    for (int k = 0; k < 3; ++k)
        if (!(cell[k] > 0.0) || cell[k] > 1e300) return ISDF_ERR_INVALID_ARG;
    const TilePlan tp = tile_plan(nx, ny, nz);
    const int ntx = tp.ntx, nty = tp.nty, ntz = tp.ntz;
    const int n_tiles = tp.n_tiles;
    const WsLayout L = ws_layout(n_r, n_mu, n_tiles);
    if (!ws || ws_bytes < L.total || !aligned(ws, 256)) return ISDF_ERR_WORKSPACE;
    char *base = static_cast<char *>(ws);

    KmArgs a;
    a.w = w;
    a.nx = nx;
    a.ny = ny;
    a.nz = nz;
    a.hx = cell[0] / nx;
    a.hy = cell[1] / ny;
    a.hz = cell[2] / nz;
    double hmin = a.hx < a.hy ? a.hx : a.hy;
    hmin = hmin < a.hz ? hmin : a.hz;
    a.tie_floor = hmin * hmin;
    a.n_mu = n_mu;
    double lmax = 1.0;
    for (int k = 0; k < 3; ++k) lmax = cell[k] > lmax ? cell[k] : lmax;
    int el = 0;
    frexp(lmax, &el);
    a.s_base = 126 - (bits_of((uint64_t)n_r) + el);
    a.ntx = ntx;
    a.nty = nty;
    a.ntz = ntz;
    a.cent = reinterpret_cast<double *>(base + L.cent);
    a.c32 = reinterpret_cast<float4 *>(base + L.c32);
    a.acc = reinterpret_cast<unsigned long long *>(base + L.acc);
    a.labels = labels ? labels : reinterpret_cast<int32_t *>(base + L.labels);
    a.dist = reinterpret_cast<double *>(base + L.dist);
    a.jpart = reinterpret_cast<double *>(base + L.jpart);
    a.best = reinterpret_cast<unsigned long long *>(base + L.best);
    a.idx_u = reinterpret_cast<unsigned long long *>(base + L.idx_u);
    a.ctl = reinterpret_cast<KmCtl *>(base + L.ctl);
    a.early_stop = (flags & ISDF_KMEANS_EARLY_STOP) ? 1 : 0;
    a.want_obj = objective ? 1 : 0;
    a.h32[0] = (float)a.hx;
    a.h32[1] = (float)a.hy;
    a.h32[2] = (float)a.hz;
    a.lmax32 = (float)lmax;
    a.tie_floor32 = (float)a.tie_floor;
    // |float(c) - c| + |float(o) - o| + rounding of their difference, for |c|, |o| <= L
    a.scan_err = (float)(4.0 * 5.9604644775390625e-8 * lmax * 1.01);

    cudaStream_t st = as_stream(stream);
    // the lists live in the final pass's distances: what a tile's share of them holds, 16 bits a centroid
    const int64_t words = n_r * 4 / n_tiles - 1;
    a.list_cap = (int)(words > 4096 ? 4096 : words);
    a.h_ref = (float)((a.hx + a.hy + a.hz) / 3.0);
    const int64_t nmax = n_r > n_mu ? n_r : n_mu;
    const unsigned ginit = (unsigned)((nmax + 255) / 256 < 4096 ? (nmax + 255) / 256 : 4096);
    km_init<<<ginit, 256, 0, st>>>(a, init_idx, n_r); isdf_note_launch();
    km_wmax<<<(unsigned)((n_r + 255) / 256 < 1024 ? (n_r + 255) / 256 : 1024), 256, 0, st>>>(a, n_r); isdf_note_launch();
    km_check_scale<<<1, 32, 0, st>>>(a); isdf_note_launch();
    ISDF_LAUNCH_CHECK();
    const unsigned gmu = (unsigned)((n_mu + kUpd - 1) / kUpd) + 1;   // the last block: the objective
    const int resident = 152 * (tp.half ? 8 : 4);   // CTAs of km_crowded; none when shared memory holds all centroids
    const int crowds = n_mu <= kCand ? 0 : n_tiles < resident ? n_tiles : resident;
    for (int t = 0; t < max_iter; ++t) {
        if (tp.half) ISDF_CUDA_TRY(launch_chained(km_assign<false, 4>, n_tiles, 128, st, a, t));
        else ISDF_CUDA_TRY(launch_chained(km_assign<false, 8>, n_tiles, kThreads, st, a, t));
        isdf_note_launch();
        if (crowds) {
            if (tp.half) ISDF_CUDA_TRY(launch_chained(km_crowded<false, 4>, crowds, 128, st, a, t));
            else ISDF_CUDA_TRY(launch_chained(km_crowded<false, 8>, crowds, kThreads, st, a, t));
            isdf_note_launch();
        }
        ISDF_CUDA_TRY(launch_chained(km_update, gmu, 256, st, a, t, n_tiles, objective));
        isdf_note_launch();
    }
    if (tp.half) km_assign<true, 4><<<n_tiles, 128, 0, st>>>(a, max_iter);
    else km_assign<true, 8><<<n_tiles, kThreads, 0, st>>>(a, max_iter);
    isdf_note_launch();
    if (crowds) {
        if (tp.half) km_crowded<true, 4><<<crowds, 128, 0, st>>>(a, max_iter);
        else km_crowded<true, 8><<<crowds, kThreads, 0, st>>>(a, max_iter);
        isdf_note_launch();
    }
    km_snap<<<(unsigned)((n_r + 255) / 256 < 4096 ? (n_r + 255) / 256 : 4096), 256, 0, st>>>(a, n_r); isdf_note_launch();
    km_finish<<<1, 256, 0, st>>>(a, max_iter, n_tiles, idx, centroids, objective, stats); isdf_note_launch();
    ISDF_LAUNCH_CHECK();
    return ISDF_OK;
}

extern "C" isdf_status isdf_kmeans_status(const int64_t *stats, void *stream)
{
    if (!stats) return ISDF_ERR_INVALID_ARG;
    ISDF_CUDA_TRY(cudaStreamSynchronize(as_stream(stream)));
    int64_t h[4] = {0, 0, 0, 0};
    ISDF_CUDA_TRY(cudaMemcpy(h, stats, sizeof(h), cudaMemcpyDeviceToHost));
    if (h[2] == -2) return ISDF_ERR_INVALID_ARG;
    if (h[2] < 0) return ISDF_ERR_NONFINITE;
    return h[2] > 0 ? ISDF_ERR_EMPTY_CLUSTER : ISDF_OK;
}
