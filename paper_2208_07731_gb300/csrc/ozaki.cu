// FP64 complex GEMM on the tcgen05 tensor cores by exact integer slicing
// (Ozaki, Ogita, Oishi and Rump, 2012; on FP16 tensor cores whose integer
// products are exact: Mukunoki, Ozaki, Ogita and Imamura, 2020).
//
// Real form: an interleaved complex row of op(A) is a real row of length 2K;
// for x = conj(op(B)(k, n)) the rotated real rows
//     Bh[2n] = (Re x, Im x, ...),   Bh[2n+1] = (-Im x, Re x, ...)
// make (A Bh^T)[m][2n + p] part p of (op(A) op(B))[m][n].
//
// Slicing: every real row r gets E_r with max |x| < 2^E_r, and each entry is
// rounded to F = round(x 2^(56 - E_r)) and written in balanced base 256,
// F = sum_{s=1..7} d_s 2^(56 - 8 s) with d_2..d_7 in [-128, 127] and
// |d_1| <= 256, so x = sum_s d_s 2^(E_r - 8 s) up to a rounding below
// 2^(E_r - 57); integer operations only, no FP64 arithmetic.
//
// Products: for every pair (s, t) with s + t <= 8 (28 pairs), an FP16 GEMM of
// the digit matrices gives integers. A product of two digits is at most 2^14
// (2^15 with one leading digit, 2^16 with both), so 64 real terms of a pair
// add up to at most 1, 2 or 4 units of 2^20, and every TMEM accumulation takes
// at most 16 units: all its partial sums are integers up to 2^24, exact in the
// FP32 accumulator in any order. The epilogue converts an accumulation to
// int32 and adds those of one group g = s + t exactly (K slabs of at most
// 14,336 real terms keep a group's sum below 2^31). The result is
// alpha 2^(E_m + E_n - 64) S, S = sum_g 2^(8 (8 - g)) S_g an integer below
// 2^80, rounded to FP64 by integer operations, once or (round_steps) group by
// group. The neglected pairs
// (s + t > 8, digits of either sign) and the rounding of the operands stay
// below ~2^-55 K max|a| max|b| per output, the size of an FP64 GEMM's rounding
// error.
//
// Kernel (oz_gemm): persistent CTA pairs (clusters of two, cta_group::2) on
// 256 x 256 tiles, 320 threads a CTA: a TMA warp (6-stage ring of one 128 x 64
// digit tile of A and one of B per CTA), an MMA warp in the leader and 8
// epilogue warps; the 256-column TMEM accumulator is double buffered. Per MMA
// each SM reads 64 operand bytes a clock from shared memory; 128 x 128 tiles on
// single CTAs read 128, the limit, and their 28 segment-wise drains per 256
// real terms (16 conversions a clock per SM) took as long as the MMAs: the
// unit rule needs 11. The list of a tile's (pair, K chunk) steps may be cut into
// pieces so that the work items fill the chip; an item writes its groups' int32
// sums to memory (integer atomics where a group is cut: the order does not
// matter) and oz_combine rounds them. Outputs larger than the sums' buffer run
// in chunks of rows, two tiles per CTA pair at a time. (Rounding inside the GEMM
// instead: 8 or 16 epilogue warps a SM against 64 of oz_combine, and the sums of
// the tiles in flight, 139 MB, thrash L2 all the same; the fit below 30.0 ms
// against 27.0.)
// Measured against 128 x 128 single-CTA tiles with a drain per 256 real terms of
// a pair: FP64 Theta fit of 108,000 rows, N = 120, N_mu = 1000, 70.1 -> 27.0 ms
// (GEMM 20.6, of which the MMAs are 18; oz_combine 4.1, at HBM speed); the FP64
// autograd pass of 32^3, N = 48, N_mu = 320, 52.9 -> 13.2 ms (its reductions over
// 32,768 grid rows had 15 CTAs: pieces fill the chip). Narrowing the MMA of a last
// column tile to the columns that exist gave nothing (27.0 -> 27.3, 12.3 -> 12.4):
// operand feed and epilogue set the pace, and the full tiles paid for the test.
#include <cudaTypedefs.h>

#include "ozaki.cuh"
#include "tc.cuh"

namespace {

constexpr int OPM = 256, OPN = 256;             // pair tile: rows, real columns
constexpr int OSTAGES = 6;
constexpr int OTILE = OTM * OTK * 2;            // bytes of one digit tile
constexpr int OSTAGE = 2 * OTILE;               // per CTA
constexpr int NGROUP = 7, NPAIR = 28;           // groups g = 2..8, pairs s + t <= 8
constexpr int UNITS = 16;                       // 2^20 units of one TMEM accumulation: sums up to 2^24
constexpr int OEPI = 8;
constexpr int OHC = OPN / (OEPI / 4);           // columns of an epilogue thread
constexpr int OTHREADS = 64 + 32 * OEPI;
constexpr int OSMEM = OSTAGES * OSTAGE + 1024;
constexpr int64_t GTILE = (int64_t)OPM * OPN;   // outputs of a pair tile
constexpr long long OWAIT = 200000000LL;        // SM cycles (~0.1 s)

struct OzArgs {
    int M, N, K;            // complex sizes; K of this slab
    int k0;                 // first complex k of this slab (for the triangular K ranges)
    int Ra, Rb;             // padded real rows of one slice of A / of Bh
    int kchunks;            // padded real K of the slab / 64
    int batch, n_tm, n_tn;  // pair tiles per batch product
    int per;                // computed tiles per batch product (lower_only: those on or below the diagonal)
    int pieces;             // work items per tile
    int row0;               // first row of this launch (a multiple of OPM)
    int kmode, k_to_m_end, lower_only, beta;
    int lower_tiles;        // tiles are listed by tile_of's triangular rule
    double alpha;
    double2 *C;
    int64_t ldc, bsc;
    const int *ea, *eb;     // row exponents E: max |x| < 2^E (batch-major: M and N per product)
    int *gsum;              // exact group sums [tile][g - 2][CTA][column][128 rows]
    int *err;               // 1: a bounded wait gave up; 2: a non-finite operand entry
    long long budget;       // cycle budget of the pipeline waits (the drain waits keep OWAIT)
    long long never;        // > 0: test hook, the MMA issuer first waits this long on a barrier nothing signals
};

// The 28 pairs in the order they are run: group g = s + t, slice s, units of 2^20 per chunk of 64 real terms. Groups
// 8 | 7, 2 | 6, 3 | 5, 4 hold seven pairs each: a list cut in two or four pieces is cut between groups.
__constant__ unsigned char kPairG[NPAIR] = {8, 8, 8, 8, 8, 8, 8, 7, 7, 7, 7, 7, 7, 2, 6, 6, 6, 6, 6, 3, 3, 5, 5, 5, 5, 4, 4, 4};
__constant__ unsigned char kPairS[NPAIR] = {1, 2, 3, 4, 5, 6, 7, 1, 2, 3, 4, 5, 6, 1, 1, 2, 3, 4, 5, 1, 2, 1, 2, 3, 4, 1, 2, 3};
__constant__ unsigned char kPairU[NPAIR] = {2, 1, 1, 1, 1, 1, 2, 2, 1, 1, 1, 1, 2, 4, 2, 1, 1, 1, 2, 2, 2, 2, 1, 1, 2, 2, 1, 2};

// The 7 balanced base-256 digits of x relative to 2^E (|x| < 2^E), from the bits of x: F = round(x 2^(56 - E)) (half
// away from zero), then d_7 .. d_2 in [-128, 127] from the bottom and d_1 = what remains (|d_1| <= 256), so that x ~
// sum_s d_s 2^(E - 8 s). Returned as G = F + sum_{k < 6} 128 256^k: byte k of G is d_(7 - k) + 128, G >> 48 is d_1.
__device__ __forceinline__ long long digits(double x, int E)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (ef ? (1ull << 52) : 0ull);
    const int sh = (ef ? ef : 1) - 1019 - E;   // |x| 2^(56 - E) = m 2^sh
    long long f = 0;
    if (sh >= 0 && sh < 8) f = (long long)(m << sh);
    else if (sh < 0 && sh > -64) f = (long long)((m + (1ull << (-sh - 1))) >> (-sh));
    if (b >> 63) f = -f;
    return f + 0x808080808080ll;
}

// digits s of two entries as FP16 (x in the low half): 0x6400 + v is 1024 + v in FP16 for 0 <= v < 1024
__device__ __forceinline__ __half2 digit_pair(long long gx, long long gy, int s)
{
    uint32_t w, bias;
    if (s > 0) {
        const int k = NSLICE - 1 - s;   // byte of G
        const uint32_t x = k < 4 ? (uint32_t)gx : (uint32_t)(gx >> 32), y = k < 4 ? (uint32_t)gy : (uint32_t)(gy >> 32);
        w = __byte_perm(x, y, (k & 3) | 0x0080 | (4 + (k & 3)) << 8 | 0x8000) & 0x00FF00FFu;
        bias = 0x64806480u;             // 1152
    } else {
        w = (uint32_t)((int)(gx >> 48) + 512) | (uint32_t)((int)(gy >> 48) + 512) << 16;
        bias = 0x66006600u;             // 1536
    }
    w |= 0x64006400u;
    return __hsub2(*reinterpret_cast<const __half2 *>(&w), *reinterpret_cast<const __half2 *>(&bias));
}

// complex128 entry, or complex64 widened exactly by moving bits (no FP64 instruction)
__device__ __forceinline__ double2 load_c(const double2 *p, int64_t i) { return p[i]; }
__device__ __forceinline__ double2 load_c(const float2 *p, int64_t i)
{
    const float2 v = p[i];
    return make_double2(f2d_int(v.x), f2d_int(v.y));
}

// ---- operand preparation: two launches per product for both operands (row maxima; exponents and digit slices)
constexpr int SK = 128;      // complex k of one slicing block

// an operand read as R rows of K complex entries X[r sr + k sk] (product b at X + b bs): plain (A role: real row r =
// (Re, Im) interleaved over k) or rotated (B role: rows 2r and 2r+1 of Bh for x = value, conjugated when conj is set)
struct OzOperand {
    const void *X;
    int64_t sr, sk, bs;
    int R, Rp;               // rows; padded real rows of a slice
    int conj, rotated;
    unsigned int *part;      // [k part][b][R]: max of the entries' high words (sign off): the exponent is all that counts
    int *e;                  // [b][R]: row exponents
    __half *out;             // slice s of row r of product b at out[((b NSLICE + s) Rp + row) Kp + column]
};

__device__ __forceinline__ unsigned int high_max(double2 v)
{
    const unsigned int a = (unsigned int)__double2hiint(v.x) & 0x7FFFFFFFu, b = (unsigned int)__double2hiint(v.y) & 0x7FFFFFFFu;
    return a > b ? a : b;
}

// rows r0 .. r0 + 31, k part q
template <typename T>
__device__ void max_part(const OzOperand &o, int K, int r0, int q, int b, int batch, int *err, unsigned int (*sh)[32])
{
    const T *X = static_cast<const T *>(o.X) + (int64_t)b * o.bs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k0 = q * PK;
    if (o.sk == 1) {   // lanes along k, four rows a warp
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + 4 * warp + i;
            unsigned int m = 0u;
            if (r < o.R) {
#pragma unroll
                for (int j = 0; j < PK / 32; ++j) {
                    const int k = k0 + 32 * j + lane;
                    if (k < K) m = max(m, high_max(load_c(X, (int64_t)r * o.sr + k)));
                }
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) sh[0][4 * warp + i] = m;
        }
    } else {           // lanes along r
        const int r = r0 + lane;
        unsigned int m = 0u;
        if (r < o.R) {
#pragma unroll 8
            for (int j = 0; j < PK / 8; ++j) {
                const int k = k0 + 8 * j + warp;
                if (k < K) m = max(m, high_max(load_c(X, (int64_t)r * o.sr + (int64_t)k * o.sk)));
            }
        }
        sh[warp][lane] = m;
        __syncthreads();
        if (warp == 0)
            for (int i = 1; i < 8; ++i) sh[0][lane] = max(sh[0][lane], sh[i][lane]);
    }
    __syncthreads();
    if (warp == 0 && r0 + lane < o.R) {
        const unsigned int m = sh[0][lane];
        o.part[((int64_t)q * batch + b) * o.R + r0 + lane] = m;
        // an infinity or NaN (exponent field all ones) cannot be sliced: recorded, not computed on
        if (m >= 0x7FF00000u) atomicCAS(err, 0, 2);
    }
}

// The row-maximum parts of both operands; the blocks after them clear the group sums that pieces will be added to.
template <typename TA, typename TB>
__global__ void __launch_bounds__(256) oz_rowmax(OzOperand A, OzOperand B, int K, int parts, int *err, int4 *zero, int64_t nz)
{
    __shared__ unsigned int sh[8][32];
    const int na = (A.R + 31) / 32 * parts, nb = (B.R + 31) / 32 * parts, bid = blockIdx.x, b = blockIdx.y;
    if (bid < na) {
        max_part<TA>(A, K, bid / parts * 32, bid % parts, b, gridDim.y, err, sh);
    } else if (bid < na + nb) {
        max_part<TB>(B, K, (bid - na) / parts * 32, (bid - na) % parts, b, gridDim.y, err, sh);
    } else if (b == 0) {
        const int64_t step = (int64_t)(gridDim.x - na - nb) * 256;
        for (int64_t i = (int64_t)(bid - na - nb) * 256 + threadIdx.x; i < nz; i += step) zero[i] = make_int4(0, 0, 0, 0);
    }
}

// rows r0 .. r0 + 31 (padding rows and columns are written as zeros), complex columns k0 .. k0 + SK - 1
template <typename T>
__device__ void slice_part(const OzOperand &o, int K, int64_t Kp, int parts, int r0, int kb, int b, int batch, double2 (*t)[33],
                           int *ex)
{
    const T *X = static_cast<const T *>(o.X) + (int64_t)b * o.bs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rpad = o.rotated ? o.Rp / 2 : o.Rp;
    const int64_t kp2 = Kp / 2;
    if (warp == 0) {
        unsigned int m = 0u;
        const int r = r0 + lane;
        if (r < o.R)
            for (int q = 0; q < parts; ++q) m = max(m, o.part[((int64_t)q * batch + b) * o.R + r]);
        ex[lane] = (int)(m >> 20) - 1022;
        if (kb == 0 && r < o.R) o.e[(int64_t)b * o.R + r] = ex[lane];
    }
    __half2 *o2 = reinterpret_cast<__half2 *>(o.out);
    const bool kfast = o.sk == 1;
    for (int k0 = kb; k0 < min((int)kp2, kb + SK); k0 += 32) {
        __syncthreads();
        for (int i = warp; i < 32; i += 8) {
            const int r = kfast ? r0 + i : r0 + lane, k = kfast ? k0 + lane : k0 + i;
            double2 v = make_double2(0.0, 0.0);
            if (r < o.R && k < K) {
                v = load_c(X, (int64_t)r * o.sr + (int64_t)k * o.sk);
                if (o.conj) v.y = -v.y;
            }
            if (kfast) t[i][lane] = v;
            else t[lane][i] = v;
        }
        __syncthreads();
        for (int i = warp; i < 32; i += 8) {
            const int r = r0 + i, k = k0 + lane;
            if (r >= rpad || k >= kp2) continue;
            const double2 v = t[i][lane];   // zero outside R x K
            const long long gx = digits(v.x, ex[i]), gy = digits(v.y, ex[i]);
#pragma unroll
            for (int s = 0; s < NSLICE; ++s) {
                const int64_t sl = (int64_t)b * NSLICE + s;
                const __half2 d = digit_pair(gx, gy, s);
                if (!o.rotated) {
                    o2[(sl * o.Rp + r) * kp2 + k] = d;
                } else {
                    o2[(sl * o.Rp + 2 * r) * kp2 + k] = d;
                    o2[(sl * o.Rp + 2 * r + 1) * kp2 + k] = __halves2half2(__hneg(__high2half(d)), __low2half(d));
                }
            }
        }
    }
}

template <typename TA, typename TB>
__global__ void __launch_bounds__(256) oz_slice(OzOperand A, OzOperand B, int K, int64_t Kp, int parts)
{
    __shared__ double2 t[32][33];
    __shared__ int ex[32];
    const int kblocks = (int)((Kp / 2 + SK - 1) / SK), bid = blockIdx.x, b = blockIdx.y;
    const int na = A.Rp / 32 * kblocks;   // A is plain, B rotated
    if (bid < na) slice_part<TA>(A, K, Kp, parts, bid / kblocks * 32, bid % kblocks * SK, b, gridDim.y, t, ex);
    else slice_part<TB>(B, K, Kp, parts, (bid - na) / kblocks * 32, (bid - na) % kblocks * SK, b, gridDim.y, t, ex);
}

// the K range of a tile in chunks of 64 real terms of the slab (complex rows m0.., complex columns c0..)
__device__ __forceinline__ void tile_krange(const OzArgs &a, int m0, int c0, int &kb, int &ke)
{
    int kmin = 0, kmax = a.K;
    if (a.kmode == ZG_K_FROM_MAX_MN) kmin = max(kmin, max(m0, c0) - a.k0);
    else if (a.kmode == ZG_K_FROM_N0) kmin = max(kmin, c0 - a.k0);
    if (a.k_to_m_end) kmax = min(kmax, m0 + OPM - a.k0);
    kb = (2 * kmin) / OTK;
    ke = min(a.kchunks, (2 * max(kmax, 0) + OTK - 1) / OTK);
    if (ke < kb) ke = kb;
}

// pair tile t of the computed ones: batch b, row tile i, column tile j. With lower_only, row tile i holds column
// tiles 0 .. min(n_tn, 2 i + 2) - 1 (a column tile is 128 complex columns), i (i + 1) tiles above it.
__device__ __forceinline__ void tile_of(const OzArgs &a, int t, int &b, int &i, int &j)
{
    b = t / a.per;
    const int r = t - b * a.per;
    if (!a.lower_tiles) {
        // groups of 8 row tiles, all column tiles of a group before the next (the tiles in flight share panels in L2)
        const int per = 8 * a.n_tn, g = r / per, q = r - g * per, gm = min(8, a.n_tm - 8 * g);
        i = 8 * g + q % gm;
        j = q / gm;
    } else {
        i = (int)((sqrtf(4.f * (float)r + 1.f) - 1.f) * 0.5f);
        if ((i + 1) * (i + 2) <= r) ++i;
        if (i * (i + 1) > r) --i;
        j = r - i * (i + 1);
    }
}

// cut between groups: every group's sums come from one item
__host__ __device__ __forceinline__ bool whole_groups(int pieces) { return pieces == 1 || pieces == 2 || pieces == 4; }

// One work item: steps [lo, hi) of its tile's list of 28 * kc (pair, K chunk) steps
struct OzItem {
    int b, i, j, kb, kc, lo, hi;
    __device__ __forceinline__ OzItem(const OzArgs &a, int w)
    {
        const int t = w / a.pieces, p = w - t * a.pieces;
        tile_of(a, t, b, i, j);
        int ke;
        tile_krange(a, a.row0 + i * OPM, j * (OPN / 2), kb, ke);
        kc = a.lower_only && j > 2 * (a.row0 / OPM + i) + 1 ? 0 : ke - kb;
        lo = (int)((int64_t)NPAIR * kc * p / a.pieces);
        hi = (int)((int64_t)NPAIR * kc * (p + 1) / a.pieces);
    }
    // the end of the TMEM accumulation that starts at step l: steps of one group, at most UNITS units
    __device__ __forceinline__ int drain_end(int l) const
    {
        int q = l / kc, units = 0;
        const int g = kPairG[q];
        while (l < hi && q < NPAIR && kPairG[q] == g) {
            const int u = kPairU[q], r = min((q + 1) * kc, hi) - l, n = min(r, (UNITS - units) / u);
            l += n;
            units += n * u;
            if (n < r) break;
            ++q;
        }
        return l;
    }
};

// s 2^e rounded to nearest even once, for an integer s = t 2^32 + u below 2^100: integer operations only (the FP64
// pipe issues 2 operations a clock per SM)
__device__ __forceinline__ double round_sum(long long t, long long u, int e)
{
    unsigned long long lo = (unsigned long long)t << 32, hi = (unsigned long long)(t >> 32);
    lo += (unsigned long long)u;
    hi += (unsigned long long)(u >> 63) + (lo < (unsigned long long)u ? 1ull : 0ull);
    const bool neg = (long long)hi < 0;
    if (neg) {
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    if ((hi | lo) == 0ull) return 0.0;
    const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
    // the top 64 bits, what lies below them as a sticky bit
    unsigned long long top, rest;
    if (z >= 64) {
        top = lo << (z - 64);
        rest = 0ull;
    } else {
        top = z ? (hi << z) | (lo >> (64 - z)) : hi;
        rest = z ? lo << z : lo;
    }
    unsigned long long q = top >> 11;
    const unsigned long long low = (top & 0x7FFull) << 1 | (rest ? 1ull : 0ull);   // half is 0x800
    q += (low > 0x800ull || (low == 0x800ull && (q & 1ull))) ? 1ull : 0ull;
    // q in [2^52, 2^53]: the leading bit has weight 2^(127 - z + e)
    const int x = 127 - z + e + 1023;
    if (x >= 1 && x <= 2045) {
        const unsigned long long b = ((unsigned long long)(x - 1) << 52) + q;   // q's bit 52 (or 53) carries into x
        return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
    }
    const double d = ldexp((double)(long long)q, 127 - z + e - 52);
    return neg ? -d : d;
}

// the same from the group sums S_2 .. S_8. The common case, a sum of at least 64 bits, takes a third of the
// instructions of the general one: the magnitude as three words, a shift to the top, round to nearest even by one
// addition.
__device__ __forceinline__ double round_groups(const int (&s)[NGROUP], int e)
{
    const long long t = (long long)s[0] * 65536 + ((long long)s[1] * 256 + s[2]);
    const long long u = (long long)s[3] * 16777216 + ((long long)s[4] * 65536 + ((long long)s[5] * 256 + s[6]));
    long long h = t + (u >> 32);   // the sum is h 2^32 + l
    uint32_t l = (uint32_t)u;
    const bool neg = h < 0;
    if (neg) {
        h = ~h + (l == 0u ? 1 : 0);
        l = 0u - l;
    }
    const uint32_t h1 = (uint32_t)(h >> 32), h0 = (uint32_t)h;
    const int z = __clz((int)h1);
    const uint32_t w1 = __funnelshift_l(h0, h1, z), w0 = __funnelshift_l(l, h0, z), rest = l << (z & 31);
    const int x = 95 - z + e + 1023;   // biased exponent of the leading bit (bit 95 - z of the 96)
    if (h1 == 0u || x < 1 || x > 2044 || w1 == 0xFFFFFFFFu) return round_sum(t, u, e);
    const unsigned long long m = ((unsigned long long)w1 << 32 | w0) + (0x3FFu + ((w0 >> 11 & 1u) | (rest ? 1u : 0u)));
    const unsigned long long b = ((unsigned long long)(x - 1) << 52) + (m >> 11);
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// The group sums added from the leading one on, every partial sum rounded to FP64 (nearest even): the value of v <-
// fma(S_g, 2^(E - 8 g), v), g = 2 .. 8, in integers (14 FP64 instructions an output are 2.5 ms of a plan update at N_mu
// = 4096). Products with ZGemm::stepwise are rounded this way, those of the update of ISDF_MIXED plans: the FP16 digits
// of M^-1 follow its last bits, and the mode's complex128 gradients follow the digits, so M^-1 keeps the bits that this
// order of additions has always given.
__device__ __forceinline__ double round_steps(const int (&s)[NGROUP], int e)
{
    long long m = (long long)s[0] * 65536 + ((long long)s[1] * 256 + s[2]);   // S_2 .. S_4: below 2^48, exact
    int k = 0;   // the partial sum is m 2^k, |m| <= 2^53; k > 0 only with |m| >= 2^52
#pragma unroll
    for (int g = 3; g < NGROUP; ++g) {
        const long long b = m * 256 + (s[g] >> k);                   // floor; k < 28
        const uint32_t lo = (uint32_t)b, rest = (uint32_t)s[g] & ((1u << k) - 1u);   // what lies below
        const int hi = (int)(b >> 32), drop = 11 - __clz(hi ^ (hi >> 31));           // bits beyond 53, at most 9
        m = b;
        if (drop > 0) {   // always when k > 0: b has 60 bits or more then
            const uint32_t odd = rest ? 1u : lo >> drop & 1u;        // a half is rounded up
            const long long u = b + (long long)((1u << (drop - 1)) - 1u + odd);
            m = (long long)((unsigned long long)(uint32_t)((int)(u >> 32) >> drop) << 32 |
                            __funnelshift_r((uint32_t)u, (uint32_t)(u >> 32), drop));
            k += drop;
        }
    }
    if (m == 0) return 0.0;
    const unsigned long long a = m < 0 ? 0ull - (unsigned long long)m : (unsigned long long)m;
    const int z = __clzll((long long)a), x = 63 - z + k + e + 1023;   // biased exponent of the leading bit
    if (x < 1 || x > 2046) return ldexp((double)m, k + e);
    return __longlong_as_double((long long)(((unsigned long long)(x - 1) << 52) + ((a << z) >> 11) | (m < 0 ? 0x8000000000000000ull : 0ull)));
}

// beta C + alpha v with the multiplications that change nothing left out
__device__ __forceinline__ double2 oz_result(const OzArgs &a, double2 v, const double2 *c)
{
    if (a.alpha == -1.0) v = make_double2(-v.x, -v.y);
    else if (a.alpha != 1.0) v = make_double2(a.alpha * v.x, a.alpha * v.y);
    if (a.beta) {
        const double2 o = *c;
        v = make_double2(o.x + v.x, o.y + v.y);
    }
    return v;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(OTHREADS, 1)
    oz_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, OzArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[OSTAGES];
    __shared__ __align__(8) uint64_t empty_bar[OSTAGES];
    __shared__ __align__(8) uint64_t peer_bar;    // leader: the peer's producer has finished (count below)
    __shared__ volatile int peer_issued;
    __shared__ __align__(8) uint64_t tfull[2];
    __shared__ __align__(8) uint64_t tempty[2];
    __shared__ __align__(8) uint64_t drain_bar;
    __shared__ __align__(8) uint64_t never_bar;   // signalled by nothing (the test hook waits on it)
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int failed;
    __shared__ uint32_t skip;

    const uint32_t rank = tc::cluster_rank();
    const bool leader = rank == 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t raw = tc::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sbase = smem_raw + (base - raw);
    const int n_pairs = gridDim.x >> 1, pair = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < OSTAGES; ++s) {
            tc::mbar_init(&full_bar[s], 1);
            tc::mbar_init(&empty_bar[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&tfull[i], 1);
            tc::mbar_init(&tempty[i], 2 * OEPI);
        }
        tc::mbar_init(&drain_bar, 1);
        tc::mbar_init(&never_bar, 1);
        tc::mbar_init(&peer_bar, 1);
        failed = 0;
        skip = *(volatile int *)a.err ? 1u : 0u;   // only the leader's reading is used
        tc::fence_barrier_init();
    }
    __syncthreads();
    tc::cluster_sync();   // both CTAs' barriers initialised before any remote arrive
    const bool run = tc::ld_shared_cluster(tc::map_shared(&skip, 0)) == 0u;
    if (warp == 0) tc::tmem_alloc_pair(&tmem_slot, 2 * OPN);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    const int n_work = run ? a.batch * a.per * a.pieces : 0;

    if (warp == 0) {
        if (lane == 0) {
            tc::prefetch_map(&ta);
            tc::prefetch_map(&tb);
            const uint32_t full0 = tc::map_shared(&full_bar[0], 0);   // the leader's full barriers
            int c = 0, issued = 0;
            for (int w = pair; w < n_work && !failed; w += n_pairs) {
                const OzItem it(a, w);
                const int ra = a.row0 + it.i * OPM + (int)rank * OTM, rb = it.j * OPN + (int)rank * OTM;
                for (int l = it.lo; l < it.hi && !failed;) {
                    const int q = l / it.kc, s = kPairS[q], t = kPairG[q] - s;
                    const int ya = (it.b * NSLICE + s - 1) * a.Ra + ra, yb = (it.b * NSLICE + t - 1) * a.Rb + rb;
                    const int l1 = min((q + 1) * it.kc, it.hi);
                    for (int kc = it.kb + l - q * it.kc; l < l1; ++l, ++kc, ++c) {
                        const int st = c % OSTAGES, use = c / OSTAGES;
                        if (!tc::mbar_wait(&empty_bar[st], (use & 1) ^ 1, a.budget)) {
                            atomicExch(a.err, 1);
                            failed = 1;
                            break;
                        }
                        if (leader) tc::mbar_expect_tx(&full_bar[st], 2 * OSTAGE);   // both CTAs' bytes
                        uint8_t *sp = sbase + st * OSTAGE;
                        const uint32_t fb = full0 + (uint32_t)(st * sizeof(uint64_t));
                        tc::tma_load_2d_pair(sp, &ta, fb, kc * OTK, ya);
                        tc::tma_load_2d_pair(sp + OTILE, &tb, fb, kc * OTK, yb);
                        issued = c + 1;
                    }
                }
            }
            // every copy of either CTA completes on a leader barrier: the leader drains them all before the pair
            // exits (the peer reports its count; stages only the peer loaded are armed for its bytes alone)
            if (!leader) {
                tc::st_shared_cluster(tc::map_shared((const void *)&peer_issued, 0), (uint32_t)issued);
                tc::mbar_arrive_cluster(tc::map_shared(&peer_bar, 0));
            } else {
                int hi = issued;
                if (tc::mbar_wait_cluster(&peer_bar, 0, OWAIT)) hi = max(hi, (int)peer_issued);
                for (int c2 = hi - OSTAGES > 0 ? hi - OSTAGES : 0; c2 < hi; ++c2) {
                    if (c2 >= issued) tc::mbar_expect_tx(&full_bar[c2 % OSTAGES], OSTAGE);
                    tc::mbar_wait(&full_bar[c2 % OSTAGES], (c2 / OSTAGES) & 1, OWAIT);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            constexpr uint32_t idesc = tc::idesc_f16(OPM, OPN);
            int c = 0, tl = 0;
            bool ok = true;
            if (a.never > 0 && !tc::mbar_wait(&never_bar, 0, a.never)) {
                atomicExch(a.err, 1);
                failed = 1;
                ok = false;
            }
            for (int w = pair; w < n_work && ok && !failed; w += n_pairs) {
                const OzItem it(a, w);
                for (int l = it.lo; l < it.hi && ok; ++tl) {
                    const int acc = tl & 1, use = tl >> 1, l0 = l, l1 = it.drain_end(l);
                    if (!tc::mbar_wait(&tempty[acc], (use & 1) ^ 1, a.budget)) {
                        atomicExch(a.err, 1);
                        failed = 1;
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    const uint32_t d = tmem + (uint32_t)acc * OPN;
                    for (; l < l1; ++l, ++c) {
                        const int st = c % OSTAGES, fu = c / OSTAGES;
                        if (!tc::mbar_wait(&full_bar[st], fu & 1, a.budget)) {
                            atomicExch(a.err, 1);
                            failed = 1;
                            ok = false;
                            break;
                        }
                        tc::fence_after();
                        const uint32_t sa = base + st * OSTAGE;
                        const uint64_t da = tc::desc_sw128(sa), db = tc::desc_sw128(sa + OTILE);
#pragma unroll
                        for (int kk = 0; kk < OTK / 16; ++kk)
                            tc::mma_f16_pair(d, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                                             (l > l0 || kk > 0) ? 1u : 0u);
                        tc::mma_commit_pair(&empty_bar[st], 0x3);
                    }
                    if (!ok) break;
                    tc::mma_commit_pair(&tfull[acc], 0x3);
                }
            }
            // no MMA of the pair may still be running when either CTA releases its TMEM
            tc::mma_commit_pair(&drain_bar, 0x1);
            tc::mbar_wait(&drain_bar, 0, OWAIT);
        }
        __syncwarp();
    } else {
        const int quarter = warp & 3;          // TMEM lane quarter this warp may access
        const int part = (warp - 2) >> 2;      // which 64 of the tile's 256 real columns
        const uint32_t tempty0 = tc::map_shared(&tempty[0], 0);
        const int rt = quarter * 32 + lane;    // row of this CTA's 128
        int tl = 0;
        bool ok = true;
        int acc32[OHC];
#pragma unroll
        for (int q = 0; q < OHC; ++q) acc32[q] = 0;
        for (int w = pair; w < n_work && ok && !failed; w += n_pairs) {
            const OzItem it(a, w);
            for (int l = it.lo; l < it.hi; ++tl) {
                const int accb = tl & 1, use = tl >> 1, g = kPairG[l / it.kc], l1 = it.drain_end(l);
                if (!tc::mbar_wait(&tfull[accb], use & 1, a.budget)) {
                    atomicExch(a.err, 1);
                    failed = 1;
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint32_t ta0 = tmem + (uint32_t)accb * OPN + ((uint32_t)(quarter * 32) << 16) + part * OHC;
#pragma unroll
                for (int j = 0; j < OHC / 16; ++j) {
                    uint32_t r[16];
                    tc::tmem_ld16(ta0 + 16 * j, r);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 16; ++q) acc32[16 * j + q] += __float2int_rn(__uint_as_float(r[q]));
                }
                tc::fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_cluster(tempty0 + (uint32_t)(accb * sizeof(uint64_t)));
                l = l1;
                if (l < it.hi && kPairG[l / it.kc] == g) continue;
                // the group (or this item's part of it) is complete
                const int64_t tile = ((int64_t)it.b * a.n_tm + it.i) * a.n_tn + it.j;
                int *gr = a.gsum + (tile * NGROUP + (g - 2)) * GTILE + (int64_t)rank * (OTM * OPN) +
                          (int64_t)(part * OHC) * OTM + rt;
                if (whole_groups(a.pieces)) {
#pragma unroll
                    for (int q = 0; q < OHC; ++q) gr[q * OTM] = acc32[q];
                } else {
#pragma unroll
                    for (int q = 0; q < OHC; ++q) atomicAdd(gr + q * OTM, acc32[q]);
                }
#pragma unroll
                for (int q = 0; q < OHC; ++q) acc32[q] = 0;
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::cluster_sync();   // both CTAs done with TMEM, shared memory and the remote barriers
    if (warp == 0) tc::tmem_dealloc_pair(tmem, 2 * OPN);
}

// FP64 result of a product from its group sums: one CTA of 32 x 8 threads per 32 rows x 32 complex columns.
// The sums are read along the rows of a column (the layout the GEMM writes coalesced), the result is transposed
// through shared memory and written along the columns of a row.
template <bool STEPWISE>
__global__ void __launch_bounds__(256) oz_combine(OzArgs a)
{
    __shared__ double2 tile[32][33];
    const int c0 = blockIdx.x * 32, rl = blockIdx.y * 32, r0 = a.row0 + rl, b = blockIdx.z;
    const int i = rl / OPM, j = c0 / (OPN / 2);
    if (a.lower_only && j > 2 * (r0 / OPM) + 1) return;   // tile not computed: C untouched
    int kb, ke;
    tile_krange(a, r0 / OPM * OPM, j * (OPN / 2), kb, ke);
    const int64_t gt = ((int64_t)b * a.n_tm + i) * a.n_tn + j;
    const int rin = rl % OPM + threadIdx.x, row = r0 + threadIdx.x;
    const int *gp = a.gsum + gt * NGROUP * GTILE + (int64_t)(rin / OTM) * (OTM * OPN) + rin % OTM;
    for (int q = threadIdx.y; q < 32; q += 8) {
        const int c = c0 + q;
        double2 v = make_double2(0.0, 0.0);
        if (kb < ke && row < a.M && c < a.N) {
            const int *p = gp + (int64_t)(2 * (c % (OPN / 2))) * OTM;
            int s[2][NGROUP];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int g = 0; g < NGROUP; ++g) s[h][g] = p[g * GTILE + h * OTM];
            const int e = a.ea[(int64_t)b * a.M + row] + a.eb[(int64_t)b * a.N + c] - 64;
            v = STEPWISE ? make_double2(round_steps(s[0], e), round_steps(s[1], e))
                         : make_double2(round_groups(s[0], e), round_groups(s[1], e));
        }
        tile[threadIdx.x][q] = v;
    }
    __syncthreads();
    for (int q = threadIdx.y; q < 32; q += 8) {
        const int r = r0 + q, c = c0 + (int)threadIdx.x;
        if (r >= a.M || c >= a.N) continue;
        double2 *cp = a.C + (int64_t)b * a.bsc + (int64_t)r * a.ldc + c;
        *cp = oz_result(a, tile[q][threadIdx.x], cp);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 oz_encode()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

bool oz_map(CUtensorMap *m, const void *base, uint64_t inner, uint64_t rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = oz_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {inner, rows};
    cuuint64_t strides[1] = {inner * 2};
    cuuint32_t box[2] = {OTK, OTM};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int oz_sms()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    }
    return n;
}

isdf_status oz_attributes()
{
    static bool done[64] = {false};
    int dev = 0;
    ISDF_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return ISDF_ERR_CUDA;
    if (done[dev]) return ISDF_OK;
    ISDF_CUDA_TRY(cudaFuncSetAttribute(oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, OSMEM));
    done[dev] = true;
    return ISDF_OK;
}

int64_t tiles_m(int64_t M) { return (M + OPM - 1) / OPM; }
int64_t tiles_n(int64_t N) { return (2 * N + OPN - 1) / OPN; }

// Work items per tile: the cut of its 28 * kchunks steps that ends first when the CTA pairs take the items in turn.
// Each item pays about 12 steps (512 clocks each) to fill the ring and to write its sums, and 12 more when groups are
// cut: atomic additions to sums cleared before.
int pieces_for(int64_t tiles, int kchunks, int pairs)
{
    const int64_t steps = (int64_t)NPAIR * kchunks;
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int p = 1; p <= 32 && steps / p >= 14; ++p) {
        const int64_t waves = (tiles * p + pairs - 1) / pairs;
        const int64_t c = waves * ((steps + p - 1) / p + (whole_groups(p) ? 12 : 24));
        if (c < cost) {
            cost = c;
            best = p;
        }
    }
    return best;
}

}  // namespace

size_t oz_gsum_ints(int M, int N, int batch) { return (size_t)batch * tiles_m(M) * tiles_n(N) * NGROUP * GTILE; }

size_t oz_chunk_ints(int M, int N)
{
    const int64_t tn = tiles_n(N), want = (2 * (oz_sms() / 2) + tn - 1) / tn, tm = tiles_m(M);
    return (size_t)(want < tm ? want : tm) * tn * NGROUP * GTILE;
}

bool oz_fits(const ZGemm &g, const OzWork &w)
{
    if (g.dual || g.ctype != ZG_C128 || g.scn != 1) return false;
    if (g.M < 1 || g.N < 1 || g.K < 1 || !w.sa || !w.sb || !w.ma || !w.mb) return false;
    const int batch = g.batch > 1 ? g.batch : 1;
    size_t ha, hb, ra, rb;
    oz_sizes(g.M, g.N, g.K, batch, &ha, &hb, &ra, &rb);
    if (ha > w.cap_a || hb > w.cap_b || ra > w.cap_ma || rb > w.cap_mb) return false;
    // all group sums at once, or (single products) at least those of one row of tiles
    return w.gsum && (oz_gsum_ints(g.M, g.N, batch) <= w.cap_g || (batch == 1 && oz_gsum_ints(OPM, g.N, 1) <= w.cap_g));
}

isdf_status oz_zgemm(const ZGemm &g, const OzWork &w, int *err, cudaStream_t st)
{
    if (!oz_fits(g, w) || !err) return ISDF_ERR_INVALID_ARG;
    ISDF_TRY(oz_attributes());
    const int batch = g.batch > 1 ? g.batch : 1;
    const int slab = oz_slab(g.K);
    const int64_t Ra = oz_round_up(g.M, OTM), Rb = oz_round_up(2 * (int64_t)g.N, OTM);
    // rows whose group sums fit at a time: all of them, or whole row tiles
    const bool all = oz_gsum_ints(g.M, g.N, batch) <= w.cap_g;
    const int chunk = all ? g.M : (int)(w.cap_g / oz_gsum_ints(OPM, g.N, 1)) * OPM;
    const size_t ea = g.A1.type == ZG_C64 ? 8 : 16, eb = g.B1.type == ZG_C64 ? 8 : 16;
    for (int k0 = 0; k0 < g.K; k0 += slab) {
        const int K = g.K - k0 < slab ? g.K - k0 : slab;
        const int64_t Kp = oz_round_up(2 * (int64_t)K, OTK);
        const char *pa = static_cast<const char *>(g.A1.p) + (int64_t)k0 * g.A1.s1 * (int64_t)ea;
        const char *pb = static_cast<const char *>(g.B1.p) + (int64_t)k0 * g.B1.s0 * (int64_t)eb;
        const int pairs = oz_sms() / 2, crow = g.M < chunk ? g.M : chunk;
        OzArgs a;
        a.n_tm = (int)tiles_m(crow);
        a.n_tn = (int)tiles_n(g.N);
        a.per = a.n_tm * a.n_tn;
        a.lower_only = g.lower_only;
        a.lower_tiles = g.lower_only && all;   // only the tiles on or below the diagonal are listed
        if (a.lower_tiles) {   // sum over the row tiles of min(n_tn, 2 i + 2)
            a.per = 0;
            for (int i = 0; i < a.n_tm; ++i) a.per += 2 * i + 2 < a.n_tn ? 2 * i + 2 : a.n_tn;
        }
        a.kchunks = (int)(Kp / OTK);
        a.pieces = pieces_for((int64_t)batch * a.per, a.kchunks, pairs);
        if (crow < g.M && !whole_groups(a.pieces)) a.pieces = 4;   // the sums are cleared once, before the first chunk
        // A role: rows m, entries A[m s0 + k s1]; B role: rows n, entries B[k s0 + n s1], x = conj(op(B))
        const int parts = (K + PK - 1) / PK;
        OzOperand oa{pa, g.A1.s0, g.A1.s1, g.bsa, g.M, (int)Ra, g.A1.conj, 0, nullptr, w.ma, w.sa};
        OzOperand ob{pb, g.B1.s1, g.B1.s0, g.bsb, g.N, (int)Rb, !g.B1.conj, 1, nullptr, w.mb, w.sb};
        oa.part = reinterpret_cast<unsigned int *>(w.ma + (size_t)batch * g.M);
        ob.part = reinterpret_cast<unsigned int *>(w.mb + (size_t)batch * g.N);
        const int64_t nz = !whole_groups(a.pieces) ? (int64_t)oz_gsum_ints(g.M, g.N, batch) / 4 : 0;   // int4s of group sums to clear
        const int64_t zb = nz ? (nz + 4 * 256 - 1) / (4 * 256) : 0;
        const dim3 gm((unsigned)(((g.M + 31) / 32 + (g.N + 31) / 32) * parts + (zb < 1024 ? zb : 1024)), batch);
        const int64_t kblocks = (Kp / 2 + SK - 1) / SK;
        const dim3 gs((unsigned)((Ra / 32 + Rb / 64) * kblocks), batch);
        auto prepare = [&](auto max_kernel, auto slice_kernel) {
            max_kernel<<<gm, 256, 0, st>>>(oa, ob, K, parts, err, reinterpret_cast<int4 *>(w.gsum), nz);
            isdf_note_launch();
            slice_kernel<<<gs, 256, 0, st>>>(oa, ob, K, Kp, parts);
            isdf_note_launch();
        };
        if (g.A1.type == ZG_C64 && g.B1.type == ZG_C64) prepare(oz_rowmax<float2, float2>, oz_slice<float2, float2>);
        else if (g.A1.type == ZG_C64) prepare(oz_rowmax<float2, double2>, oz_slice<float2, double2>);
        else if (g.B1.type == ZG_C64) prepare(oz_rowmax<double2, float2>, oz_slice<double2, float2>);
        else prepare(oz_rowmax<double2, double2>, oz_slice<double2, double2>);
        ISDF_LAUNCH_CHECK();
        CUtensorMap ta, tb;
        if (!oz_map(&ta, w.sa, (uint64_t)Kp, (uint64_t)batch * NSLICE * Ra) ||
            !oz_map(&tb, w.sb, (uint64_t)Kp, (uint64_t)batch * NSLICE * Rb))
            return ISDF_ERR_CUDA;
        a.M = g.M;
        a.N = g.N;
        a.K = K;
        a.k0 = k0;
        a.Ra = (int)Ra;
        a.Rb = (int)Rb;
        a.batch = batch;
        a.kmode = g.kmode;
        a.k_to_m_end = g.k_to_m_end;
        a.beta = k0 > 0 ? 1 : g.beta;
        a.alpha = g.alpha;
        a.C = static_cast<double2 *>(g.C);
        a.ldc = g.scm;
        a.bsc = g.bsc;
        a.ea = w.ma;
        a.eb = w.mb;
        a.err = err;
        a.budget = w.wait_budget > 0 ? w.wait_budget : OWAIT;
        a.never = w.wait_budget < 0 ? -w.wait_budget : 0;
        a.gsum = w.gsum;
        for (a.row0 = 0; a.row0 < g.M; a.row0 += crow) {
            const int rows = g.M - a.row0 < crow ? g.M - a.row0 : crow;
            if (!a.lower_tiles) {
                a.n_tm = (int)tiles_m(rows);
                a.per = a.n_tm * a.n_tn;
            }
            const int64_t work = (int64_t)batch * a.per * a.pieces;
            oz_gemm<<<(unsigned)(2 * (work < pairs ? work : pairs)), OTHREADS, OSMEM, st>>>(ta, tb, a);
            isdf_note_launch();
            const dim3 gc((g.N + 31) / 32, (rows + 31) / 32, batch), bc(32, 8);
            if (g.stepwise) oz_combine<true><<<gc, bc, 0, st>>>(a);
            else oz_combine<false><<<gc, bc, 0, st>>>(a);
            isdf_note_launch();
        }
        ISDF_LAUNCH_CHECK();
    }
    return ISDF_OK;
}
