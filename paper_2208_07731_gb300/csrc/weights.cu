// Step 1: the K-means weight function (Sec. 2.2, Eq. weight function 2 for
// SSM and its alpha family, Eq. weight function for PSM).
//
// Every sum of the weight is the exact sum of its terms rounded once, so the
// result does not depend on summation order (and equals the oracle bit for
// bit). For alpha = 2 the terms are the exact squares x^2 of the real
// components x = Re z, Im z: with E = max floor(log2|x|) over the row's
// non-zero components,
//     sum = RN( sum_x floor(x^2 2^(110 - 2E)) ) 2^(2E - 110),
// where x = m 2^p (integer mantissa m, exponent p of its format) makes each
// term the integer m^2 shifted by 2p + 110 - 2E, accumulated in 128 bits with
// integer instructions only. For alpha != 2 the terms are |z|^alpha in FP64
// and the same exact summation runs on floor(t 2^(110 - E_t)).
//
// One warp owns one grid row. Rows of at most 512 complex64 or 256 complex128
// columns a set, 16-byte aligned, are read once into registers (weights_rows);
// others twice: pass 1 reads the row and reduces the exponent window E, pass 2
// reads it again (from L1/L2: the row was just read) and accumulates. The lane
// sums are added across the warp by 26-bit limbs and rounded once by integer
// operations: GB300 runs an FP64 warp instruction in 64 clocks of an SM quarter,
// so FP64 is kept out of the row loop altogether.
//
// Complex64 rows take a shorter integer path. A float component x = m 2^p
// (p = max(b, 1) - 150 for the biased exponent b) has the term
// floor((m 2^k)^2) with k = p + 55 - E. Whenever k >= 0 (every normal
// component within 2^32 of the row maximum) y = m 2^k is an integer below
// 2^56, and with y = yh 2^28 + yl,
//     y^2 = yh^2 2^56 + yh yl 2^29 + yl^2,
// three products below 2^56 that each lane sums in plain 64-bit registers
// (128 of them stay below 2^63) and folds into its 128-bit sum every 128
// terms. Pass 1 finds the smallest magnitude of the row as well as the
// largest; a row whose components are all normal with k >= 0 runs a loop
// without branches (k <= 32 there, so yh and yl are two clamped funnel
// shifts of m 2^4), any other row checks each component and gives zeros,
// subnormals and components with k < 0 (whose term is floored) the general
// formula. The integer sum, hence the weight, is the same either way. Pass 1
// marks the row's L2 lines evict-last and pass 2 evict-first, so that the
// second read finds them in L2.

#include "common.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kNoExp = -0x40000000;   // no non-zero component seen

struct U128 {
    unsigned long long lo, hi;
};

// L2 eviction priorities for the two reads of a row: the first read marks its lines evict-last so
// that they are still in L2 for the second, which marks them evict-first
__device__ __forceinline__ unsigned long long l2_evict_last()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ unsigned long long l2_evict_first()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint4 ld_policy(const uint4 *p, unsigned long long pol)
{
    uint4 r;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p), "l"(pol));
    return r;
}

__device__ __forceinline__ void add_u128(U128 &a, unsigned long long lo, unsigned long long hi)
{
    const unsigned long long l = a.lo + lo;
    a.hi += hi + (l < lo ? 1ull : 0ull);
    a.lo = l;
}

// a += floor((vhi:vlo) 2^sh) for sh <= 63
__device__ __forceinline__ void add_shifted128(U128 &a, unsigned long long vlo, unsigned long long vhi, int sh)
{
    if (sh >= 0) {
        if (sh == 0) add_u128(a, vlo, vhi);
        else add_u128(a, vlo << sh, (vhi << sh) | (vlo >> (64 - sh)));
    } else {
        const int t = -sh;
        if (t < 64) add_u128(a, (vlo >> t) | (vhi << (64 - t)), vhi >> t);
        else if (t < 128) add_u128(a, vhi >> (t - 64), 0ull);
    }
}

// floor(log2|x|) and the integer form |x| = m 2^p of a float / a double (x != 0)
__device__ __forceinline__ int exp_of(uint32_t u)
{
    const int b = (int)((u >> 23) & 0xFF);
    const uint32_t f = u & 0x7FFFFFu;
    if (b) return b - 127;
    return f ? (31 - __clz((int)f)) - 149 : kNoExp;
}
__device__ __forceinline__ int exp_of(unsigned long long u)
{
    const int b = (int)((u >> 52) & 0x7FF);
    const unsigned long long f = u & 0xFFFFFFFFFFFFFull;
    if (b) return b - 1023;
    return f ? (63 - __clzll((long long)f)) - 1074 : kNoExp;
}

// the term floor(x^2 2^(110 - 2E)) of one component, added to a
__device__ __forceinline__ void add_square(U128 &a, unsigned long long u, int E)
{
    const int b = (int)((u >> 52) & 0x7FF);
    const unsigned long long f = u & 0xFFFFFFFFFFFFFull;
    if (!b && !f) return;
    const unsigned long long m = b ? (f | (1ull << 52)) : f;
    const int p = b ? b - 1075 : -1074;
    add_shifted128(a, m * m, __umul64hi(m, m), 2 * p + 110 - 2 * E);     // m^2 < 2^106, shift <= 6
}

// round-to-nearest-even of a 128-bit integer, times 2^scale
__device__ __forceinline__ double u128_scaled(U128 a, int scale)
{
    const int n = a.hi ? __clzll((long long)a.hi) : 64 + __clzll((long long)a.lo);
    const int x = 127 - n + scale + 1023;   // biased exponent of the leading bit
    if (n < 128 && x >= 1 && x <= 2045) {   // a normal result: integer operations only
        const unsigned long long top = n >= 64 ? a.lo << (n - 64) : n ? (a.hi << n) | (a.lo >> (64 - n)) : a.hi;
        const unsigned long long rest = n >= 64 ? 0ull : n ? a.lo << n : a.lo;
        const unsigned long long low = (top & 0x7FFull) << 1 | (rest ? 1ull : 0ull);   // half is 0x800
        unsigned long long q = top >> 11;
        q += (low > 0x800ull || (low == 0x800ull && (q & 1ull))) ? 1ull : 0ull;
        return __longlong_as_double((long long)(((unsigned long long)(x - 1) << 52) + q));
    }
    double d;
    if (a.hi == 0ull) {
        d = __ull2double_rn(a.lo);
    } else {
        unsigned long long top = n ? ((a.hi << n) | (a.lo >> (64 - n))) : a.hi;
        if (a.lo << n) top |= 1ull;   // sticky: the bits below top decide ties
        d = ldexp(__ull2double_rn(top), 64 - n);
    }
    return ldexp(d, scale);
}

// the sum over the warp (below 2^128), valid in every lane: five 26-bit limbs, each summed by one warp reduction
__device__ __forceinline__ U128 warp_sum(U128 v)
{
    constexpr unsigned int m = (1u << 26) - 1u;
    const unsigned long long l0 = __reduce_add_sync(0xffffffffu, (unsigned int)v.lo & m);
    const unsigned long long l1 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.lo >> 26) & m);
    const unsigned long long l2 = __reduce_add_sync(0xffffffffu, (unsigned int)((v.lo >> 52) | (v.hi << 12)) & m);
    const unsigned long long l3 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.hi >> 14) & m);
    const unsigned long long l4 = __reduce_add_sync(0xffffffffu, (unsigned int)(v.hi >> 40) & m);   // 24 bits
    U128 r{l0, 0ull};
    add_u128(r, l1 << 26, l1 >> 38);
    add_u128(r, l2 << 52, l2 >> 12);
    r.hi += (l3 << 14) + (l4 << 40);
    return r;
}

// The component bits of one complex128 orbital row, visited by the lanes of a warp
template <typename F>
__device__ __forceinline__ void for_components(const double2 *row, int n, int lane, F &&fn)
{
    const ulonglong2 *v = reinterpret_cast<const ulonglong2 *>(row);
#pragma unroll 4
    for (int i = lane; i < n; i += 32) {
        const ulonglong2 q = __ldg(v + i);
        fn(q.x);
        fn(q.y);
    }
}

// floor(log2 max |x|) over a row's components from the largest magnitude bit pattern (the bit
// patterns of non-negative floats / doubles order like their values), kNoExp for an all-zero row
__device__ __forceinline__ int exp_of_max(uint32_t m) { return m ? exp_of(m) : kNoExp; }
__device__ __forceinline__ int exp_of_max(unsigned long long m) { return m ? exp_of(m) : kNoExp; }

__device__ __forceinline__ int row_exp(const double2 *row, int n, int lane)
{
    unsigned long long m = 0;
    for_components(row, n, lane, [&](unsigned long long u) { m = max(m, u & 0x7FFFFFFFFFFFFFFFull); });
    return __reduce_max_sync(0xffffffffu, exp_of_max(m));
}

// The complex64 terms of one lane between two folds: sums of yh^2, yh yl, yl^2 and of the floored
// terms (each below 2^46)
struct Sq64 {
    unsigned long long a2, a1, a0, as;
};

__device__ __forceinline__ void add_y(Sq64 &q, uint32_t m, int k)   // y = m 2^k < 2^56
{
    const unsigned long long y = (unsigned long long)m << k;
    const uint32_t yh = (uint32_t)(y >> 28), yl = (uint32_t)y & 0xFFFFFFFu;
    q.a2 += (unsigned long long)yh * yh;
    q.a1 += (unsigned long long)yh * yl;
    q.a0 += (unsigned long long)yl * yl;
}

// one component: k = max(b, 1) - 95 - E; zeros, subnormals and components far below the row maximum
// (k < 0: the term is floor(m^2 2^(2k)), m^2 < 2^48) leave the common branch
__device__ __forceinline__ void add_square_c64(Sq64 &q, uint32_t u, int kbase)
{
    const int b = (int)((u >> 23) & 0xFFu);
    uint32_t m = (u | 0x800000u) & 0xFFFFFFu;
    int k = b + kbase;
    if (b == 0 || k < 0) {
        if (b == 0) {
            m = u & 0x7FFFFFu;
            k = 1 + kbase;
        }
        if (k < 0) {
            if (k > -24) q.as += ((unsigned long long)m * m) >> (-2 * k);
            return;
        }
    }
    add_y(q, m, k);
}

__device__ __forceinline__ void fold(U128 &a, Sq64 &q)
{
    add_u128(a, q.a2 << 56, q.a2 >> 8);
    add_u128(a, q.a1 << 29, q.a1 >> 35);
    add_u128(a, q.a0, 0ull);
    add_u128(a, q.as, 0ull);
    q = Sq64{0ull, 0ull, 0ull, 0ull};
}

// A normal component with k = b - 95 - E >= 0 (then k <= 32, since y = m 2^k < 2^56 and m >= 2^23):
// yh and yl come from m 2^4 < 2^28 by two clamped funnel shifts, without a branch.
__device__ __forceinline__ void add_normal_c64(Sq64 &q, uint32_t u, int kbase)
{
    const uint32_t m4 = ((u << 4) & 0x7FFFFF0u) | 0x8000000u;
    const unsigned k = (unsigned)((int)((u >> 23) & 0xFFu) + kbase);
    const uint32_t yh = __funnelshift_lc(m4, 0u, k);        // floor(m 2^(k - 28))
    const uint32_t yl = __funnelshift_lc(0u, m4, k) >> 4;   // (m 2^k) mod 2^28
    q.a2 += (unsigned long long)yh * yh;
    q.a1 += (unsigned long long)yh * yl;
    q.a0 += (unsigned long long)yl * yl;
}

// The terms of one complex64 row in the window E, added to a; every lane folds after at most 128 terms.
// NORMAL: every component of the row is normal and within 2^32 of the maximum (checked by the caller).
template <bool NORMAL>
__device__ __forceinline__ void row_squares_c64(const float2 *row, int n, int lane, int E, U128 &a,
                                                unsigned long long pol)
{
    const int kbase = -95 - E;
    Sq64 q{0ull, 0ull, 0ull, 0ull};
    auto add = [&](uint32_t u) {
        if (NORMAL) add_normal_c64(q, u, kbase);
        else add_square_c64(q, u, kbase);
    };
    if ((reinterpret_cast<uintptr_t>(row) & 15) == 0) {
        const uint4 *v = reinterpret_cast<const uint4 *>(row);
        const int n2 = n >> 1;
        for (int c0 = 0; c0 < n2; c0 += 32 * 32) {
            const int c1 = min(n2, c0 + 32 * 32);
#pragma unroll 4
            for (int i = c0 + lane; i < c1; i += 32) {
                const uint4 t = ld_policy(v + i, pol);
                add(t.x);
                add(t.y);
                add(t.z);
                add(t.w);
            }
            fold(a, q);
        }
        if ((n & 1) && lane == 0) {
            const uint2 t = __ldg(reinterpret_cast<const uint2 *>(row) + (n - 1));
            add(t.x);
            add(t.y);
            fold(a, q);
        }
    } else {
        for (int c0 = 0; c0 < n; c0 += 64 * 32) {
            const int c1 = min(n, c0 + 64 * 32);
            for (int i = c0 + lane; i < c1; i += 32) {
                const uint2 t = __ldg(reinterpret_cast<const uint2 *>(row) + i);
                add(t.x);
                add(t.y);
            }
            fold(a, q);
        }
    }
}

// The largest and smallest component magnitudes of a complex64 row as bit patterns (lane-local; the
// caller reduces them over the warp)
__device__ __forceinline__ void row_range_c64(const float2 *row, int n, int lane, unsigned long long pol,
                                              uint32_t &mx, uint32_t &mn)
{
    auto see = [&](uint32_t u) {
        const uint32_t v = u & 0x7FFFFFFFu;
        mx = max(mx, v);
        mn = min(mn, v);
    };
    if ((reinterpret_cast<uintptr_t>(row) & 15) == 0) {
        const uint4 *v = reinterpret_cast<const uint4 *>(row);
        const int n2 = n >> 1;
#pragma unroll 4
        for (int i = lane; i < n2; i += 32) {
            const uint4 q = ld_policy(v + i, pol);
            see(q.x);
            see(q.y);
            see(q.z);
            see(q.w);
        }
        if ((n & 1) && lane == 0) {
            const uint2 q = __ldg(reinterpret_cast<const uint2 *>(row) + (n - 1));
            see(q.x);
            see(q.y);
        }
    } else {
        for (int i = lane; i < n; i += 32) {
            const uint2 q = __ldg(reinterpret_cast<const uint2 *>(row) + i);
            see(q.x);
            see(q.y);
        }
    }
}

// row window E and whether the row takes the branch-free path: the smallest magnitude is a normal
// number with k = b_min - 95 - E >= 0
__device__ __forceinline__ bool all_normal(uint32_t mn, int E) { return (int)(mn >> 23) >= max(1, 95 + E); }

template <bool NORMAL>
__device__ __forceinline__ void row_pair_c64(const float2 *a, int na, const float2 *b, int nb, int lane, int E,
                                             bool both, U128 &s, unsigned long long pol)
{
    row_squares_c64<NORMAL>(a, na, lane, E, s, pol);
    if (both) row_squares_c64<NORMAL>(b, nb, lane, E, s, pol);
}

// alpha = 2 on complex64 rows: SSM (one window over both sets) or PSM (one per set, multiplied)
__global__ void __launch_bounds__(kThreads, 4) weights_squares_c64(const float2 *__restrict__ phi, int64_t ld_phi,
                                                                int n_phi, const float2 *__restrict__ psi,
                                                                int64_t ld_psi, int n_psi, int64_t n_r, int psm,
                                                                double *__restrict__ w, int acc)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned long long keep = l2_evict_last(), drop = l2_evict_first();
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n_r; r += nw) {
        const float2 *a = phi + r * ld_phi, *b = psi + r * ld_psi;
        uint32_t mxa = 0u, mna = 0xFFFFFFFFu, mxb = 0u, mnb = 0xFFFFFFFFu;
        row_range_c64(a, n_phi, lane, keep, mxa, mna);
        row_range_c64(b, n_psi, lane, keep, mxb, mnb);
        mxa = __reduce_max_sync(0xffffffffu, mxa);
        mna = __reduce_min_sync(0xffffffffu, mna);
        mxb = __reduce_max_sync(0xffffffffu, mxb);
        mnb = __reduce_min_sync(0xffffffffu, mnb);
        const int ea = exp_of_max(mxa), eb = exp_of_max(mxb);
        double v;
        if (!psm) {
            const int E = max(ea, eb);
            U128 s{0ull, 0ull};
            if (E != kNoExp) {
                if (all_normal(min(mna, mnb), E)) row_pair_c64<true>(a, n_phi, b, n_psi, lane, E, true, s, drop);
                else row_pair_c64<false>(a, n_phi, b, n_psi, lane, E, true, s, drop);
            }
            s = warp_sum(s);
            v = E == kNoExp ? 0.0 : u128_scaled(s, 2 * E - 110);
        } else {
            U128 sa{0ull, 0ull}, sb{0ull, 0ull};
            if (ea != kNoExp) {
                if (all_normal(mna, ea)) row_pair_c64<true>(a, n_phi, b, n_psi, lane, ea, false, sa, drop);
                else row_pair_c64<false>(a, n_phi, b, n_psi, lane, ea, false, sa, drop);
            }
            if (eb != kNoExp) {
                if (all_normal(mnb, eb)) row_pair_c64<true>(b, n_psi, a, n_phi, lane, eb, false, sb, drop);
                else row_pair_c64<false>(b, n_psi, a, n_phi, lane, eb, false, sb, drop);
            }
            sa = warp_sum(sa);
            sb = warp_sum(sb);
            const double xa = ea == kNoExp ? 0.0 : u128_scaled(sa, 2 * ea - 110);
            const double xb = eb == kNoExp ? 0.0 : u128_scaled(sb, 2 * eb - 110);
            v = __dmul_rn(xa, xb);
        }
        if (lane == 0) w[r] = acc ? __dadd_rn(w[r], v) : v;   // shared weight of several pairs: one rounding per pair
    }
}

// alpha = 2 on complex128 rows: SSM (one window over both sets) or PSM (one per set, multiplied)
__global__ void __launch_bounds__(kThreads) weights_squares_c128(const double2 *__restrict__ phi, int64_t ld_phi,
                                                                 int n_phi, const double2 *__restrict__ psi,
                                                                 int64_t ld_psi, int n_psi, int64_t n_r, int psm,
                                                                 double *__restrict__ w, int acc)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    auto squares = [&](const double2 *row, int n, int E, U128 &s) {
        for_components(row, n, lane, [&](unsigned long long u) { add_square(s, u, E); });
    };
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n_r; r += nw) {
        const double2 *a = phi + r * ld_phi, *b = psi + r * ld_psi;
        const int ea = row_exp(a, n_phi, lane), eb = row_exp(b, n_psi, lane);
        double v;
        if (!psm) {
            const int E = max(ea, eb);
            U128 s{0ull, 0ull};
            if (E != kNoExp) {
                squares(a, n_phi, E, s);
                squares(b, n_psi, E, s);
            }
            s = warp_sum(s);
            v = E == kNoExp ? 0.0 : u128_scaled(s, 2 * E - 110);
        } else {
            U128 sa{0ull, 0ull}, sb{0ull, 0ull};
            if (ea != kNoExp) squares(a, n_phi, ea, sa);
            if (eb != kNoExp) squares(b, n_psi, eb, sb);
            sa = warp_sum(sa);
            sb = warp_sum(sb);
            const double xa = ea == kNoExp ? 0.0 : u128_scaled(sa, 2 * ea - 110);
            const double xb = eb == kNoExp ? 0.0 : u128_scaled(sb, 2 * eb - 110);
            v = __dmul_rn(xa, xb);
        }
        if (lane == 0) w[r] = acc ? __dadd_rn(w[r], v) : v;
    }
}

// ---- rows held in registers: NV 16-byte pieces per lane and set (two complex64 or one complex128 each)
// The complex64 kernel above reads a row twice (the second time from L2) and spends a fifth of its issue slots and, at
// rows of a few hundred columns, most of the FP64 pipe on the end of a row. 96^3 rows of 2 x 256 complex64: 1.13 ->
// 0.97 ms (3.75 TB/s, ALU pipe 57 %, issue 56 %); 48^3 rows of 2 x 128 complex128: 258 -> 139 us (the general 128-bit
// shifts of the terms were the most of it).
//
// Bound by the ALU pipe (2 clocks a warp instruction; shifts, masks, min and max), so what multiplications can do runs
// on the FMA pipe: a shift by a constant is a product (low or high half) with a power of two that is a kernel argument,
// or the compiler would turn it back into a shift; exponents are compared two at a time (16-bit min and max).
struct Pow2 {
    uint32_t p1, p4, p8, p28;   // 2^1, 2^4, 2^8, 2^28
};

template <typename T> struct Piece;
template <> struct Piece<float2> {
    static constexpr int kComplex = 2;
    // upper halves of the magnitudes (exponent, 7 bits of the mantissa), packed largest and smallest
    __device__ static void range(uint4 q, uint32_t &mx, uint32_t &mn)
    {
        const uint32_t a = __byte_perm(q.x, q.y, 0x7632) & 0x7FFF7FFFu, b = __byte_perm(q.z, q.w, 0x7632) & 0x7FFF7FFFu;
        mx = __vmaxu2(mx, __vmaxu2(a, b));
        mn = __vminu2(mn, __vminu2(a, b));
    }
    // the window's exponent; -1000 when no component is normal (the general formula then looks at all bits)
    __device__ static int exponent(uint32_t mx)
    {
        const int e = (int)(max(mx >> 16, mx & 0xFFFFu) >> 7);
        return e ? e - 127 : -1000;
    }
    __device__ static bool plain(uint32_t mn, int E) { return (int)(min(mn >> 16, mn & 0xFFFFu) >> 7) >= max(1, 95 + E); }
    __device__ static int exact_exponent(uint4 q)
    {
        return exp_of_max(max(max(q.x & 0x7FFFFFFFu, q.y & 0x7FFFFFFFu), max(q.z & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu)));
    }
    // add_normal_c64 with its constant shifts as products
    __device__ static void add_plain(Sq64 &q, uint32_t u, int kbase, const Pow2 &c)
    {
        const uint32_t m4 = ((u * c.p4) & 0x7FFFFF0u) | 0x8000000u;
        uint32_t k, yl;
        asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(k) : "r"(u * c.p1), "r"(c.p8), "r"((uint32_t)kbase));   // b + kbase
        const uint32_t yh = __funnelshift_lc(m4, 0u, k);
        asm("mul.hi.u32 %0, %1, %2;" : "=r"(yl) : "r"(__funnelshift_lc(0u, m4, k)), "r"(c.p28));        // >> 4
        q.a2 += (unsigned long long)yh * yh;
        q.a1 += (unsigned long long)yh * yl;
        q.a0 += (unsigned long long)yl * yl;
    }
    template <bool PLAIN, int NV>
    __device__ static void squares(const uint4 (&v)[NV], int pieces, int lane, int E, U128 &s, const Pow2 &c)
    {
        static_assert(4 * NV <= 128, "lane sums of 128 terms");
        Sq64 q{0ull, 0ull, 0ull, 0ull};
        const int kbase = -95 - E;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (lane + 32 * i >= pieces) continue;
            const uint32_t u[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (PLAIN) add_plain(q, u[j], kbase, c);
                else add_square_c64(q, u[j], kbase);
            }
        }
        fold(s, q);
    }
};
template <> struct Piece<double2> {
    static constexpr int kComplex = 1;
    // upper 16 bits of the magnitudes (exponent, 4 bits of the mantissa)
    __device__ static void range(uint4 q, uint32_t &mx, uint32_t &mn)
    {
        const uint32_t a = __byte_perm(q.y, q.w, 0x7632) & 0x7FFF7FFFu;
        mx = __vmaxu2(mx, a);
        mn = __vminu2(mn, a);
    }
    __device__ static int exponent(uint32_t mx)
    {
        const int e = (int)(max(mx >> 16, mx & 0xFFFFu) >> 4);
        return e ? e - 1023 : -10000;
    }
    // normal components within 2^15 of the largest
    __device__ static bool plain(uint32_t mn, int E)
    {
        return (int)(min(mn >> 16, mn & 0xFFFFu) >> 4) >= max(1, E + 1023 - 15);
    }
    __device__ static int exact_exponent(uint4 q)
    {
        const unsigned long long a = (unsigned long long)(q.y & 0x7FFFFFFFu) << 32 | q.x, b = (unsigned long long)(q.w & 0x7FFFFFFFu) << 32 | q.z;
        return exp_of_max(max(a, b));
    }
    // floor(x^2 2^(110 - 2E)) of a normal x = m 2^(e - 52) with t = 2 (E - e) <= 30: (8 m)^2 2^-t, (8 m)^2 < 2^112
    __device__ static void add_plain(U128 &s, uint32_t lo, uint32_t hi, int E)
    {
        const int t = 2 * (E + 1023 - (int)((hi >> 20) & 0x7FFu));
        const uint32_t y0 = lo << 3, y1 = __funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, 3);   // 8 m < 2^56
        const unsigned long long p0 = (unsigned long long)y0 * y0, p1 = (unsigned long long)y0 * y1,
                                 p2 = (unsigned long long)y1 * y1;
        const unsigned long long l = p0 + (p1 << 33), h = p2 + (p1 >> 31) + (l < p0 ? 1ull : 0ull);
        const uint32_t w0 = (uint32_t)l, w1 = (uint32_t)(l >> 32), w2 = (uint32_t)h, w3 = (uint32_t)(h >> 32);
        const unsigned long long rl = (unsigned long long)__funnelshift_r(w0, w1, t) | (unsigned long long)__funnelshift_r(w1, w2, t) << 32;
        const unsigned long long rh = (unsigned long long)__funnelshift_r(w2, w3, t) | (unsigned long long)(w3 >> t) << 32;
        add_u128(s, rl, rh);
    }
    template <bool PLAIN, int NV>
    __device__ static void squares(const uint4 (&v)[NV], int pieces, int lane, int E, U128 &s, const Pow2 &)
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (lane + 32 * i >= pieces) continue;
            if (PLAIN) {
                add_plain(s, v[i].x, v[i].y, E);
                add_plain(s, v[i].z, v[i].w, E);
            } else {
                add_square(s, (unsigned long long)v[i].y << 32 | v[i].x, E);
                add_square(s, (unsigned long long)v[i].w << 32 | v[i].z, E);
            }
        }
    }
};

template <typename T, int NV>
__global__ void __launch_bounds__(kThreads, NV > 4 ? 2 : 4) weights_rows(const T *__restrict__ phi, int64_t ld_phi, int n_phi,
                                                                         const T *__restrict__ psi, int64_t ld_psi, int n_psi,
                                                                         int64_t n_r, int psm, double *__restrict__ w, int acc, Pow2 c)
{
    using P = Piece<T>;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int np[2] = {n_phi / P::kComplex, n_psi / P::kComplex};
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n_r; r += nw) {
        const uint4 *src[2] = {reinterpret_cast<const uint4 *>(phi + r * ld_phi), reinterpret_cast<const uint4 *>(psi + r * ld_psi)};
        uint4 v[2][NV];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int i = 0; i < NV; ++i)
                v[s][i] = lane + 32 * i < np[s] ? __ldcs(src[s] + lane + 32 * i) : make_uint4(0u, 0u, 0u, 0u);
        uint32_t mx[2] = {0u, 0u}, mn[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
#pragma unroll
        for (int s = 0; s < 2; ++s) {
#pragma unroll
            for (int i = 0; i < NV; ++i)
                if (lane + 32 * i < np[s]) P::range(v[s][i], mx[s], mn[s]);
            if (psm || s == 1) {
                if (!psm) {   // one window
                    mx[1] = __vmaxu2(mx[0], mx[1]);
                    mn[1] = __vminu2(mn[0], mn[1]);
                }
                mx[s] = __reduce_max_sync(0xffffffffu, max(mx[s] >> 16, mx[s] & 0xFFFFu));
                mn[s] = __reduce_min_sync(0xffffffffu, min(mn[s] >> 16, mn[s] & 0xFFFFu));
                mn[s] |= mn[s] << 16;
            }
        }
        if (!psm) {
            mx[0] = mx[1];
            mn[0] = mn[1];
        }
        U128 sum[2] = {{0ull, 0ull}, {0ull, 0ull}};
        int E[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            E[s] = P::exponent(mx[s]);
            if (E[s] <= -1000) {   // no normal component: the window from the full patterns
                int m = kNoExp;
#pragma unroll
                for (int z = 0; z < 2; ++z)
#pragma unroll
                    for (int i = 0; i < NV; ++i)
                        if (z == s || !psm) m = max(m, P::exact_exponent(v[z][i]));
                E[s] = __reduce_max_sync(0xffffffffu, m);
            }
            if (E[s] == kNoExp) continue;
            U128 one{0ull, 0ull};
            if (P::plain(mn[s], E[s])) P::template squares<true>(v[s], np[s], lane, E[s], one, c);
            else P::template squares<false>(v[s], np[s], lane, E[s], one, c);
            if (psm) sum[s] = one;
            else add_u128(sum[0], one.lo, one.hi);
        }
        sum[0] = warp_sum(sum[0]);
        double x = E[0] == kNoExp ? 0.0 : u128_scaled(sum[0], 2 * E[0] - 110);
        if (psm) {
            sum[1] = warp_sum(sum[1]);
            x = __dmul_rn(x, E[1] == kNoExp ? 0.0 : u128_scaled(sum[1], 2 * E[1] - 110));
        }
        if (lane == 0) w[r] = acc ? __dadd_rn(w[r], x) : x;   // shared weight of several pairs: one rounding per pair
    }
}

// |z|^alpha in FP64 for alpha != 2: m = re*re + im*im with each operation rounded (for complex64
// input the products are exact, so one fused multiply-add gives the same bits)
template <int AK>  // 1, 3, 4: sqrt/product forms; 0: pow
__device__ __forceinline__ double modulus_pow(double re, double im, bool exact_products, double half_alpha)
{
    const double m = exact_products ? __fma_rn(re, re, __dmul_rn(im, im))
                                    : __dadd_rn(__dmul_rn(re, re), __dmul_rn(im, im));
    if (AK == 1) return __dsqrt_rn(m);
    if (AK == 3) return __dmul_rn(m, __dsqrt_rn(m));
    if (AK == 4) return __dmul_rn(m, m);
    return pow(m, half_alpha);
}

template <typename T, int AK, typename F>
__device__ __forceinline__ void for_terms(const T *row, int n, int lane, double half_alpha, F &&fn)
{
    for (int i = lane; i < n; i += 32) {
        const double2 z = cload(row, i);
        fn(modulus_pow<AK>(z.x, z.y, sizeof(T) == 8, half_alpha));
    }
}

// floor(t 2^s) of a non-negative double as a 128-bit integer (t 2^s < 2^127)
__device__ __forceinline__ void add_fixed(U128 &a, double t, int s)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(t);
    const int b = (int)((u >> 52) & 0x7FF);
    const unsigned long long f = u & 0xFFFFFFFFFFFFFull;
    if (!b && !f) return;
    const unsigned long long m = b ? (f | (1ull << 52)) : f;
    add_shifted128(a, m, 0ull, (b ? b - 1075 : -1074) + s);
}

// alpha != 2: the FP64 terms summed exactly over both sets (the terms are formed twice: once for
// the window, once for the sum; this path serves the weight-function study)
template <typename T, int AK>
__global__ void __launch_bounds__(kThreads) weights_terms(const T *__restrict__ phi, int64_t ld_phi, int n_phi,
                                                          const T *__restrict__ psi, int64_t ld_psi, int n_psi,
                                                          int64_t n_r, double half_alpha, double *__restrict__ w,
                                                          int acc)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n_r; r += nw) {
        const T *a = phi + r * ld_phi, *b = psi + r * ld_psi;
        int e = kNoExp;
        auto mx = [&](double t) {
            if (t != 0.0) e = max(e, exp_of((unsigned long long)__double_as_longlong(t)));
        };
        for_terms<T, AK>(a, n_phi, lane, half_alpha, mx);
        for_terms<T, AK>(b, n_psi, lane, half_alpha, mx);
        const int E = __reduce_max_sync(0xffffffffu, e);
        U128 s{0ull, 0ull};
        if (E != kNoExp) {
            auto add = [&](double t) { add_fixed(s, t, 110 - E); };
            for_terms<T, AK>(a, n_phi, lane, half_alpha, add);
            for_terms<T, AK>(b, n_psi, lane, half_alpha, add);
        }
        s = warp_sum(s);
        const double v = E == kNoExp ? 0.0 : u128_scaled(s, E - 110);
        if (lane == 0) w[r] = acc ? __dadd_rn(w[r], v) : v;
    }
}

unsigned grid_rows(int64_t n_r)
{
    // 4 blocks of 8 warps per SM: enough loads in flight, and the rows between a warp's two passes
    // (about 32 warps x 152 SMs rows) stay in L2 for the second read
    const int64_t g = (n_r + 7) / 8;
    return (unsigned)(g < 152 * 4 ? (g < 1 ? 1 : g) : 152 * 4);
}

template <typename T>
isdf_status launch_weights(const void *phi, int64_t ld_phi, int n_phi, const void *psi, int64_t ld_psi,
                           int n_psi, int64_t n_r, int psm, double alpha, double *w, int acc, cudaStream_t st)
{
    const unsigned grid = grid_rows(n_r);
    const T *a = static_cast<const T *>(phi);
    const T *b = static_cast<const T *>(psi);
    const double ha = 0.5 * alpha;
    // registers: whole 16-byte pieces, every row aligned, at most 8 pieces a lane and set
    constexpr int kc = Piece<T>::kComplex;
    const int widest = n_phi > n_psi ? n_phi : n_psi;
    const bool rows = n_phi % kc == 0 && n_psi % kc == 0 && ld_phi % kc == 0 && ld_psi % kc == 0 && aligned(phi, 16) &&
                      aligned(psi, 16) && widest <= 8 * 32 * kc;
    if ((psm || alpha == 2.0) && rows) {
        const int nv = (widest / kc + 31) / 32;
        const unsigned g = (unsigned)((n_r + 7) / 8 < 152 * 4 ? (n_r + 7) / 8 : 152 * 4);
#define ROWS_CASE(NV) weights_rows<T, NV><<<g, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, psm, w, acc, \
                                                                   Pow2{2u, 16u, 256u, 1u << 28})
        if (nv <= 1) ROWS_CASE(1);
        else if (nv <= 2) ROWS_CASE(2);
        else if (nv <= 4) ROWS_CASE(4);
        else ROWS_CASE(8);
#undef ROWS_CASE
    } else if (psm || alpha == 2.0) {
        if constexpr (sizeof(T) == 8)
            weights_squares_c64<<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, psm, w, acc);
        else
            weights_squares_c128<<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, psm, w, acc);
    }
    else if (alpha == 1.0)
        weights_terms<T, 1><<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, ha, w, acc);
    else if (alpha == 3.0)
        weights_terms<T, 3><<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, ha, w, acc);
    else if (alpha == 4.0)
        weights_terms<T, 4><<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, ha, w, acc);
    else
        weights_terms<T, 0><<<grid, kThreads, 0, st>>>(a, ld_phi, n_phi, b, ld_psi, n_psi, n_r, ha, w, acc);
    isdf_note_launch();
    ISDF_LAUNCH_CHECK();
    return ISDF_OK;
}

}  // namespace

extern "C" isdf_status isdf_weights(const void *phi, int64_t ld_phi, int32_t n_phi, const void *psi,
                                    int64_t ld_psi, int32_t n_psi, int64_t n_r, int32_t dtype, int32_t kind,
                                    double alpha, double *w, void *stream)
{
    if (n_r < 0 || n_phi < 1 || n_psi < 1 || ld_phi < n_phi || ld_psi < n_psi) return ISDF_ERR_INVALID_ARG;
    if (dtype != ISDF_C128 && dtype != ISDF_C64) return ISDF_ERR_INVALID_ARG;
    const int acc = (kind & ISDF_W_ACCUMULATE) ? 1 : 0;
    kind &= ~ISDF_W_ACCUMULATE;
    if (kind != ISDF_W_SSM && kind != ISDF_W_PSM) return ISDF_ERR_INVALID_ARG;
    if (!(alpha > 0.0) || alpha > 1e6) return ISDF_ERR_INVALID_ARG;
    if (n_r == 0) return ISDF_OK;
    if (!phi || !psi || !w) return ISDF_ERR_INVALID_ARG;
    const size_t el = dtype == ISDF_C128 ? 16 : 8;
    if (!aligned(phi, el) || !aligned(psi, el) || !aligned(w, 8)) return ISDF_ERR_INVALID_ARG;
    cudaStream_t st = as_stream(stream);
    if (dtype == ISDF_C128)
        return launch_weights<double2>(phi, ld_phi, n_phi, psi, ld_psi, n_psi, n_r, kind == ISDF_W_PSM, alpha, w, acc,
                                       st);
    return launch_weights<float2>(phi, ld_phi, n_phi, psi, ld_psi, n_psi, n_r, kind == ISDF_W_PSM, alpha, w, acc, st);
}

static unsigned long long g_launches = 0;

void isdf_note_launch() { __atomic_add_fetch(&g_launches, 1ull, __ATOMIC_RELAXED); }

extern "C" unsigned long long isdf_kernel_launches(void) { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

extern "C" const char *isdf_status_string(isdf_status s)
{
    switch (s) {
    case ISDF_OK: return "ok";
    case ISDF_ERR_INVALID_ARG: return "invalid argument";
    case ISDF_ERR_CUDA: return "CUDA runtime error";
    case ISDF_ERR_NOT_HPD: return "C C^H is not Hermitian positive definite";
    case ISDF_ERR_EMPTY_CLUSTER: return "empty K-means cluster";
    case ISDF_ERR_NONFINITE: return "non-finite value";
    case ISDF_ERR_TIMEOUT: return "bounded device wait timed out";
    case ISDF_ERR_WORKSPACE: return "workspace missing or too small";
    case ISDF_ERR_UNSUPPORTED: return "unsupported size";
    }
    return "unknown status";
}
