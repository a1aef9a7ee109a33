// FP64 blocked Cholesky of M = C C^H (the paper solves its least-squares
// normal equations with a linear solver, Sec. 2.4), the inverse of the
// Cholesky factor and M^-1 = L^-H L^-1.
//
// Right-looking Cholesky with 16-wide panels, one launch per block column
// (chol_step): the diagonal block is factored in shared memory, the panel below,
// L21 = A21 L11^-H, is a forward substitution with L11 (two rows per warp), and
// the trailing lower triangle is updated by A22 -= L21 L21^H of the column
// before. The diagonal blocks are then inverted together, and L^-1 is
// assembled bottom-up from them, one batched launch per level:
// inv([[A, 0], [B, C]]) = [[A^-1, 0], [-C^-1 B A^-1, C^-1]].
// Above 512 rows (with the tensor-core FP64 products enabled) the matrix is
// split in halves recursively: the factor and the inverse of the leading half
// give L21 = A21 L11^-H as one product, the Schur complement A22 - L21 L21^H is
// one more, and the inverse's off-diagonal block two more, so that most flops
// run as large exact-slicing products instead of 16-wide FP64 steps.
#include "chol.cuh"
#include "plan.cuh"
#include "zgemm.cuh"
#include "ozaki.cuh"

namespace {

constexpr int NB = 16;    // diagonal block edge (short per-block FP64 chains on the critical path)
constexpr int EW = 256;   // element threads of the diagonal-block kernel (2 warps per SMSP hide FP64 latency)
constexpr int DT = EW + 32;   // plus one pivot warp
constexpr int kSms = 152;
constexpr int MAXE = (NB * (NB + 1) / 2 + EW - 1) / EW;   // elements per thread and step

// 1/d for a positive normal d: a float seed (integer conversion, rcp.approx) refined by
// two Newton-Raphson steps r <- r + r (1 - d r), each doubling the correct bits
// (22 -> 44 -> 88), i.e. a result within about one ulp in four dependent FMAs.
__device__ __forceinline__ double recip_pos(double d)
{
    const int e = (int)((__double_as_longlong(d) >> 52) & 0x7FF) - 1023;
    if (e < -120 || e > 120) return 1.0 / d;
    float f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(d2f_int(d)));
    double r = f2d_int(f);
    double t = fma(-d, r, 1.0);
    r = fma(r, t, r);
    t = fma(-d, r, 1.0);
    return fma(r, t, r);
}

// GB300 issues one FP64 warp instruction per 16 clocks and SM, so on this one-CTA critical path the FP64 instruction
// count and its dependency chains set the time. A diagonal block is factored as L^ D L^H by elimination, one barrier
// per pivot: step j subtracts m_i conj(A_cj) from A_ic (j < c <= i), m_i = A_ij / d_j. The active entries of a step
// are numbered contiguously and dealt to 256 threads, each loading all of its (up to 2) entries before computing
// them, so that their FP64 chains overlap and warps run full. A ninth warp meanwhile updates the next pivot and forms
// 1/d_{j+1}. Afterwards L = (eliminated columns) D^-1/2. The inverse of L_kk is not on this critical path: the panel
// is a forward substitution with L_kk and the inverses of all diagonal blocks are formed together after the
// factorisation (inv_diag).
//
// The elimination of an nb x nb block held in shared memory (lower triangle of T; d0s its original diagonal
// entries of M), by every thread of a DT-thread CTA. Afterwards T's columns hold the eliminated values with
// d_j on the diagonal. Returns false (status set) at a pivot not above 1e-13 of d0 or not finite.
__device__ bool factor_block(double2 (*T)[NB + 1], const double *d0s, double *rpiv, int *bad, int k, int nb,
                             DeviceStatus *st)
{
    const int tid = threadIdx.x;
    if (tid == 0) {
        const double d = T[0][0].x;
        bad[0] = (!(d > 1e-13 * d0s[0]) || isinf(d)) ? 1 : 0;
        rpiv[0] = recip_pos(d);
    }
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        const int b = bad[j & 1];   // uniform: written before the last barrier, not rewritten until the next
        if (b) {
            if (tid == 0) set_status(st, isnan(T[b - 1][b - 1].x) ? ISDF_ERR_NONFINITE : ISDF_ERR_NOT_HPD, k + b - 1);
            return false;
        }
        const double r = rpiv[j];
        const int rows = nb - 1 - j;               // i = j+1 .. nb-1
        const int nT = rows * (rows + 1) / 2;      // j < c <= i; entry 0 is the next pivot (j+1, j+1)
        if (tid < EW) {
            int ii[MAXE], cc[MAXE];
            bool on[MAXE];
            double2 av[MAXE], bv[MAXE], tv[MAXE];
#pragma unroll
            for (int q = 0; q < MAXE; ++q) {
                const int e = 1 + tid + q * EW;
                on[q] = e < nT;
                int i = 0, c = 0;
                if (on[q]) {
                    // counted from the last column backwards: column nb-1-p holds p+1 entries
                    const int qq = nT - 1 - e;
                    int p = (int)((sqrtf(8.f * (float)qq + 1.f) - 1.f) * 0.5f);
                    if ((p + 1) * (p + 2) / 2 <= qq) ++p;
                    if (p * (p + 1) / 2 > qq) --p;
                    c = nb - 1 - p;
                    i = nb - 1 - (qq - p * (p + 1) / 2);
                    const double2 bb = T[c][j];
                    bv[q] = make_double2(bb.x, -bb.y);
                    tv[q] = T[i][c];
                    av[q] = T[i][j];
                }
                ii[q] = i;
                cc[q] = c;
            }
#pragma unroll
            for (int q = 0; q < MAXE; ++q) {
                if (on[q]) {   // t -= m conj(b), m = a / d_j
                    const double mx = av[q].x * r, my = av[q].y * r;
                    tv[q].x = fma(-mx, bv[q].x, fma(my, bv[q].y, tv[q].x));
                    tv[q].y = fma(-mx, bv[q].y, fma(-my, bv[q].x, tv[q].y));
                }
            }
#pragma unroll
            for (int q = 0; q < MAXE; ++q)
                if (on[q]) T[ii[q]][cc[q]] = tv[q];
        } else if (tid == EW && nT > 0) {   // the next pivot: A_{j+1,j+1} -= |A_{j+1,j}|^2 / d_j
            const double2 a = T[j + 1][j];
            const double d = fma(-fma(a.x, a.x, a.y * a.y), r, T[j + 1][j + 1].x);
            T[j + 1][j + 1] = make_double2(d, 0.0);
            bad[(j + 1) & 1] = (!(d > 1e-13 * d0s[j + 1]) || isinf(d)) ? j + 2 : 0;
            rpiv[j + 1] = recip_pos(d);
        }
        __syncthreads();
    }
    return true;
}

// 1/sqrt(d) for a positive normal d: a float seed, two Newton-Raphson steps y <- y + y (1/2 - d/2 y y) (22 -> 44 ->
// 88 correct bits); about one ulp in eight dependent FP64 operations
__device__ __forceinline__ double rsqrt_pos(double d)
{
    const int e = (int)((__double_as_longlong(d) >> 52) & 0x7FF) - 1023;
    if (e < -120 || e > 120) return 1.0 / sqrt(d);
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(d2f_int(d)));
    double y = f2d_int(f);
    const double h = 0.5 * d;
    y = fma(y, fma(-h * y, y, 0.5), y);
    return fma(y, fma(-h * y, y, 0.5), y);
}

// One step of the right-looking factorisation in a single launch. Block column k (NB wide) is final (none for
// k < 0); the next one is at k1, nb1 wide, with `rows` rows below its diagonal block. CTAs 0 .. n_panel - 1 advance
// block column k1:
//   D   = A[k1:k1+nb1, k1:k1+nb1] - P P^H,  P = L[k1:k1+nb1, k:k+NB]   every panel CTA, in shared memory
//   L11 = chol(D)                                                      every panel CTA, the same elimination
//   x_r L11^H = A[r, k1:k1+nb1] - L[r, k:k+NB] P^H                      this CTA's rpc rows r, two per warp
// (a pivot not above 1e-13 of M's original diagonal entry M0 is reported). Every panel CTA reads the old diagonal
// block before anyone may overwrite it: the one that arrives last on the status word's counter (after its reads)
// writes L11 back and resets the counter; no CTA waits for another. The other CTAs, and the panel's when they are
// done, take 16 x 16 tiles of the trailing update A[k1+nb1:, k1+nb1:] -= L21 L21^H (lower triangle, L21 = rows
// k1+nb1.. of block column k) from a counter of this step.
//
// Bound: FP64 issue (a 16 x 16 x 16 complex product takes 8.2k clocks of an SM's FP64 pipe) and the chain launch ->
// D -> 16 pivots -> substitution. One launch a step in one stream; two streams joined by events every step, a launch
// each for the panel (8 rows a CTA on half-empty warps) and the trailing update (32 x 32 tiles) made the plan update
// of N_mu = 1024 0.5 ms and of 4096 2.1 ms longer (30.6 -> 28.5 ms).
__global__ void __launch_bounds__(DT) chol_step(double2 *A, int64_t lda, const double2 *M0, int k, int k1, int nb1,
                                               int rows, int n_panel, int rpc, int *tiles, DeviceStatus *st)
{
    __shared__ double2 T[NB][NB + 1];
    __shared__ double2 P[NB][NB + 1];
    __shared__ double d0s[NB], rpiv[NB], rs[NB];
    __shared__ int bad[2];
    __shared__ int last, tile_sh;
    if (st->code != 0) return;
    const int tid = threadIdx.x;
    const double2 zero = make_double2(0.0, 0.0);
    if (blockIdx.x < n_panel) {
        for (int e = tid; e < NB * NB; e += DT) {
            const int i = e / NB, l = e % NB;
            P[i][l] = k >= 0 && i < nb1 ? A[(int64_t)(k1 + i) * lda + (k + l)] : zero;
        }
        if (tid < nb1) d0s[tid] = M0[(int64_t)(k1 + tid) * lda + (k1 + tid)].x;
        // D = A - P P^H: the 136 entries of the lower triangle on consecutive threads
        int i = 0, j = 0;
        double2 t = zero;
        if (tid < NB * (NB + 1) / 2) {
            i = (int)((sqrtf(8.f * (float)tid + 1.f) - 1.f) * 0.5f);
            if ((i + 1) * (i + 2) / 2 <= tid) ++i;
            if (i * (i + 1) / 2 > tid) --i;
            j = tid - i * (i + 1) / 2;
            if (i < nb1) t = A[(int64_t)(k1 + i) * lda + (k1 + j)];
        }
        __syncthreads();
        if (tid < NB * (NB + 1) / 2) {
            if (k >= 0) {
#pragma unroll 4
                for (int l = 0; l < NB; ++l) {   // t -= P_il conj(P_jl)
                    const double2 a = P[i][l], b = P[j][l];
                    t.x = fma(-a.x, b.x, fma(-a.y, b.y, t.x));
                    t.y = fma(-a.y, b.x, fma(a.x, b.y, t.y));
                }
            }
            T[i][j] = t;
        }
        __syncthreads();   // this CTA's reads of the old diagonal block are done
        if (tid == 0) {
            __threadfence();
            last = atomicAdd(&st->ticket, 1) == n_panel - 1;
        }
        if (!factor_block(T, d0s, rpiv, bad, k1, nb1, st)) return;
        if (tid < nb1) rs[tid] = rsqrt_pos(T[tid][tid].x);
        __syncthreads();
        if (tid < NB * NB) {   // L11 in place: columns scaled by d^-1/2, diagonal sqrt(d)
            const int r = tid / NB, c = tid % NB;
            double2 v = zero;
            if (r < nb1 && c < r) {
                v = make_double2(T[r][c].x * rs[c], T[r][c].y * rs[c]);
            } else if (r < nb1 && c == r) {
                const double d = T[r][r].x, s = d * rs[r];
                v.x = fma(0.5 * rs[r], fma(-s, s, d), s);   // sqrt(d), the rounding of d * rs corrected
            }
            T[r][c] = v;
            if (last && r < nb1 && c < nb1) A[(int64_t)(k1 + r) * lda + (k1 + c)] = v;
        }
        if (last && tid == 0) st->ticket = 0;
        __syncthreads();
        // rows of the panel: two per warp, lane c of each half holds column c
        const int warp = tid >> 5, c = tid & (NB - 1), r1 = min(rows, (int)(blockIdx.x + 1) * rpc);
        for (int rb = blockIdx.x * rpc + 2 * warp; rb < r1; rb += 2 * (EW / 32)) {
            if (warp >= EW / 32) break;
            const int r = rb + ((tid >> 4) & 1);
            const bool on = r < r1;
            double2 *row = A + (int64_t)(k1 + nb1 + (on ? r : rb)) * lda;
            const double2 lr = k >= 0 ? row[k + c] : zero;
            double2 acc = c < nb1 ? row[k1 + c] : zero;
            if (k >= 0) {
#pragma unroll
                for (int l = 0; l < NB; ++l) {   // acc -= L[r, k + l] conj(P_cl)
                    const double ax = __shfl_sync(0xffffffffu, lr.x, l, NB), ay = __shfl_sync(0xffffffffu, lr.y, l, NB);
                    const double2 b = P[c][l];
                    acc.x = fma(-ax, b.x, fma(-ay, b.y, acc.x));
                    acc.y = fma(-ay, b.x, fma(ax, b.y, acc.y));
                }
            }
            double2 x = zero;
            const double rc = c < nb1 ? rs[c] : 0.0;
            for (int s = 0; s < nb1; ++s) {   // forward substitution x L11^H = acc, 1 / L_ss = rs[s]
                double2 xs = make_double2(acc.x * rc, acc.y * rc);
                xs.x = __shfl_sync(0xffffffffu, xs.x, s, NB);
                xs.y = __shfl_sync(0xffffffffu, xs.y, s, NB);
                if (c == s) x = xs;
                if (c > s) {   // acc -= x_s conj(L_cs)
                    const double2 b = T[c][s];
                    acc.x = fma(-xs.x, b.x, fma(-xs.y, b.y, acc.x));
                    acc.y = fma(-xs.y, b.x, fma(xs.x, b.y, acc.y));
                }
            }
            if (on && c < nb1) row[k1 + c] = x;
        }
        __syncthreads();   // T and P are reused below
    }
    if (k < 0 || rows <= 0) return;
    const int nt = (rows + NB - 1) / NB, n_tiles = nt * (nt + 1) / 2;
    const int i = (tid >> 4) & (NB - 1), j = tid & (NB - 1);
    double2 *A2 = A + (int64_t)(k1 + nb1) * lda;   // rows of the trailing matrix
    for (;;) {
        if (tid == 0) tile_sh = atomicAdd(tiles, 1);
        __syncthreads();
        const int q = tile_sh;
        if (q >= n_tiles) return;
        int bi = (int)((sqrtf(8.f * (float)q + 1.f) - 1.f) * 0.5f);
        if ((bi + 1) * (bi + 2) / 2 <= q) ++bi;
        if (bi * (bi + 1) / 2 > q) --bi;
        const int bj = q - bi * (bi + 1) / 2;
        const int ri = bi * NB + i, rj = bj * NB + j;
        double2 c = zero;
        const bool on = tid < EW && ri < rows && rj <= ri;
        if (tid < EW) {
            T[i][j] = ri < rows ? A2[(int64_t)ri * lda + (k + j)] : zero;
            P[i][j] = bj * NB + i < rows ? A2[(int64_t)(bj * NB + i) * lda + (k + j)] : zero;
            if (on) c = A2[(int64_t)ri * lda + (k1 + nb1 + rj)];
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int l = 0; l < NB; ++l) {   // c -= L_il conj(L_jl)
                const double2 a = T[i][l], b = P[j][l];
                c.x = fma(-a.x, b.x, fma(-a.y, b.y, c.x));
                c.y = fma(-a.y, b.x, fma(a.x, b.y, c.y));
            }
            A2[(int64_t)ri * lda + (k1 + nb1 + rj)] = c;
        }
        __syncthreads();
    }
}

// Inverses of all diagonal blocks of L (one CTA each): with L^ = L D^-1 (unit
// diagonal), X = L^^-1 by elimination on [L^ | I] (step j: X_ic -= L^_ij X_jc,
// c <= j < i, one barrier per step), then L_kk^-1 = D^-1 X.
__global__ void __launch_bounds__(EW) inv_diag(const double2 *L, int64_t ld, double2 *Linv, int64_t ldi, int n,
                                              const DeviceStatus *st)
{
    __shared__ double2 T[NB][NB + 1];
    __shared__ double2 X[NB][NB + 1];
    __shared__ double rs[NB];   // 1 / L_jj
    if (st->code != 0) return;
    const int k = blockIdx.x * NB, nb = min(NB, n - k), tid = threadIdx.x;
    for (int e = tid; e < NB * NB; e += EW) {
        const int i = e / NB, j = e % NB;
        T[i][j] = (i < nb && j <= i) ? L[(int64_t)(k + i) * ld + (k + j)] : make_double2(0.0, 0.0);
        X[i][j] = make_double2(i == j && i < nb ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    if (tid < nb) rs[tid] = 1.0 / T[tid][tid].x;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        const int nX = (nb - 1 - j) * (j + 1);   // at most 16 x 16 = 256 = EW
        for (int e = tid; e < nX; e += EW) {
            const int i = j + 1 + e / (j + 1), c = e % (j + 1);
            const double2 a = T[i][j], b = X[j][c];
            const double mx = a.x * rs[j], my = a.y * rs[j];
            double2 x = X[i][c];
            x.x = fma(-mx, b.x, fma(my, b.y, x.x));
            x.y = fma(-mx, b.y, fma(-my, b.x, x.y));
            X[i][c] = x;
        }
        __syncthreads();
    }
    for (int e = tid; e < nb * nb; e += EW) {
        const int i = e / nb, j = e % nb;
        Linv[(int64_t)(k + i) * ldi + (k + j)] =
            j <= i ? make_double2(X[i][j].x * rs[i], X[i][j].y * rs[i]) : make_double2(0.0, 0.0);
    }
}

__global__ void zero_strict_upper(double2 *A, int n, int64_t lda)
{
    const int64_t total = (int64_t)n * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e % n);
        if (j > i) A[(int64_t)i * lda + j] = make_double2(0.0, 0.0);
    }
}

ZOperand op(const double2 *p, int64_t s0, int64_t s1, int conj)
{
    ZOperand o;
    o.p = p;
    o.s0 = s0;
    o.s1 = s1;
    o.conj = conj;
    o.type = ZG_C128;
    return o;
}

ZGemm single(int M, int N, int K, ZOperand A, ZOperand B, double2 *C, int64_t ldc, double alpha, int beta)
{
    ZGemm g{};
    g.M = M;
    g.N = N;
    g.K = K;
    g.A1 = A;
    g.B1 = B;
    g.C = C;
    g.scm = ldc;
    g.scn = 1;
    g.ctype = ZG_C128;
    g.alpha = alpha;
    g.beta = beta;
    g.splits = 1;
    return g;
}

// FP64 product: on the tensor cores by exact slicing when the plan enables it, the
// shape is large enough to pay for the slicing and the scratch fits; else FP64 GEMM
isdf_status product(const ZGemm &g, double2 *part, size_t part_n, const isdf_plan *tp, cudaStream_t st)
{
    if (tp && tp->use_oz && (int64_t)g.M * g.N * (g.batch > 1 ? g.batch : 1) >= (int64_t)256 * 256 &&
        g.K >= 256 && oz_fits(g, tp->oz))
        return oz_zgemm(g, tp->oz, tp->oz_err, st);
    return zgemm_auto(g, part, part_n, st);
}

// L^-1 from the inverted diagonal blocks (NB wide) already in Linv, merging
// aligned groups of blocks bottom-up: at each level, every pair (left group
// of h rows at o, right group of r <= h rows at o + h) gets
//   tmp = L[o+h:, o:o+h] Linv[o:o+h, o:o+h],  Linv[o+h:, o:o+h] = -Linv[o+h:, o+h:] tmp,
// all full pairs of a level in one batched launch, a ragged last pair apart.
isdf_status tri_inv(const double2 *L, double2 *Linv, double2 *tmp, int64_t ld, int n, double2 *part,
                    size_t part_n, const isdf_plan *tp, cudaStream_t st)
{
    const int nblk = (n + NB - 1) / NB;
    for (int g = 1; g < nblk; g *= 2) {
        const int h = g * NB;
        const int full = n / (2 * h);
        const int64_t step = (int64_t)2 * h * (ld + 1);   // from one pair's diagonal block to the next
        if (full > 0) {
            ZGemm g1 = single(h, h, h, op(L + (int64_t)h * ld, ld, 1, 0), op(Linv, ld, 1, 0), tmp, h, 1.0, 0);
            g1.kmode = ZG_K_FROM_N0;   // Linv lower: k >= n
            g1.batch = full;
            g1.bsa = step;
            g1.bsb = step;
            g1.bsc = (int64_t)h * h;
            ISDF_TRY(product(g1, part, part_n, tp, st));
            ZGemm g2 = single(h, h, h, op(Linv + (int64_t)h * (ld + 1), ld, 1, 0), op(tmp, h, 1, 0),
                              Linv + (int64_t)h * ld, ld, -1.0, 0);
            g2.k_to_m_end = 1;         // Linv lower: k <= m
            g2.batch = full;
            g2.bsa = step;
            g2.bsb = (int64_t)h * h;
            g2.bsc = step;
            ISDF_TRY(product(g2, part, part_n, tp, st));
        }
        const int o = full * 2 * h, r = n - o - h;
        if (r > 0) {
            ZGemm g1 = single(r, h, h, op(L + (int64_t)(o + h) * ld + o, ld, 1, 0),
                              op(Linv + (int64_t)o * ld + o, ld, 1, 0), tmp, h, 1.0, 0);
            g1.kmode = ZG_K_FROM_N0;
            ISDF_TRY(product(g1, part, part_n, tp, st));
            ZGemm g2 = single(r, h, r, op(Linv + (int64_t)(o + h) * ld + (o + h), ld, 1, 0), op(tmp, h, 1, 0),
                              Linv + (int64_t)(o + h) * ld + o, ld, -1.0, 0);
            g2.k_to_m_end = 1;
            ISDF_TRY(product(g2, part, part_n, tp, st));
        }
    }
    return ISDF_OK;
}

// Right-looking blocked factorisation of the diagonal block L[o:o+m, o:o+m] in place (its lower
// triangle holds the matrix; earlier columns are already final): one chol_step launch per block column.
isdf_status chol_blocked(const double2 *M0, double2 *L, int64_t ld, int o, int m, DeviceStatus *st, cudaStream_t stream,
                         int *ctr)
{
    const int end = o + m;
    for (int k1 = o; k1 < end; k1 += NB) {
        const int k = k1 > o ? k1 - NB : -1, nb1 = end - k1 < NB ? end - k1 : NB, rows = end - k1 - nb1;
        // 4 rows a panel CTA (two warps: 2.5 us of substitution) while that leaves more than half of the SMs to the
        // trailing update, else 8
        const int rpc = rows <= 256 ? 4 : 8;
        const int n_panel = rows > 0 ? ((rows + rpc - 1) / rpc < kSms ? (rows + rpc - 1) / rpc : kSms) : 1;
        const int per = (rows + n_panel - 1) / n_panel;
        const int nt = k >= 0 ? (rows + NB - 1) / NB : 0, n_tiles = nt * (nt + 1) / 2;
        // one CTA per SM (a second one slows the panel's chain down) until the tiles are several per SM
        const int room = n_tiles > 8 * kSms ? 3 * kSms : kSms;
        int grid = n_panel + n_tiles < room ? n_panel + n_tiles : room;
        if (grid < n_panel) grid = n_panel;
        chol_step<<<grid, DT, 0, stream>>>(L, ld, M0, k, k1, nb1, rows, n_panel, per > 0 ? per : 1, ctr + k1 / NB, st);
        isdf_note_launch();
        ISDF_LAUNCH_CHECK();
    }
    return ISDF_OK;
}

// The inverse of the factored diagonal block L[o:o+m, o:o+m] into Linv[o:o+m, o:o+m]: its NB-wide
// diagonal blocks inverted at once, then merged bottom-up (tri_inv).
isdf_status inverse_blocked(const double2 *L, double2 *Linv, double2 *tmp, int64_t ld, int o, int m, double2 *part,
                            size_t part_n, DeviceStatus *st, cudaStream_t stream, const isdf_plan *tp)
{
    const double2 *Lo = L + (int64_t)o * ld + o;
    double2 *Io = Linv + (int64_t)o * ld + o;
    inv_diag<<<(m + NB - 1) / NB, EW, 0, stream>>>(Lo, ld, Io, ld, m, st); isdf_note_launch();
    ISDF_LAUNCH_CHECK();
    return tri_inv(Lo, Io, tmp, ld, m, part, part_n, tp, stream);
}

// Recursive factorisation and inverse of the diagonal block [o, o+m) for large blocks, so that
// most of the (4/3) m^3 flops of each are in large products (on the tensor cores by exact slicing
// when the plan enables it): with the block split at m1,
//   L11 = chol(A11), L11^-1                 (recursively)
//   L21 = A21 L11^-H                        (product; L11^-1 is at hand)
//   A22 <- A22 - L21 L21^H                  (lower tiles)
//   L22 = chol(A22), L22^-1                 (recursively)
//   (L^-1)21 = -L22^-1 (L21 L11^-1)
// Blocks of at most kRecBase rows use the blocked factorisation and inverse above.
constexpr int kRecBase = 512;

isdf_status chol_rec(const double2 *M0, double2 *L, double2 *Linv, double2 *tmp, int64_t ld, int o, int m,
                     double2 *part, size_t part_n, DeviceStatus *st, cudaStream_t stream, isdf_plan *tp)
{
    if (m <= kRecBase) {
        ISDF_TRY(chol_blocked(M0, L, ld, o, m, st, stream, tp->chol_ctr));
        return inverse_blocked(L, Linv, tmp, ld, o, m, part, part_n, st, stream, tp);
    }
    const int m1 = ((m / 2 + NB - 1) / NB) * NB, m2 = m - m1;
    ISDF_TRY(chol_rec(M0, L, Linv, tmp, ld, o, m1, part, part_n, st, stream, tp));
    double2 *A21 = L + (int64_t)(o + m1) * ld + o;
    const double2 *I11 = Linv + (int64_t)o * ld + o;
    // L21 = A21 L11^-H into tmp (m2 x m1), then back in place
    ZGemm g = single(m2, m1, m1, op(A21, ld, 1, 0), op(I11, 1, ld, 1), tmp, m1, 1.0, 0);
    ISDF_TRY(product(g, part, part_n, tp, stream));
    ISDF_CUDA_TRY(cudaMemcpy2DAsync(A21, sizeof(double2) * ld, tmp, sizeof(double2) * m1, sizeof(double2) * m1, m2,
                                    cudaMemcpyDeviceToDevice, stream));
    // A22 -= L21 L21^H (lower tiles)
    ZGemm u = single(m2, m2, m1, op(A21, ld, 1, 0), op(A21, 1, ld, 1), L + (int64_t)(o + m1) * (ld + 1), ld, -1.0, 1);
    u.lower_only = 1;
    ISDF_TRY(product(u, part, part_n, tp, stream));
    ISDF_TRY(chol_rec(M0, L, Linv, tmp, ld, o + m1, m2, part, part_n, st, stream, tp));
    // (L^-1)21 = -L22^-1 (L21 L11^-1)
    ZGemm g1 = single(m2, m1, m1, op(A21, ld, 1, 0), op(I11, ld, 1, 0), tmp, m1, 1.0, 0);
    g1.kmode = ZG_K_FROM_N0;   // L11^-1 lower: k >= n
    ISDF_TRY(product(g1, part, part_n, tp, stream));
    ZGemm g2 = single(m2, m1, m2, op(Linv + (int64_t)(o + m1) * (ld + 1), ld, 1, 0), op(tmp, m1, 1, 0),
                      Linv + (int64_t)(o + m1) * ld + o, ld, -1.0, 0);
    g2.k_to_m_end = 1;         // L22^-1 lower: k <= m
    return product(g2, part, part_n, tp, stream);
}

}  // namespace

int chol_steps(int n) { return (n + NB - 1) / NB; }

isdf_status cholesky_inverse(const double2 *M0, double2 *L, double2 *Linv, double2 *W, double2 *tmp, int n,
                             double2 *part, size_t part_n, DeviceStatus *st, cudaStream_t stream,
                             isdf_plan *tp)
{
    const int64_t ld = n;
    timer_start(tp, 3, stream);
    ISDF_CUDA_TRY(cudaMemsetAsync(tp->chol_ctr, 0, sizeof(int) * (size_t)chol_steps(n), stream));
    ISDF_CUDA_TRY(cudaMemsetAsync(Linv, 0, sizeof(double2) * (size_t)n * n, stream));
    const bool recursive = tp->use_oz && n > kRecBase;
    if (recursive) {
        // factor and inverse together (timed as stage 3; stage 4 records nothing)
        ISDF_TRY(chol_rec(M0, L, Linv, tmp, ld, 0, n, part, part_n, st, stream, tp));
        const int64_t total = (int64_t)n * n;
        const unsigned gr = (unsigned)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
        zero_strict_upper<<<gr, 256, 0, stream>>>(L, n, ld); isdf_note_launch();
        ISDF_LAUNCH_CHECK();
        timer_stop(tp, 3, stream, n);
    } else {
        ISDF_TRY(chol_blocked(M0, L, ld, 0, n, st, stream, tp->chol_ctr));
        const int64_t total = (int64_t)n * n;
        const unsigned gr = (unsigned)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
        zero_strict_upper<<<gr, 256, 0, stream>>>(L, n, ld); isdf_note_launch();
        // the inverted diagonal blocks of L, all at once (the first level of L^-1)
        inv_diag<<<(n + NB - 1) / NB, EW, 0, stream>>>(L, ld, Linv, ld, n, st); isdf_note_launch();
        ISDF_LAUNCH_CHECK();
        timer_stop(tp, 3, stream, n);
        timer_start(tp, 4, stream);
        ISDF_TRY(tri_inv(L, Linv, tmp, ld, n, part, part_n, tp, stream));
        timer_stop(tp, 4, stream, n);
    }
    timer_start(tp, 5, stream);
    // W = Linv^H Linv: W_ij = sum_{k >= max(i, j)} conj(Linv_ki) Linv_kj (lower tiles, then mirrored)
    ZGemm w = single(n, n, n, op(Linv, 1, ld, 1), op(Linv, ld, 1, 0), W, ld, 1.0, 0);
    w.kmode = ZG_K_FROM_MAX_MN;
    w.lower_only = 1;
    ISDF_TRY(product(w, part, part_n, tp, stream));
    ISDF_TRY(hermitian_mirror(W, n, ld, stream));
    timer_stop(tp, 5, stream, n);
    return ISDF_OK;
}
