// FP64 blocked Cholesky of M = C C^H (the paper solves its least-squares
// normal equations with a linear solver, Sec. 2.4), the inverse of the
// Cholesky factor and M^-1 = L^-H L^-1.
//
// Right-looking Cholesky with 16-wide panels, one launch per block column
// (chol_step): the diagonal block is factored in shared memory, the panel below,
// L21 = A21 L11^-H, is a forward substitution with L11 (one warp per row), and the
// trailing lower triangle is updated by A22 -= L21 L21^H of the column before. The
// diagonal blocks are then inverted together, and L^-1 is assembled bottom-up from
// them, one batched launch per level:
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
constexpr int EW = 256;   // threads of a step's products and rows
constexpr int DT = EW + 32;   // plus one pivot warp
constexpr int kSms = 152;

// 1/d for a positive normal d: a float seed (integer conversion, rcp.approx) refined by
// two Newton-Raphson steps r <- r + r (1 - d r): 22 correct bits, 44, then the rounding
// of the last step, i.e. a result within about one ulp in four dependent FMAs.
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

// GB300 runs an FP64 warp instruction in 64 clocks of one SM quarter, so on this one-CTA critical path the number of
// FP64 warp instructions of each quarter and their dependency chains set the time. A diagonal block is factored as
// L^ D L^H by elimination, one barrier per pivot: step j subtracts m_i conj(A_cj) from A_ic (j < c <= i),
// m_i = A_ij / d_j; at most 119 entries, one a thread, on four warps of the quarters 1 to 3. A ninth warp (quarter 0)
// meanwhile updates the next pivot and forms 1/d_{j+1}: five dependent FP64 instructions. |A_{j+1,j}|^2 comes from the
// thread that made the entry a step before, and the pivot test is one of integers: with both in the pivot warp it issued
// ten, and a step of the factorisation took 24.5 us instead of 23.1. Afterwards L = (eliminated columns) D^-1/2.
//
// A pivot that is infinite, NaN or not above the threshold thr >= 0 (bits of non-negative doubles order like integers)
__device__ __forceinline__ bool bad_pivot(double d, double thr)
{
    const long long b = __double_as_longlong(d), t = __double_as_longlong(thr);
    return b <= (t > 0 ? t : 0) || (b >> 52) == 0x7FF;
}

// The elimination of an nb x nb block held in shared memory (lower triangle of T; thr the pivots' thresholds), by every
// thread of a DT-thread CTA. Afterwards T's columns hold the eliminated values with d_j on the diagonal. Returns false
// (status set) at a bad pivot.
__device__ bool factor_block(double2 (*T)[NB + 1], const double *thr, double *rpiv, double *sq, int *bad, int k, int nb,
                             DeviceStatus *st)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // entries are dealt to warps 1, 2, 3 and 5 in this order
    const int e = (warp >= 1 && warp <= 3) ? 32 * (warp - 1) + lane : warp == 5 ? 96 + lane : NB * NB;
    if (tid == EW) {
        const double d = T[0][0].x;
        const double2 a = T[1][0];
        sq[0] = fma(a.x, a.x, a.y * a.y);
        bad[0] = bad_pivot(d, thr[0]) ? 1 : 0;
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
        if (e < nT - 1) {
            // counted from the last column backwards: column nb-1-p holds p+1 entries
            const int qq = nT - 2 - e;
            int p = (int)((sqrtf(8.f * (float)qq + 1.f) - 1.f) * 0.5f);
            if ((p + 1) * (p + 2) / 2 <= qq) ++p;
            if (p * (p + 1) / 2 > qq) --p;
            const int c = nb - 1 - p, i = nb - 1 - (qq - p * (p + 1) / 2);
            const double2 a = T[i][j], b = T[c][j];
            double2 t = T[i][c];
            const double mx = a.x * r, my = a.y * r;   // t -= m conj(b), m = a / d_j
            t.x = fma(-mx, b.x, fma(my, -b.y, t.x));
            t.y = fma(-mx, -b.y, fma(-my, b.x, t.y));
            T[i][c] = t;
            if (e == 0) sq[(j + 1) & 1] = fma(t.x, t.x, t.y * t.y);   // entry (j + 2, j + 1)
        } else if (tid == EW && nT > 0) {   // the next pivot: A_{j+1,j+1} -= |A_{j+1,j}|^2 / d_j
            const double d = fma(-sq[j & 1], r, T[j + 1][j + 1].x);
            T[j + 1][j + 1] = make_double2(d, 0.0);
            bad[(j + 1) & 1] = bad_pivot(d, thr[j + 1]) ? j + 2 : 0;
            rpiv[j + 1] = recip_pos(d);
        }
        __syncthreads();
    }
    return true;
}

// row (i, j), i >= j, of entry e of a lower triangle counted row by row
__device__ __forceinline__ void tri_entry(int e, int &i, int &j)
{
    i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if ((i + 1) * (i + 2) / 2 <= e) ++i;
    if (i * (i + 1) / 2 > e) --i;
    j = e - i * (i + 1) / 2;
}

// One part of t -= a conj(b), t.x = fma(-a.x, b.x, fma(-a.y, b.y, t.x)), t.y = fma(-a.y, b.x, fma(a.x, b.y, t.y)):
// `own` is a's part of the same kind as t, `other` the other one (im: t is the imaginary part).
__device__ __forceinline__ double sub_part(double t, double own, double other, double2 b, bool im)
{
    return fma(-own, b.x, fma(im ? other : -other, b.y, t));
}

// One step of the right-looking factorisation in a single launch. Block column k (NB wide) is final (none for
// k < 0); the next one is at k1, nb1 wide, with `rows` rows below its diagonal block. CTAs 0 .. n_panel - 1 advance
// block column k1:
//   D   = A[k1:k1+nb1, k1:k1+nb1] - P P^H,  P = L[k1:k1+nb1, k:k+NB]   every panel CTA, in shared memory
//   L11 = chol(D)                                                      every panel CTA, the same elimination
//   x_r L11^H = A[r, k1:k1+nb1] - L[r, k:k+NB] P^H                       this CTA's rpc rows r, one per warp
// (a pivot not above 1e-13 of M's original diagonal entry M0 is reported). Every panel CTA reads the old diagonal
// block before anyone may overwrite it: the one that arrives last on the status word's counter (after its reads)
// writes L11 back and resets the counter; no CTA waits for another. The other CTAs, and the panel's when they are
// done, take 16 x 16 tiles of the trailing update A[k1+nb1:, k1+nb1:] -= L21 L21^H (lower triangle, L21 = rows
// k1+nb1.. of block column k) from a counter of this step.
//
// The order in which an entry's terms are added is part of the result: the FP16 digits of M^-1 in ISDF_MIXED plans
// follow its last bits, and the complex128 gradients of that mode follow the digits. D and the panel's update subtract
// their 16 terms one by one from the entry, the substitution goes column by column, the trailing update sums its 16
// terms first, as the general GEMM does. What is free, and taken: the real and the imaginary part of an entry are two
// threads' work.
//
// Bound: FP64 issue (a 16 x 16 x 16 complex product takes 8.2k clocks of an SM's FP64 pipe) and the chain launch ->
// D -> 16 pivots -> panel rows: 23.1 us a step (a panel formed as a product with the block's inverse, whose rounding is
// another: 22.1).
__global__ void __launch_bounds__(DT) chol_step(double2 *A, int64_t lda, const double2 *M0, int k, int k1, int nb1, int rows,
                                               int n_panel, int rpc, int *tiles, DeviceStatus *st)
{
    __shared__ double2 T[NB][NB + 1];
    __shared__ double2 P[NB][NB + 1];
    __shared__ double thr[NB], rpiv[NB], sq[2], rs[NB], rd[NB];
    __shared__ int bad[2];
    __shared__ int last, tile_sh, stop;
    grid_wait();
    const int tid = threadIdx.x;
    // an earlier failure: one thread reads it for all, as a panel CTA of this launch may be reporting one meanwhile and
    // every thread has to take the same way past the barriers (a CTA that reads 0 meets the same bad pivot itself)
    if (tid == 0) stop = *(volatile int32_t *)&st->code;
    const double2 zero = make_double2(0.0, 0.0);
    if (blockIdx.x < n_panel) {
        // rows of the panel: one per warp, the first ones on warps 4 .. 7; lanes c and 16 + c hold the real and the
        // imaginary part of column c
        const int warp = tid >> 5, lane = tid & 31, c = lane & (NB - 1), im = lane >> 4;
        const int rl = min(rows, (int)(blockIdx.x + 1) * rpc);
        int r = blockIdx.x * rpc + (warp ^ 4);
        const bool row_warp = warp < EW / 32;
        double *row = reinterpret_cast<double *>(A + (int64_t)(k1 + nb1 + r) * lda) + 2 * c + im;
        double lr = 0.0, acc = 0.0;
        auto load_row = [&]() {
            lr = k >= 0 ? row[2 * k] : 0.0;
            acc = c < nb1 ? row[2 * k1] : 0.0;
        };
        auto update_row = [&]() {   // acc -= L[r, k + l] conj(P_cl)
#pragma unroll
            for (int l = 0; l < NB; ++l) {
                const double own = __shfl_sync(0xffffffffu, lr, (lane & NB) + l);
                const double other = __shfl_sync(0xffffffffu, lr, (~lane & NB) + l);
                acc = sub_part(acc, own, other, P[c][l], im);
            }
        };
        const bool mine = row_warp && r < rl;
        if (mine) load_row();   // ahead: the block's factorisation hides the latency
        if (tid < NB * NB) {
            const int i = tid / NB, l = tid % NB;
            P[i][l] = k >= 0 && i < nb1 ? A[(int64_t)(k1 + i) * lda + (k + l)] : zero;
        }
        if (tid < nb1) thr[tid] = 1e-13 * M0[(int64_t)(k1 + tid) * lda + (k1 + tid)].x;
        // D = A - P P^H: the real parts of the lower triangle's 136 entries, then the imaginary parts of the 120 below
        // the diagonal, one a thread
        constexpr int NT = NB * (NB + 1) / 2;
        const bool dim = tid >= NT;
        int i = 0, j = 0;
        double t = 0.0;
        if (tid < NB * NB) {
            tri_entry(dim ? tid - NT : tid, i, j);
            if (dim) ++i;
            if (i < nb1) t = reinterpret_cast<const double *>(A + (int64_t)(k1 + i) * lda + (k1 + j))[dim];
        }
        __syncthreads();
        if (stop) return;
        if (tid < NB * NB) {
            if (k >= 0) {
#pragma unroll
                for (int l = 0; l < NB; ++l) {   // t -= P_il conj(P_jl)
                    const double2 a = P[i][l];
                    t = sub_part(t, dim ? a.y : a.x, dim ? a.x : a.y, P[j][l], dim);
                }
            }
            reinterpret_cast<double *>(&T[i][j])[dim] = t;
            if (i == j) T[i][j].y = 0.0;
        }
        __syncthreads();   // this CTA's reads of the old diagonal block are done
        if (tid == 0) {
            __threadfence();
            last = atomicAdd(&st->ticket, 1) == n_panel - 1;
        }
        if (!factor_block(T, thr, rpiv, sq, bad, k1, nb1, st)) return;
        if (tid < NB) {   // 1 / sqrt(d), 1 / L_ii; the other warps update their rows meanwhile
            const double d = tid < nb1 ? T[tid][tid].x : 1.0;
            rs[tid] = 1.0 / sqrt(d);
            rd[tid] = 1.0 / (d * rs[tid]);
        }
        __syncwarp();
        if (mine && k >= 0) update_row();
        __syncthreads();
        if (tid < NB * NB) {   // L11 = columns scaled by d^-1/2, zeros above the diagonal
            const int a = tid / NB, b = tid % NB;
            double2 v = zero;
            if (a < nb1 && b < a) v = make_double2(T[a][b].x * rs[b], T[a][b].y * rs[b]);
            else if (a < nb1 && b == a) v.x = T[a][a].x * rs[a];
            T[a][b] = v;
            if (last && a < nb1 && b < nb1) A[(int64_t)(k1 + a) * lda + (k1 + b)] = v;
        }
        if (last && tid == 0) st->ticket = 0;
        __syncthreads();
        for (bool on = mine; on;) {
            double x = 0.0;
#pragma unroll
            for (int s = 0; s < NB; ++s) {   // x L11^H = acc: x_s = acc_s / L_ss, acc_c -= x_s conj(L_cs) for c > s
                const double xs = acc * rd[s];
                const double own = __shfl_sync(0xffffffffu, xs, (lane & NB) + s);
                const double other = __shfl_sync(0xffffffffu, xs, (~lane & NB) + s);
                if (c == s) x = own;
                if (c > s) acc = sub_part(acc, own, other, T[c][s], im);
            }
            if (c < nb1) row[2 * k1] = x;
            r += EW / 32;
            on = r < rl;
            if (on) {
                row += (int64_t)(EW / 32) * 2 * lda;
                load_row();
                if (k >= 0) update_row();
            }
        }
    }
    __syncthreads();   // T and P are reused below
    if (stop) return;
    grid_release();
    if (k < 0 || rows <= 0) return;
    const int nt = (rows + NB - 1) / NB, n_tiles = nt * (nt + 1) / 2;
    const int i = (tid >> 4) & (NB - 1), j = tid & (NB - 1);
    double2 *A2 = A + (int64_t)(k1 + nb1) * lda;   // rows of the trailing matrix
    for (;;) {
        if (tid == 0) tile_sh = atomicAdd(tiles, 1);
        __syncthreads();
        const int q = tile_sh;
        if (q >= n_tiles) return;
        int bi, bj;
        tri_entry(q, bi, bj);
        const int ri = bi * NB + i, rj = bj * NB + j;
        double2 o = zero, c = zero;
        const bool on = tid < EW && ri < rows && rj <= ri;
        if (tid < EW) {
            T[i][j] = ri < rows ? A2[(int64_t)ri * lda + (k + j)] : zero;
            P[i][j] = bj * NB + i < rows ? A2[(int64_t)(bj * NB + i) * lda + (k + j)] : zero;
            if (on) o = A2[(int64_t)ri * lda + (k1 + nb1 + rj)];
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int l = 0; l < NB; ++l) {   // c += L_il conj(L_jl)
                const double2 a = T[i][l], b = P[j][l];
                c.x = fma(a.y, b.y, fma(a.x, b.x, c.x));
                c.y = fma(a.y, b.x, fma(a.x, -b.y, c.y));
            }
            A2[(int64_t)ri * lda + (k1 + nb1 + rj)] = make_double2(o.x - c.x, o.y - c.y);
        }
        __syncthreads();
    }
}

// Inverses of all diagonal blocks of L (one CTA each): with L^ = L D^-1 (unit
// diagonal), X = L^^-1 by elimination on [L^ | I] (step j: X_ic -= L^_ij X_jc,
// c <= j < i, one barrier per step), then L_kk^-1 = D^-1 X.
__global__ void __launch_bounds__(EW) inv_diag(const double2 *L, int64_t ld, double2 *Linv, int n, const DeviceStatus *st)
{
    __shared__ double2 T[NB][NB + 1];
    __shared__ double2 X[NB][NB + 1];
    __shared__ double rs[NB];   // 1 / L_jj
    if (st->code != 0) return;
    const int k = blockIdx.x * NB, nb = min(NB, n - k), tid = threadIdx.x, i0 = tid / NB, j0 = tid % NB;
    T[i0][j0] = (i0 < nb && j0 <= i0) ? L[(int64_t)(k + i0) * ld + (k + j0)] : make_double2(0.0, 0.0);
    X[i0][j0] = make_double2(i0 == j0 && i0 < nb ? 1.0 : 0.0, 0.0);
    __syncthreads();
    if (tid < nb) rs[tid] = 1.0 / T[tid][tid].x;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        const int nX = (nb - 1 - j) * (j + 1);   // at most 8 x 8
        if (tid < nX) {
            const int i = j + 1 + tid / (j + 1), c = tid % (j + 1);
            const double2 a = T[i][j], b = X[j][c];
            const double mx = a.x * rs[j], my = a.y * rs[j];
            double2 x = X[i][c];
            x.x = fma(-mx, b.x, fma(my, b.y, x.x));
            x.y = fma(-mx, b.y, fma(-my, b.x, x.y));
            X[i][c] = x;
        }
        __syncthreads();
    }
    if (i0 < nb && j0 < nb)
        Linv[(int64_t)(k + i0) * ld + (k + j0)] =
            j0 <= i0 ? make_double2(X[i0][j0].x * rs[i0], X[i0][j0].y * rs[i0]) : make_double2(0.0, 0.0);
}

// One level of the triangular inverse for blocks of up to kMergeMax rows, all pairs in one launch (blockIdx.y): C (M x
// N) = alpha A B with A row-major (lda), B row-major (ldb), complex128, 16 x 8 outputs a CTA, one a thread, K in chunks
// of 16 through shared memory, the next chunk loaded while this one is used. LEFT: A is lower triangular (k up to the
// tile's last row), else B is (k from the tile's first column on). The longest tiles come first. An output's terms are
// added in the order of the general GEMM with tiles of edge `tile` and `splits` partial sums over its K range
// (zgemm_shape: splits only at 128 rows): same bits, and M^-1 keeps its last ones (see chol_step). Bound by FP64 issue
// (64 clocks a warp instruction and SM quarter). A level of h rows has n / 2h pairs: the general GEMM's 32 x 32 tiles
// put h = 16 .. 128 on 8 to 32 CTAs and took 20, 39, 75 and 60 us a product at n = 512; these tiles put them on 32 to
// 256 CTAs and take 16 us on average.
constexpr int kMergeMax = 128;
template <bool LEFT, bool SPLIT>
__global__ void __launch_bounds__(128) tri_merge(const double2 *A, int64_t lda, int64_t bsa, const double2 *B, int64_t ldb,
                                                 int64_t bsb, double2 *C, int64_t ldc, int64_t bsc, int M, int N, int K,
                                                 double alpha, int tile, int splits, const DeviceStatus *st)
{
    __shared__ double2 As[NB][NB + 1];
    __shared__ double2 Bs[NB][NB / 2 + 1];
    if (st->code != 0) return;
    A += blockIdx.y * bsa;
    B += blockIdx.y * bsb;
    C += blockIdx.y * bsc;
    const int tm = (M + NB - 1) / NB, tn = (N + NB / 2 - 1) / (NB / 2);
    // LEFT: the last rows first; else the first columns first
    const int m0 = (LEFT ? tm - 1 - (int)blockIdx.x / tn : (int)blockIdx.x % tm) * NB;
    const int n0 = (LEFT ? (int)blockIdx.x % tn : (int)blockIdx.x / tm) * (NB / 2);
    const int kb = LEFT ? 0 : n0 / NB * NB, ke = LEFT ? min(K, m0 + NB) : K;   // zeros of the triangle left out
    // SPLIT: the general GEMM's K range of this tile and its partial sums; the next one begins at `cut` (a multiple of
    // 8)
    int chunk = 0, cut = 0;
    if (SPLIT) {
        const int t0 = (LEFT ? m0 : n0) / tile * tile, gb = LEFT ? 0 : t0, ge = LEFT ? min(K, t0 + tile) : K;
        chunk = ((ge - gb + splits - 1) / splits + 7) / 8 * 8;
        cut = gb + ((kb - gb) / chunk + 1) * chunk;
    }
    const int tid = threadIdx.x, i = tid >> 3, j = tid & 7;
    const double2 zero = make_double2(0.0, 0.0);
    double2 a[2], b;
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int r = m0 + (tid >> 4) + 8 * q, k = k0 + (tid & 15);
            a[q] = r < M && k < ke ? A[(int64_t)r * lda + k] : zero;
        }
        const int k = k0 + i;
        b = k < ke && n0 + j < N ? B[(int64_t)k * ldb + n0 + j] : zero;
    };
    load(kb);
    double2 acc = zero, sum = zero;
    for (int k0 = kb; k0 < ke; k0 += NB) {
        As[tid >> 4][tid & 15] = a[0];
        As[(tid >> 4) + 8][tid & 15] = a[1];
        Bs[i][j] = b;
        __syncthreads();
        if (k0 + NB < ke) load(k0 + NB);
#pragma unroll
        for (int h = 0; h < NB; h += 8) {
            if (SPLIT && k0 + h == cut) {
                sum.x += acc.x;
                sum.y += acc.y;
                acc = zero;
                cut += chunk;
            }
#pragma unroll
            for (int l = h; l < h + 8; ++l) {
                const double2 x = As[i][l], y = Bs[l][j];
                acc.x = fma(-x.y, y.y, fma(x.x, y.x, acc.x));
                acc.y = fma(x.y, y.x, fma(x.x, y.y, acc.y));
            }
        }
        __syncthreads();
    }
    if (SPLIT) acc = make_double2(sum.x + acc.x, sum.y + acc.y);
    if (m0 + i < M && n0 + j < N) C[(int64_t)(m0 + i) * ldc + n0 + j] = make_double2(alpha * acc.x, alpha * acc.y);
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
isdf_status product(ZGemm g, double2 *part, size_t part_n, const isdf_plan *tp, cudaStream_t st)
{
    g.stepwise = tp->mode == ISDF_MIXED;
    if (tp->use_oz && (int64_t)g.M * g.N * (g.batch > 1 ? g.batch : 1) >= (int64_t)256 * 256 && g.K >= 256 &&
        oz_fits(g, tp->oz))
        return oz_zgemm(g, tp->oz, tp->oz_err, st);
    return zgemm_auto(g, part, part_n, st);
}

// L^-1: the inverted diagonal blocks (NB wide), then aligned groups of blocks merged
// bottom-up: at each level, every pair (left group
// of h rows at o, right group of r <= h rows at o + h) gets
//   tmp = L[o+h:, o:o+h] Linv[o:o+h, o:o+h],  Linv[o+h:, o:o+h] = -Linv[o+h:, o+h:] tmp,
// all full pairs of a level in one batched launch each, a ragged last pair apart.
isdf_status tri_inv(const double2 *L, double2 *Linv, double2 *tmp, int64_t ld, int n, double2 *part,
                    size_t part_n, const isdf_plan *tp, DeviceStatus *status, cudaStream_t st)
{
    const int nblk = (n + NB - 1) / NB;
    inv_diag<<<nblk, EW, 0, st>>>(L, ld, Linv, n, status);
    isdf_note_launch();
    ISDF_LAUNCH_CHECK();
    // the pairs of a level whose right groups have r rows: L21, L11^-1 and L22^-1, (L^-1)21 at o, `pairs` of them
    auto merge = [&](int o, int h, int r, int pairs) -> isdf_status {
        const double2 *L21 = L + (int64_t)(o + h) * ld + o, *I11 = Linv + (int64_t)o * (ld + 1);
        const double2 *I22 = Linv + (int64_t)(o + h) * (ld + 1);
        double2 *I21 = Linv + (int64_t)(o + h) * ld + o;
        const int64_t step = (int64_t)2 * h * (ld + 1);   // from one pair's diagonal block to the next
        ZGemm g1 = single(r, h, h, op(L21, ld, 1, 0), op(I11, ld, 1, 0), tmp, h, 1.0, 0);
        g1.kmode = ZG_K_FROM_N0;   // L11^-1 lower: k >= n
        ZGemm g2 = single(r, h, r, op(I22, ld, 1, 0), op(tmp, h, 1, 0), I21, ld, -1.0, 0);
        g2.k_to_m_end = 1;         // L22^-1 lower: k <= m
        g1.batch = g2.batch = pairs;
        g1.bsa = g1.bsb = g2.bsa = g2.bsc = step;
        g1.bsc = g2.bsb = (int64_t)h * h;
        if (h <= kMergeMax) {
            zgemm_shape(g1, part != nullptr, part_n);
            zgemm_shape(g2, part != nullptr, part_n);
            const dim3 g((unsigned)(((r + NB - 1) / NB) * ((h + NB / 2 - 1) / (NB / 2))), (unsigned)pairs);
            const auto right = g1.splits > 1 ? tri_merge<false, true> : tri_merge<false, false>;
            const auto left = g2.splits > 1 ? tri_merge<true, true> : tri_merge<true, false>;
            right<<<g, 128, 0, st>>>(L21, ld, step, I11, ld, step, tmp, h, (int64_t)h * h, r, h, h, 1.0, g1.tile, g1.splits,
                                     status);
            left<<<g, 128, 0, st>>>(I22, ld, step, tmp, h, (int64_t)h * h, I21, ld, step, r, h, r, -1.0, g2.tile, g2.splits,
                                    status);
            isdf_note_launch();
            isdf_note_launch();
            ISDF_LAUNCH_CHECK();
            return ISDF_OK;
        }
        ISDF_TRY(product(g1, part, part_n, tp, st));
        return product(g2, part, part_n, tp, st);
    };
    for (int g = 1; g < nblk; g *= 2) {
        const int h = g * NB, full = n / (2 * h);
        if (full > 0) ISDF_TRY(merge(0, h, h, full));
        const int o = full * 2 * h, r = n - o - h;
        if (r > 0) ISDF_TRY(merge(o, h, r, 1));
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
        // 4 rows a panel CTA (one warp a quarter of the SM) while that leaves more than half of the SMs to the trailing
        // update, else 8
        const int rpc = rows <= 256 ? 4 : 8;
        const int n_panel = rows > 0 ? ((rows + rpc - 1) / rpc < kSms ? (rows + rpc - 1) / rpc : kSms) : 1;
        const int per = (rows + n_panel - 1) / n_panel;
        const int nt = k >= 0 ? (rows + NB - 1) / NB : 0, n_tiles = nt * (nt + 1) / 2;
        // one CTA per SM (a second one slows the panel's chain down) until the tiles are several per SM
        const int room = n_tiles > 8 * kSms ? 3 * kSms : kSms;
        int grid = n_panel + n_tiles < room ? n_panel + n_tiles : room;
        if (grid < n_panel) grid = n_panel;
        if (k < 0)   // the launch before may be a copy
            chol_step<<<grid, DT, 0, stream>>>(L, ld, M0, k, k1, nb1, rows, n_panel, per > 0 ? per : 1, ctr + k1 / NB, st);
        else
            ISDF_CUDA_TRY(launch_chained(chol_step, grid, DT, stream, L, ld, M0, k, k1, nb1, rows, n_panel,
                                         per > 0 ? per : 1, ctr + k1 / NB, st));
        isdf_note_launch();
        ISDF_LAUNCH_CHECK();
    }
    return ISDF_OK;
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
        return tri_inv(L + (int64_t)o * (ld + 1), Linv + (int64_t)o * (ld + 1), tmp, ld, m, part, part_n, tp, st, stream);
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
        ISDF_LAUNCH_CHECK();
        timer_stop(tp, 3, stream, n);
        timer_start(tp, 4, stream);
        ISDF_TRY(tri_inv(L, Linv, tmp, ld, n, part, part_n, tp, st, stream));
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
