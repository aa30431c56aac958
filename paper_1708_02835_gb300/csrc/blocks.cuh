// FP64 dense-block device routines shared by the single-problem and the
// batched drivers (included by several translation units; no relocatable
// device code needed).  Every routine is executed by a whole CTA of 256
// threads unless stated otherwise.
#pragma once
#include "egs_internal.cuh"

namespace egs {

constexpr int kPW = 16;  // panel width inside the single-CTA POTRF
constexpr int kIB = 64;  // sub-panel width of the blocked diagonal POTRF

__device__ __forceinline__ bool failed(const DevStatus *st)
{
    return *(volatile const unsigned long long *)&st->fail_index != kNoFail;
}

__device__ __forceinline__ void tri_decode(int64_t t, int &i, int &j)
{
    int ii = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while ((int64_t)ii * (ii + 1) / 2 > t) --ii;
    while ((int64_t)(ii + 1) * (ii + 2) / 2 <= t) ++ii;
    i = ii;
    j = (int)(t - (int64_t)ii * (ii + 1) / 2);
}

// ---------------------------------------------------------------------------
// Cholesky of a 64 x 64 block at A (row stride ld) held in shared memory for
// the whole factorisation (one global read and one write of the block): one
// CTA of 256 threads, right-looking over four 16-column panels -- warp 0
// factors the 16 x 16 diagonal block with warp synchronisation only, each row
// below it is solved by one thread, and the trailing lower triangle takes a
// rank-16 update (one 16-term dot product per entry) -- so the block needs 12
// CTA barriers, and its FP64 work is mostly independent FMAs.  Pivots are
// applied through 1 / sqrt(d) (one reciprocal square root per column, then
// multiplications).  A pivot that is not positive records row0 + its row in
// st->fail_index and returns false; the strict upper triangle is zeroed.
// ---------------------------------------------------------------------------
struct Potrf64Smem {
    double S[64][65];
    double rd[64];  // 1 / L_jj
    int fail_j;
};

__device__ __forceinline__ bool potrf64_smem_s(Potrf64Smem &sm, double *A, int ld, int64_t row0, DevStatus *st)
{
    constexpr int NB = 64;
    double(&S)[NB][NB + 1] = sm.S;
    int &fail_j = sm.fail_j;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) fail_j = -1;
    for (int e = tid; e < NB * NB; e += 256) {
        const int i = e / NB, j = e % NB;
        S[i][j] = (j <= i) ? A[(size_t)i * ld + j] : 0.0;
    }
    __syncthreads();
    for (int p0 = 0; p0 < NB; p0 += kPW) {
        // 1. the 16 x 16 diagonal block, column by column, by warp 0 (lane i < 16 owns row p0 + i)
        if (tid < 32) {
            for (int j = 0; j < kPW; ++j) {
                // every lane forms 1 / sqrt(d) (a warp-wide FP64 instruction
                // costs the same for one lane or 32), so the column is scaled
                // by a multiplication instead of a division
                const double d = S[p0 + j][p0 + j];
                if (!(d > 0.0)) {
                    if (lane == 0) fail_j = p0 + j;
                    break;
                }
                const double rs = rsqrt(d);
                __syncwarp();
                if (lane == j) {
                    S[p0 + j][p0 + j] = d * rs;
                    sm.rd[p0 + j] = rs;
                }
                if (lane > j && lane < kPW) S[p0 + lane][p0 + j] *= rs;
                __syncwarp();
                if (lane > j && lane < kPW) {
                    const double lij = S[p0 + lane][p0 + j];
                    for (int l = j + 1; l <= lane; ++l) S[p0 + lane][p0 + l] -= lij * S[p0 + l][p0 + j];
                }
                __syncwarp();
            }
        }
        __syncthreads();
        if (fail_j >= 0) {
            if (tid == 0) atomicMin(&st->fail_index, (unsigned long long)(row0 + fail_j));
            return false;
        }
        const int q0 = p0 + kPW;
        // 2. rows below the panel: x L_pp^T = row, one thread per row
        if (tid < NB - q0) {
            const int i = q0 + tid;
            double x[kPW];
#pragma unroll
            for (int j = 0; j < kPW; ++j) {
                double v = S[i][p0 + j];
#pragma unroll
                for (int l = 0; l < j; ++l) v -= x[l] * S[p0 + j][p0 + l];
                x[j] = v * sm.rd[p0 + j];
            }
#pragma unroll
            for (int j = 0; j < kPW; ++j) S[i][p0 + j] = x[j];
        }
        __syncthreads();
        // 3. rank-16 update of the trailing lower triangle (rows and columns q0..NB-1)
        const int m = NB - q0;
        for (int e = tid; e < m * m; e += 256) {
            const int i = q0 + e / m, l = q0 + e % m;
            if (l <= i) {
                double acc = 0.0;
#pragma unroll
                for (int j = 0; j < kPW; ++j) acc = fma(S[i][p0 + j], S[l][p0 + j], acc);
                S[i][l] -= acc;
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < NB * NB; e += 256) {
        const int i = e / NB, j = e % NB;
        A[(size_t)i * ld + j] = (j <= i) ? S[i][j] : 0.0;
    }
    return true;
}

__device__ __forceinline__ bool potrf64_smem(double *A, int ld, int64_t row0, DevStatus *st)
{
    __shared__ Potrf64Smem sm;
    return potrf64_smem_s(sm, A, ld, row0, st);
}

// ---------------------------------------------------------------------------
// Cholesky of a 64 x 64 block by one CTA of 256 threads, with the right-hand side (z, may be
// NULL) carried along as a 65th row, so that it leaves as y = L^-1 z.
//
// Bound by the FP64 pipe's issue rate within one SM: a warp-wide FP64 instruction occupies
// its sub-partition for 64 clocks whether 1 or 32 lanes are active (measured; a dependent one
// can follow at once), so what counts is the number of FP64 instructions on the longest
// sub-partition, not latency:
//  - L D L^T (no square root between pivots): with y ~ 1 / d from the hardware's approximation,
//    e = 1 - d y, the column a / d = a y (1 + e + e^2) (Newton's iteration one order up) costs
//    four instructions; the square roots are taken for all 64 columns at the end.  A pivot whose
//    reciprocal leaves the normal doubles is divided by instead;
//  - panels of 4 columns: warps 0 .. 2 each factor the 4 x 4 block in lanes 0 .. 3, redundantly
//    (each has a sub-partition of its own), while lanes 4 .. 31 carry 28 rows below it, so that
//    the rows below cost no instruction;
//  - the 4-term updates of the entries right of the panel are spread over all lanes, those of
//    the next panel's columns at once, the others while the next panel is factored.
// 64 pivots x 22 / 4 instructions of panels, about 400 of updates: 43 us with the launch (115 us
// with 16-column panels, a thread per row below them and a square root per pivot).
//
// Leaves L (zero upper half), y in row 64 and 1 / L_jj in sm; false if a pivot is not positive and
// finite (its row is recorded as row0 + j).
// ---------------------------------------------------------------------------
struct Chol64Smem {
    double S[65][65];
    double W[2][65][5];  // a / d of the columns of this panel and the one before
    double rd[64];
    int fail_j, claim;
};

// Positive with a biased exponent of 2 .. 2044: 1 / d and its approximation are normal numbers too.
__device__ __forceinline__ bool recip_normal(double d)
{
    return (unsigned)__double2hiint(d) - 0x00200000u < 0x7FB00000u;
}

// 1 / sqrt(d), d > 0: the hardware's approximation and one step of Householder's third-order
// iteration.
__device__ __forceinline__ double rsqrt_iter(double d)
{
    if (!recip_normal(d)) return 1.0 / sqrt(d);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-(d * y), y, 1.0);
    return fma(fma(e, 0.375, 0.5), y * e, y);
}

__device__ __forceinline__ bool chol64_s(Chol64Smem &sm, const double *A, int ld, const double *z, int64_t row0,
                                         DevStatus *st)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int e = tid + 256 * q;
        v[q] = (e & 63) <= (e >> 6) ? A[(size_t)(e >> 6) * ld + (e & 63)] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) sm.S[(tid + 256 * q) >> 6][tid & 63] = v[q];
    if (z && tid < 64) sm.S[64][tid] = z[tid];
    if (tid == 0) {
        sm.fail_j = -1;
        sm.claim = 0;
    }
    __syncthreads();
    const int zr = z ? 1 : 0;
#pragma unroll 1
    for (int p0 = 0; p0 < 64; p0 += 4) {
        double(&W)[65][5] = sm.W[(p0 >> 2) & 1];
        const double(&Wp)[65][5] = sm.W[((p0 >> 2) & 1) ^ 1];
        const int q0 = p0 + 4, m = 64 - q0;  // rows and columns left
        double a[4];
        if (28 * warp < m + zr || warp == 0) {
            const int t = 28 * warp + lane - 4;  // index among the rows below, z the last
            const int i = lane < 4 ? p0 + lane : (t < m ? q0 + t : 64);
            double w[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) a[c] = sm.S[i][p0 + c];
            bool ok = true;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double d = __shfl_sync(0xffffffffu, a[j], j);
                if (recip_normal(d)) {
                    double y;
                    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
                    const double e = fma(-d, y, 1.0);
                    const double ay = a[j] * y, u = fma(e, e, e);
                    w[j] = fma(ay, u, ay);
                } else {
                    if (ok && !(d > 0.0 && d < __longlong_as_double(0x7FF0000000000000ll))) {
                        ok = false;
                        if (tid == 0) sm.fail_j = p0 + j;
                    }
                    w[j] = a[j] / d;
                }
#pragma unroll
                for (int c = j + 1; c < 4; ++c) a[c] = fma(-a[j], __shfl_sync(0xffffffffu, w[j], c), a[c]);
            }
            if (lane >= 4 && t < m + zr) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sm.S[i][p0 + c] = a[c];
                    W[i][c] = w[c];
                }
            }
        }
        // the columns right of this panel by the panel before, 64 entries at a time to whichever
        // warp is free: lower triangle from q0 on, then the z row (the triangle's next row but for
        // its last entry)
        if (p0 > 0) {
            const int cnt = m * (m + 1) / 2 + (zr ? m : 0);
            for (;;) {
                int base = 0;
                if (lane == 0) base = atomicAdd(&sm.claim, 64);
                base = __shfl_sync(0xffffffffu, base, 0);
                if (base >= cnt) break;
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const int e = base + 32 * h2 + lane;
                    if (e < cnt) {
                        int ii = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                        if (ii * (ii + 1) / 2 > e) --ii;
                        if ((ii + 1) * (ii + 2) / 2 <= e) ++ii;
                        const int i = ii < m ? q0 + ii : 64, c = q0 + e - ii * (ii + 1) / 2;
                        double acc = sm.S[i][c];
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc = fma(-sm.S[i][p0 - 4 + j], Wp[c][j], acc);
                        sm.S[i][c] = acc;
                    }
                }
            }
        }
        __syncthreads();
        if (tid < 4) {  // only now: every warp has read the block
#pragma unroll
            for (int c = 0; c < 4; ++c) sm.S[p0 + tid][p0 + c] = a[c];
        }
        if (sm.fail_j >= 0) {
            if (tid == 0) atomicMin(&st->fail_index, (unsigned long long)(row0 + sm.fail_j));
            return false;
        }
        // the next panel's four columns by this one
        if (tid == 0) sm.claim = 0;
        const int ri = tid >> 2, c = q0 + (tid & 3), i = ri < m ? q0 + ri : 64;
        if (m > 0 && ri < m + zr && i >= c) {
            double acc = sm.S[i][c];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc = fma(-sm.S[i][p0 + j], W[c][j], acc);
            sm.S[i][c] = acc;
        }
        __syncthreads();
    }
    if (tid < 64) {
        const double r = rsqrt_iter(sm.S[tid][tid]);
        sm.rd[tid] = r;
    }
    __syncthreads();
    const int jc = tid & 63;
    const double rj = sm.rd[jc];
    for (int i = tid >> 6; i < 64 + zr; i += 4) sm.S[i][jc] = jc <= i ? sm.S[i][jc] * rj : 0.0;
    __syncthreads();
    return true;
}

// The inverses of L's eight 8 x 8 diagonal blocks into winv (row-major, 64 p on), column c of
// block p by thread 8 p + c (forward substitution); sm as chol64_s left it.
constexpr int kWinvDoubles = 8 * 8 * 8;
__device__ __forceinline__ void inv8_blocks(const Chol64Smem &sm, double *winv)
{
    const int tid = threadIdx.x;
    if (tid >= 64) return;
    const int p = tid >> 3, c = tid & 7, q0 = 8 * p;
    double w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = i == c ? 1.0 : 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        w[i] *= sm.rd[q0 + i];
#pragma unroll
        for (int l = i + 1; l < 8; ++l) w[l] = fma(-sm.S[q0 + l][q0 + i], w[i], w[l]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) winv[p * 64 + i * 8 + c] = w[i];
}

// Diagonal block j of a tile (A: its corner, row stride ld; `right` columns of the tile to its
// right, zeroed): chol64_s and the write-back of L, y and the inverses.  256 threads.
__device__ __forceinline__ bool diag64_block(Chol64Smem &sm, double *A, int ld, int right, double *z, double *winv,
                                             int64_t row0, DevStatus *st)
{
    const int tid = threadIdx.x;
    if (!chol64_s(sm, A, ld, z, row0, st)) return false;
    inv8_blocks(sm, winv);
    if (z && tid < 64) z[tid] = sm.S[64][tid];
    for (int e = tid; e < 64 * 64; e += 256) A[(size_t)(e >> 6) * ld + (e & 63)] = sm.S[e >> 6][e & 63];
    for (int r = tid >> 5; r < 64; r += 8)
        for (int c = tid & 31; c < right; c += 32) A[(size_t)r * ld + 64 + c] = 0.0;
    return true;
}

// X L^T = A for RB rows of 64 columns by 8 RB threads, L a 64 x 64 diagonal block: thread (row, c)
// has column c of each 8-column block, X_p = (A_p - sum_{i<p} X_i L_pi^T) W_p^T with the
// inverses W_p of L's 8 x 8 diagonal blocks.  FP64-pipe bound: 288 FMAs a thread at 64 clocks a
// warp and sub-partition, 9 us for one warp on each (RB = 16), 18 us for two.
template <int RB>
struct Solve64Smem {
    double Ls[56][57];  // L below its 8 x 8 diagonal blocks: rows 8 .. 63, columns 0 .. 55
    double Xs[RB][65];
    double Ws[64][9];
};

template <int RB>
__device__ __forceinline__ void solve64_stage(Solve64Smem<RB> &sm, const double *L, int ld, const double *winv)
{
    constexpr int NT = 8 * RB;
    const int tid = threadIdx.x;
#pragma unroll 16
    for (int e = tid; e < 64 * 64; e += NT) {
        const int r = e >> 6, c = e & 63;
        if (r >= 8 && c < 56 && c < r) sm.Ls[r - 8][c] = L[(size_t)r * ld + c];
    }
    for (int e = tid; e < kWinvDoubles; e += NT) sm.Ws[e >> 3][e & 7] = winv[e];
}

// Xs holds A on entry and X on return; barriers around it are the caller's.
template <int RB>
__device__ __forceinline__ void solve64_rows(Solve64Smem<RB> &sm)
{
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        double r = sm.Xs[ty][8 * p + tx];
#pragma unroll 8
        for (int l = 0; l < 8 * p; ++l) r = fma(-sm.Xs[ty][l], sm.Ls[8 * (p - 1) + tx][l], r);
        // a row's 8 entries belong to 8 lanes of one warp
        __syncwarp();
        sm.Xs[ty][8 * p + tx] = r;
        __syncwarp();
        double x = 0.0;
#pragma unroll
        for (int l = 0; l < 8; ++l) x = fma(sm.Xs[ty][8 * p + l], sm.Ws[8 * p + tx][l], x);
        __syncwarp();
        sm.Xs[ty][8 * p + tx] = x;
        __syncwarp();
    }
}

// A 16 x 16 sub-block of a panel's update by its 64-column block j (K = 64), one entry a thread of
// 256: columns c0 .. c0 + 15 of the rows at `row` minus X_row X_col^T, X in columns 64 j .. 64 j + 63 of
// the rows at `row` and `col` (row stride b).  4.3 us of FP64 pipe.
__device__ __forceinline__ void inner16(double (&As)[16][65], double (&Bs)[16][65], double *row, const double *col, int b,
                                        int j, int c0)
{
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int e = tid; e < 16 * 64; e += 256) {
        As[e >> 6][e & 63] = row[(size_t)(e >> 6) * b + j * 64 + (e & 63)];
        Bs[e >> 6][e & 63] = col[(size_t)(e >> 6) * b + j * 64 + (e & 63)];
    }
    double *C = row + (size_t)ty * b + c0 + tx;
    const double c = *C;
    __syncthreads();
    double acc = 0.0;
#pragma unroll 8
    for (int l = 0; l < 64; ++l) acc = fma(As[ty][l], Bs[tx][l], acc);
    *C = c - acc;
}

// X_row . y over 64 columns, two per lane (y0, y1: the lane's entries of y); the sum in lane 0.
__device__ __forceinline__ double dot64(double x0, double x1, double y0, double y1)
{
    double v = fma(x0, y0, x1 * y1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// ---------------------------------------------------------------------------
// C (32 x 32, row stride ldc) -= Am (32 x K) An (32 x K)^T; 2 x 2 outputs per
// thread (rows ty + 16 i, columns tx + 16 j).  FP64 or FP32 operands, FP64
// arithmetic.  256 threads.
// ---------------------------------------------------------------------------
struct Gemm32Smem {
    double As[kPW][33];
    double Bs[kPW][33];
};

template <typename EA, typename EB>
__device__ __forceinline__ void gemm_sub32_s(Gemm32Smem &sm, const EA *Am, int lda, const EB *An, int ldb, int K,
                                             double *C, int ldc)
{
    double(&As)[kPW][33] = sm.As;
    double(&Bs)[kPW][33] = sm.Bs;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    for (int p = 0; p < K; p += kPW) {
        for (int e = tid; e < 32 * kPW; e += 256) {
            const int r = e >> 4, l = e & 15;
            As[l][r] = (double)Am[(size_t)r * lda + p + l];
            Bs[l][r] = (double)An[(size_t)r * ldb + p + l];
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < kPW; ++l) {
            const double a0 = As[l][ty], a1 = As[l][ty + 16], b0 = Bs[l][tx], b1 = Bs[l][tx + 16];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) C[(size_t)(ty + 16 * i) * ldc + tx + 16 * j] -= acc[i][j];
}

template <typename EA, typename EB>
__device__ __forceinline__ void gemm_sub32(const EA *Am, int lda, const EB *An, int ldb, int K, double *C, int ldc)
{
    __shared__ Gemm32Smem sm;
    gemm_sub32_s(sm, Am, lda, An, ldb, K, C, ldc);
}

// ---------------------------------------------------------------------------
// X L^T = A for RB rows (RB in {16, 64}): X and A at Xp (row stride ldx,
// ncols columns), L lower ncols x ncols at Lp (row stride ldl).  32-column
// blocks: a GEMM-style update with the already-solved columns, then a
// 32-wide substitution in shared memory.  256 threads; fewer rows per CTA put
// more SMs on a panel when the panel is short.  TX =
// float: X and all arithmetic in FP32 (L rounded to FP32 as it is staged).
// ---------------------------------------------------------------------------
template <int RB, typename TX>
struct TrsmSmem {
    TX Xs[RB][kPW + 1];
    TX Ls[32][kPW + 1];
    TX Ab[RB][33];
    TX Ld[32][33];
};

template <int RB, typename TX = double>
__device__ __forceinline__ void trsm_rows_s(TrsmSmem<RB, TX> &sm, const double *Lp, int ldl, TX *Xp, int ldx,
                                            int ncols)
{
    constexpr int RPG = RB / 8;  // rows per thread group (8 groups of 32 threads)
    TX(&Xs)[RB][kPW + 1] = sm.Xs;
    TX(&Ls)[32][kPW + 1] = sm.Ls;
    TX(&Ab)[RB][33] = sm.Ab;
    TX(&Ld)[32][33] = sm.Ld;
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    for (int c0 = 0; c0 < ncols; c0 += 32) {
        TX acc[RPG];
#pragma unroll
        for (int i = 0; i < RPG; ++i) acc[i] = Xp[(size_t)(ty * RPG + i) * ldx + c0 + tx];
        for (int p = 0; p < c0; p += kPW) {
            for (int e = tid; e < RB * kPW; e += 256) {
                const int r = e >> 4, l = e & 15;
                Xs[r][l] = Xp[(size_t)r * ldx + p + l];
            }
            for (int e = tid; e < 32 * kPW; e += 256) {
                const int c = e >> 4, l = e & 15;
                Ls[c][l] = (TX)Lp[(size_t)(c0 + c) * ldl + p + l];
            }
            __syncthreads();
#pragma unroll
            for (int l = 0; l < kPW; ++l) {
                const TX lv = Ls[tx][l];
#pragma unroll
                for (int i = 0; i < RPG; ++i) acc[i] = fma(-Xs[ty * RPG + i][l], lv, acc[i]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < RPG; ++i) Ab[ty * RPG + i][tx] = acc[i];
        for (int e = tid; e < 32 * 32; e += 256) {
            const int r = e >> 5, c = e & 31;
            Ld[r][c] = (c <= r) ? (TX)Lp[(size_t)(c0 + r) * ldl + c0 + c] : (TX)0;
        }
        __syncthreads();
        if (tid < RB) {
            for (int j = 0; j < 32; ++j) {
                TX s = Ab[tid][j];
                for (int l = 0; l < j; ++l) s -= Ab[tid][l] * Ld[j][l];
                Ab[tid][j] = s / Ld[j][j];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RPG; ++i) Xp[(size_t)(ty * RPG + i) * ldx + c0 + tx] = Ab[ty * RPG + i][tx];
        __syncthreads();
    }
}

template <int RB, typename TX = double>
__device__ __forceinline__ void trsm_rows(const double *Lp, int ldl, TX *Xp, int ldx, int ncols)
{
    __shared__ TrsmSmem<RB, TX> sm;
    trsm_rows_s<RB, TX>(sm, Lp, ldl, Xp, ldx, ncols);
}

// ---------------------------------------------------------------------------
// C (64 x 64, row stride ldc) -= Am (64 x K) An (64 x K)^T with row strides
// lda, ldb; the operands may be FP64 or FP32 and are converted to the
// accumulation type TC on staging (TC = double: FP64 products and sums of
// FP64 or FP32 operands; TC = float: an FP32 update of an FP32 tile).  4 x 4 outputs per thread (rows ty + 16 i, columns tx + 16 j, so a
// half-warp touches 128 contiguous bytes).  256 threads.
// ---------------------------------------------------------------------------
// Staging buffers of gemm_sub64, one set per accumulation type in a kernel
// (however many operand-type combinations it instantiates).
template <typename TC>
struct GemmSmem {
    TC As[kPW][65];
    TC Bs[kPW][65];
};
template <typename TC>
__device__ __forceinline__ GemmSmem<TC> &gemm_smem()
{
    __shared__ GemmSmem<TC> sm;
    return sm;
}

template <typename EA, typename EB, typename TC = double>
__device__ __forceinline__ void gemm_sub64_s(GemmSmem<TC> &sm, const EA *Am, int lda, const EB *An, int ldb, int K,
                                             TC *C, int ldc)
{
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    TC acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = (TC)0;
    for (int p = 0; p < K; p += kPW) {
        for (int e = tid; e < 64 * kPW; e += 256) {
            const int r = e >> 4, l = e & 15;
            sm.As[l][r] = (TC)Am[(size_t)r * lda + p + l];
            sm.Bs[l][r] = (TC)An[(size_t)r * ldb + p + l];
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < kPW; ++l) {
            TC a[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = sm.As[l][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = sm.Bs[l][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) C[(size_t)(ty + 16 * i) * ldc + tx + 16 * j] -= acc[i][j];
}

template <typename EA, typename EB, typename TC = double>
__device__ __forceinline__ void gemm_sub64(const EA *Am, int lda, const EB *An, int ldb, int K, TC *C, int ldc)
{
    gemm_sub64_s<EA, EB, TC>(gemm_smem<TC>(), Am, lda, An, ldb, K, C, ldc);
}

// Fixed-order tree reduction of one value per thread (any blockDim.x <= 1024).
// Returns the total (valid in every thread after the last barrier).
__device__ __forceinline__ double block_sum(double v, double *red)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    red[tid] = v;
    __syncthreads();
    int p2 = 1;
    while (p2 < nt) p2 <<= 1;
    for (int s = p2 >> 1; s > 0; s >>= 1) {
        if (tid < s && tid + s < nt) red[tid] += red[tid + s];
        __syncthreads();
    }
    return red[0];
}

// A tile's sums of log L_ii and y_i^2 into out[0] and out[stride]; red: 256 doubles, 256 threads.
__device__ __forceinline__ void logdet_quad_tile(const double *L, int b, const double *y, double *red, double *out,
                                                 size_t stride)
{
    double a = 0.0, q = 0.0;
    for (int i = threadIdx.x; i < b; i += 256) {
        a += log(L[(size_t)i * (b + 1)]);
        q = fma(y[i], y[i], q);
    }
    const double lsum = block_sum(a, red);
    __syncthreads();
    const double qsum = block_sum(q, red);
    if (threadIdx.x == 0) {
        out[0] = lsum;
        out[stride] = qsum;
    }
}

// Forward substitution on one diagonal tile: y = L^-1 r in place on v
// (b entries), blockDim.x = b threads (thread i owns row i).  32-column
// blocks: the owning warp solves its 32 x 32 block with shuffles, then every
// later row subtracts the block's contribution (32 consecutive entries of its
// own row of L).  If ld_q is not NULL, ld_q[0] = sum_i log L_ii and
// ld_q[1] = sum_i y_i^2 (fixed-order trees).
__device__ __forceinline__ void trsv_fwd_tile(const double *__restrict__ L, int b, double *__restrict__ v,
                                              double *ld_q)
{
    __shared__ double yv[1024];
    __shared__ double red[1024];
    __shared__ double D[32][33];
    const int i = threadIdx.x, lane = i & 31, w = i >> 5;
    const double *Li = L + (size_t)i * b;
    double r = v[i];
    for (int cb = 0; cb < b / 32; ++cb) {
        const int c0 = cb * 32;
        // stage the 32 x 32 diagonal block so the warp's serial solve reads
        // shared memory instead of global memory
        for (int e = i; e < 32 * 32; e += b) D[e >> 5][e & 31] = L[(size_t)(c0 + (e >> 5)) * b + c0 + (e & 31)];
        __syncthreads();
        if (w == cb) {
            for (int jj = 0; jj < 32; ++jj) {
                const double yj = __shfl_sync(0xffffffffu, r, jj) / D[jj][jj];
                if (lane == jj) yv[c0 + jj] = yj;
                if (lane > jj) r = fma(-D[lane][jj], yj, r);
            }
        }
        __syncthreads();
        if (i >= c0 + 32) {
            double s = 0.0;
#pragma unroll 8
            for (int jj = 0; jj < 32; ++jj) s = fma(Li[c0 + jj], yv[c0 + jj], s);
            r -= s;
        }
    }
    __syncthreads();
    const double y = yv[i];
    v[i] = y;
    if (ld_q) {
        const double ld = block_sum(log(Li[i]), red);
        __syncthreads();
        const double q = block_sum(y * y, red);
        if (i == 0) {
            ld_q[0] = ld;
            ld_q[1] = q;
        }
    }
}

// z_m[r] -= L_mk[r][:] . y for the 64 rows r0..r0+63 of one panel tile, one
// warp per 8 rows with a fixed shuffle tree.  ys: the b entries of y in
// shared memory.  256 threads.
template <typename E>
__device__ __forceinline__ void gemv_rows(const E *__restrict__ A, int b, int r0, const double *ys,
                                          double *__restrict__ out)
{
    // the warp's 8 rows are swept together (8 loads in flight per lane); each
    // row's sum keeps its order, so results equal a row-by-row sweep
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const E *rows = A + (size_t)(r0 + warp * 8) * b;
    double s[8];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) s[rr] = 0.0;
    for (int c = lane; c < b; c += 32) {
        const double y = ys[c];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) s[rr] = fma((double)rows[(size_t)rr * b + c], y, s[rr]);
    }
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        double v = s[rr];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) out[r0 + warp * 8 + rr] -= v;
    }
}

// Backward substitution on one diagonal tile: L^T x = r in place on v (b
// entries), blockDim.x = b (thread i owns row i).  32-column blocks from the
// last: the owning warp solves its 32 x 32 block with shuffles, then every
// thread with a smaller row index subtracts the block's contribution (L read
// along its rows).
__device__ __forceinline__ void trsv_bwd_tile(const double *__restrict__ L, int b, double *__restrict__ v)
{
    __shared__ double xv[1024];
    __shared__ double D[32][33];
    const int i = threadIdx.x, lane = i & 31, w = i >> 5;
    double r = v[i];
    for (int cb = b / 32 - 1; cb >= 0; --cb) {
        const int c0 = cb * 32;
        for (int e = i; e < 32 * 32; e += b) D[e >> 5][e & 31] = L[(size_t)(c0 + (e >> 5)) * b + c0 + (e & 31)];
        __syncthreads();
        if (w == cb) {
            for (int jj = 31; jj >= 0; --jj) {
                const double xj = __shfl_sync(0xffffffffu, r, jj) / D[jj][jj];
                if (lane == jj) xv[c0 + jj] = xj;
                if (lane < jj) r = fma(-D[jj][lane], xj, r);
            }
        }
        __syncthreads();
        if (i < c0) {
            double s = 0.0;
#pragma unroll 8
            for (int jj = 0; jj < 32; ++jj) s = fma(L[(size_t)(c0 + jj) * b + i], xv[c0 + jj], s);
            r -= s;
        }
    }
    __syncthreads();
    v[i] = xv[i];
}

__device__ __forceinline__ double col_dot(const double *__restrict__ A, int b, int c, int g, const double *xs,
                                          const float *)
{
    // eight independent partial sums (rows g + 4 u mod 32) keep eight loads
    // in flight; they are combined in a fixed order
    double s[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) s[u] = 0.0;
    for (int r = g; r < b; r += 32) {
#pragma unroll
        for (int u = 0; u < 8; ++u) s[u] = fma(A[(size_t)(r + 4 * u) * b + c], xs[r + 4 * u], s[u]);
    }
    return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

// Off-band (FP32) tiles: products and the partial sum in FP32 (the tile is
// only FP32 accurate; the refinement recovers the quadratic form in FP64).
__device__ __forceinline__ double col_dot(const float *__restrict__ A, int b, int c, int g, const double *,
                                          const float *xs32)
{
    float s[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) s[u] = 0.0f;
    for (int r = g; r < b; r += 32) {
#pragma unroll
        for (int u = 0; u < 8; ++u) s[u] = fmaf(A[(size_t)(r + 4 * u) * b + c], xs32[r + 4 * u], s[u]);
    }
    return (double)(((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7])));
}

// vj[c0 .. c0+63] -= (L_kj^T xk)[c0 .. c0+63] for one tile (FP64 or FP32):
// 64 columns x 4 row groups, reduced in a fixed order.  256 threads.
__device__ __forceinline__ void gemv_T_cols(const Tiles &tl, int k, int j, int c0, const double *xk, double *vj)
{
    __shared__ double xs[1024];
    __shared__ float xs32[1024];
    __shared__ double red[4][64];
    const int b = tl.b;
    const int tx = threadIdx.x & 63, g = threadIdx.x >> 6;
    for (int c = threadIdx.x; c < b; c += 256) {
        xs[c] = xk[c];
        xs32[c] = (float)xs[c];
    }
    __syncthreads();
    const double s = tl.is64(k, j) ? col_dot(tl.t64(k, j), b, c0 + tx, g, xs, xs32)
                                   : col_dot(tl.t32(k, j), b, c0 + tx, g, xs, xs32);
    red[g][tx] = s;
    __syncthreads();
    if (g == 0) vj[c0 + tx] -= ((red[0][tx] + red[1][tx]) + red[2][tx]) + red[3][tx];
}

// FP32 variant for the off-band tiles of the mixed-precision solves: the
// products and the row sum run in FP32 (the tile itself is only FP32
// accurate, and the quadratic form is recovered by the FP64 refinement); the
// FP32 row sum is subtracted from the FP64 residual.  ys32: y in FP32.
__device__ __forceinline__ void gemv_rows_f32(const float *__restrict__ A, int b, int r0, const float *ys32,
                                              double *__restrict__ out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float *rows = A + (size_t)(r0 + warp * 8) * b;
    float s[8];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) s[rr] = 0.0f;
    for (int c = lane; c < b; c += 32) {
        const float y = ys32[c];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) s[rr] = fmaf(rows[(size_t)rr * b + c], y, s[rr]);
    }
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        float v = s[rr];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) out[r0 + warp * 8 + rr] -= (double)v;
    }
}

}  // namespace egs
