// FP64 trailing update of the tile Cholesky (Section 5.2, SYRK / GEMM tasks) on
// the BF16 tensor cores: C_mn -= P_m P_n^T with FP64 operands and results, every
// product formed from exact BF16 slices (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59 (2012)).
//
// Why: GB300's FP64 pipe issues 2 FMAs per clock per SM (1.25 TFLOP/s for the chip;
// the DFMA update ran at 99% of it), its BF16 tensor cores about 4,096.  28 exact
// slice products per FP64 product still leave a factor of more than 30.
//
// Splitting.  A row x (length K) with |x| < 2^e is read as x = 2^(e-8) sum_i q_i 2^-8i,
// i = 0..6, with integer digits |q_0| <= 256, |q_i| <= 128 (balanced base 256, from the
// 57-bit fixed-point value rounded once), each exact in BF16.  For two rows
//   x . y = 2^(ex + ey - 16) sum_L 2^-8L sum_{i+j=L} q_i(x) . q_j(y)
// and the levels L = 0..6 (28 pairs) are kept.  The dropped ones and the rounding of the
// last digit amount to about 2^-53.8 sqrt(K / 512) of |x|_max |y|_max, below the rounding
// of a length-K chain of DFMAs.  That bound is relative to the rows' largest entries, i.e. to
// sqrt(a_mm a_nn), as Cholesky's backward error is; relative to |x| . |y| of the entry itself a
// DFMA chain keeps more where that is far smaller (n = 4,096, range 0.03: absolute error 8.5e-17 against
// 3.4e-16, relative to |x| . |y| up to 8e-4 against 3e-15), so entries of L far below
// sqrt(a_mm) have their digits relative to it and not to themselves.
// Each level has its own FP32 accumulator in TMEM, flushed to FP64 every K = 256 columns, and a sum
// of integers in units of its level is exact as long as it stays within 2^24 of them.  Over 256
// columns levels 0 and 1 always do.  With S the largest sum of |q_0| over such 256 columns in either
// row, level 2 is at most 128 * 2 S + 2^22 and level 3 at most 128 * 2 S + 2^23, so both are exact for
// S <= 32,768 = half of what 256 digits can sum to, which the rows of a covariance's factor keep far
// below.  The slicing marks the rows that do not; an output block with such a row is flushed every
// 128 columns, where every level up to 5 is within 2^24 whatever the digits (rows with all leading
// digits large, of one sign: off by 1.9e-9 of 250 without, 2.8e-14 so; n = 51,200 without such rows,
// all updates: 967 and 973 ms).  Of the levels from 4 on, the FP32 rounding over 256 columns is below
// 2^-50 of the level-0 range.
//
// Kernel: persistent, one CTA per SM, 320 threads, output blocks of 128 x 64.  A K chunk
// of 64 is 7 A boxes (128 rows) and one B box of all 7 slices (64 rows each, back to
// back).  A slice i multiplies B slices 0 .. 6-i in one or two MMAs (N <= 256) whose D
// address is shifted by 64 i columns, so the block of B slice j lands in level i + j:
// each A slice is read from shared memory once or twice per K step instead of once per
// pair; 128 x 64 with 7 x 64 accumulator columns is the largest block that fits TMEM.
// A slots are freed slice by slice (7 slots of 16 KB), B is double buffered (2 x 56 KB).
// What bounds it (ncu, n = 8,192, K = 512): the tensor pipe is busy 56% of the time and shared
// memory 48%; the rest is the A slices' single buffering, a slot being refilled 21 of 28 product
// units before its next use, and the epilogue before the accumulators are free.
// Measured (n = 16,900, tile 512, all 33 updates): 1,361 ms with DFMA, 40.8 ms here with FP64
// additions in the epilogue, 33 ms with integer ones, i.e. 53 TFLOP/s of FP64-equivalent work,
// 1,490 executed on the tensor cores.  Error of the factor, rms of Sigma - L L^T in twice the
// precision (n = 2,304, tile 256): 2.5e-17 against 3.2e-17 with DFMA (theta = (1, 0.1, 0.5)), 2.9e-17 / 6.3e-17 (nu = 1.3), 9.9e-18 / 1.0e-17
// (range 0.03).
#include "blocks.cuh"
#include "tc_common.cuh"
#include "tc64.cuh"

#include <cudaTypedefs.h>

namespace egs {

namespace {

constexpr int FM = 128, FN = 64, FKC = 64;  // output block and K chunk
constexpr int FA_SL = FM * 128, FB_SL = FN * 128;
constexpr int FB_BUF = kF64Slices * FB_SL;
constexpr int FSMEM = kF64Slices * FA_SL + 2 * FB_BUF + 1024;
constexpr int FTHREADS = 320;      // warp 0 TMA, warp 1 MMA, warps 2..9 epilogue
constexpr int FRING = 4;           // work items posted ahead by the producer
constexpr int FLUSH = 256 / FKC;   // K chunks per accumulator flush
constexpr int FLUSH_DENSE = 128 / FKC;  // with a dense row
static_assert(FLUSH == 4 && FLUSH_DENSE == 2, "powers of two, as the masks and shifts have them");
constexpr int kDenseSum = 32768;   // sum of |q_0| over 256 columns above which a row is dense
constexpr uint32_t FTMEM = 512;
constexpr int kBadRow = 1 << 20;   // exponent of a row holding an infinity or a NaN

// ---- slicing ----------------------------------------------------------------

// 57-bit fixed point of x relative to 2^e (|x| < 2^e): rint(x 2^(56 - e)), ties away.
__device__ __forceinline__ long long fixed57(double x, int e)
{
    const long long bits = __double_as_longlong(x);
    int ex = (int)((bits >> 52) & 0x7FF);
    long long m = bits & 0xFFFFFFFFFFFFFll;
    if (ex) m |= 0x10000000000000ll;
    else ex = 1;
    const int sh = 1019 + e - ex;  // >= -3
    long long f;
    if (sh <= 0) f = m << (-sh);
    else if (sh < 56) f = (m + (1ll << (sh - 1))) >> sh;
    else f = 0;
    return bits < 0 ? -f : f;
}

// The seven digits of f (balanced base 256) as BF16 bit patterns q_i 2^-8i; returns |q_0|.
__device__ __forceinline__ int digits7(long long f, uint32_t (&d)[kF64Slices])
{
    int lead = 0;
#pragma unroll
    for (int i = kF64Slices - 1; i >= 0; --i) {
        int q;
        if (i > 0) {
            q = (int)(signed char)(f & 0xFF);
            f = (f - q) >> 8;
        } else {
            q = (int)f;
            lead = abs(q);
        }
        const float v = __int_as_float(0x4B400000 + q) - 12582912.0f;  // (float)q, |q| <= 256
        d[i] = __float_as_uint(v * __int_as_float((127 - 8 * i) << 23)) >> 16;  // exact: 8 significant bits
    }
    return lead;
}

// One warp slices one row of b doubles (b <= 1024, a multiple of 64): slice i of the row
// to dst[i * stride + c], the exponent to *ep, whether it is dense to *dense (and into *any).  Lanes
// take two consecutive columns.
__device__ __forceinline__ void slice7_row(const double *__restrict__ src, int b, uint16_t *__restrict__ dst,
                                           size_t stride, int *ep, uint8_t *dense, unsigned long long *any)
{
    const int lane = threadIdx.x & 31;
    unsigned mh = 0;
    for (int c = 2 * lane; c < b; c += 64) {
        const double2 v = make_double2(src[c], src[c + 1]);
        const unsigned h0 = (unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, h1 = (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu;
        mh = max(mh, max(h0, h1));
    }
    mh = __reduce_max_sync(0xffffffffu, mh);
    const int emax = (int)(mh >> 20);
    const bool bad = emax == 0x7FF;
    const int e = mh == 0 ? 0 : max(emax, 1) - 1022;
    if (lane == 0) *ep = bad ? kBadRow : e;
    int lead = 0, most = 0;  // sum of |q_0| over the 256 columns at hand, the largest so far
    for (int c = 2 * lane; c < b; c += 64) {
        const double2 v = make_double2(src[c], src[c + 1]);
        uint32_t d0[kF64Slices], d1[kF64Slices];
        lead += digits7(bad || mh == 0 ? 0ll : fixed57(v.x, e), d0);
        lead += digits7(bad || mh == 0 ? 0ll : fixed57(v.y, e), d1);
#pragma unroll
        for (int i = 0; i < kF64Slices; ++i)
            *reinterpret_cast<uint32_t *>(dst + (size_t)i * stride + c) = d0[i] | (d1[i] << 16);
        if ((c >> 6 & 3) == 3 || c + 64 >= b) {
            most = max(most, __reduce_add_sync(0xffffffffu, lead));
            lead = 0;
        }
    }
    if (lane == 0) {
        *dense = most > kDenseSum;
        if (most > kDenseSum) atomicOr(any, 1ull);
    }
}

// Panel rows of step k (tiles m0 .. T - 1 of column k) -> slices; one warp per row.
// Memory bound: 8 bytes read (twice, the second time from L1 / L2) and 14 written per entry.
// src: 0 the tiles of column k; 1 the band rows' Y; 2 the rows of L_kk, into their own slices.
__global__ void __launch_bounds__(256) k_slice_panel64(const __grid_constant__ F64Set set, int k, int src)
{
    const F64Prob &P = set.get(blockIdx.y);
    const Tiles &tl = P.tl;
    const int b = tl.b;
    const int64_t pr = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if ((src != 2 && pr >= (int64_t)(tl.T - 1 - k) * b) || failed(P.st)) return;
    const F64Rows &to = src == 2 ? P.l : P.panel;
    const size_t r = to.row0 + pr;
    const double *x = src == 0 ? tl.t64(k + 1 + (int)(pr / b), k) + (pr % b) * b : (src == 1 ? P.y : tl.t64(k, k)) + pr * b;
    slice7_row(x, b, to.sl + r * b, to.rows * b, to.ex + r, to.dense + r, P.ctr + tc64_dense_slot(b, k));
}

// ---- the panel ----------------------------------------------------------------
//
// Tile column k is factored in 64-column blocks, each in three launches:
//   k_diag64    L_jj = chol of the 64 x 64 diagonal block and the inverses of its eight
//               8 x 8 diagonal blocks, one CTA;
//   k_solve64   the rows below, in the tile and in every tile under it: X L_jj^T = A by
//               8-column blocks, X_p = (A_p - sum_{i<p} X_i L_pi^T) L_pp^-T, and X's slices
//               (K = 64, exponents of their own);
//   k_tc_f64    the update of the panel's columns right of the block (inner work).
// Why 64: the FP64 pipe does n^2 w / 2 FMAs in all solves of width w, 14.7 ms at
// n = 16,900 for w = 64 and 118 ms for whole 512-column tiles, while each step costs three
// launches and one 64 x 64 Cholesky of latency.  Measured (n = 16,900, tile 512): 36 ms of
// diagonal tiles and 100 ms of whole-tile solves became 30 + 17 + 12 ms; the evaluation went
// from 193 to 120 ms, that of n = 5,000 (tile 256) from 27.0 to 18.9 ms.
constexpr int PW = kF64Panel;
static_assert(PW == 64, "the block routines' size");

// One CTA per problem, 256 threads.  The block of the right-hand side becomes y_j.
__global__ void __launch_bounds__(256) k_diag64(const __grid_constant__ F64Set set, int k, int j)
{
    __shared__ Chol64Smem sm;
    const F64Prob &P = set.get(blockIdx.y);
    const Tiles &tl = P.tl;
    // one answer for the CTA: work on the other stream may give up meanwhile, and the block's warps
    // hand each other indexes
    if (k >= tl.T || __syncthreads_or(failed(P.st))) return;
    const int b = tl.b;
    diag64_block(sm, tl.t64(k, k) + (size_t)j * PW * (b + 1), b, b - (j + 1) * PW,
                 P.z ? P.z + (size_t)k * b + j * PW : nullptr, P.winv + (j & 1) * kWinvDoubles,
                 (int64_t)k * b + j * PW, P.st);
}

// One warp slices the 64 entries of a row: lane's entries 2 lane, 2 lane + 1.
__device__ __forceinline__ void slice7_row64(double x0, double x1, uint16_t *__restrict__ dst, size_t stride, int *ep)
{
    const int lane = threadIdx.x & 31;
    const unsigned h0 = (unsigned)__double2hiint(x0) & 0x7FFFFFFFu, h1 = (unsigned)__double2hiint(x1) & 0x7FFFFFFFu;
    const unsigned mh = __reduce_max_sync(0xffffffffu, max(h0, h1));
    const int emax = (int)(mh >> 20);
    const bool bad = emax == 0x7FF;
    const int e = mh == 0 ? 0 : max(emax, 1) - 1022;
    if (lane == 0) *ep = bad ? kBadRow : e;
    uint32_t d0[kF64Slices], d1[kF64Slices];
    digits7(bad || mh == 0 ? 0ll : fixed57(x0, e), d0);
    digits7(bad || mh == 0 ? 0ll : fixed57(x1, e), d1);
#pragma unroll
    for (int i = 0; i < kF64Slices; ++i)
        *reinterpret_cast<uint32_t *>(dst + (size_t)i * stride + 2 * lane) = d0[i] | (d1[i] << 16);
}

// Panel rows (j + 1) 64 .. (T - k) b - 1, RB rows and 8 RB threads per CTA.  RB = 32 (the staged
// block of L serves twice the rows) once RB = 16 fills the SMs.  first: the rows before it are
// left to another launch (64: those of the next diagonal block).
template <int RB>
__global__ void __launch_bounds__(8 * RB) k_solve64(const __grid_constant__ F64Set set, int k, int j, int first)
{
    constexpr int NT = 8 * RB;
    __shared__ Solve64Smem<RB> sm;
    const F64Prob &P = set.get(blockIdx.y);
    const Tiles &tl = P.tl;
    const int b = tl.b, tid = threadIdx.x, lane = tid & 31;
    const int64_t below = (int64_t)((set.solo ? k + 1 : tl.T) - k) * b - (j + 1) * PW;
    const int64_t i0 = (int64_t)blockIdx.x * RB + first;
    if (i0 >= below + (P.vinv ? (j + 1) * PW : 0) || failed(P.st)) return;
    // the rows below, then V's rows 0 .. 64 (j + 1) - 1 (the later ones are zero in these columns)
    const int pr0 = i0 < below ? (j + 1) * PW + (int)i0 : b + (int)(i0 - below);
    double *X = (i0 < below ? tl.t64(k + pr0 / b, k) : P.vinv + (size_t)k * tl.bb()) + (size_t)(pr0 % b) * b + j * PW;
#pragma unroll
    for (int e = tid; e < RB * PW; e += NT) sm.Xs[e >> 6][e & 63] = X[(size_t)(e >> 6) * b + (e & 63)];
    solve64_stage(sm, tl.t64(k, k) + (size_t)j * PW * (b + 1), b, P.winv + (j & 1) * kWinvDoubles);
    // z_row -= X_row . y_j: the forward solve, while the rows are here
    double y0 = 0.0, y1 = 0.0;
    if (P.z) {
        y0 = P.z[(size_t)k * b + j * PW + 2 * lane];
        y1 = P.z[(size_t)k * b + j * PW + 2 * lane + 1];
    }
    __syncthreads();
    solve64_rows(sm);
    __syncthreads();
    for (int r = tid >> 5; r < RB; r += NT / 32) {
        const size_t sr = P.inner.row0 + pr0 + r;
        const double x0 = sm.Xs[r][2 * lane], x1 = sm.Xs[r][2 * lane + 1];
        // two 8-byte stores: a caller's tiles may start at any double
        X[(size_t)r * b + lane] = sm.Xs[r][lane];
        X[(size_t)r * b + 32 + lane] = sm.Xs[r][32 + lane];
        if (P.inner.sl) slice7_row64(x0, x1, P.inner.sl + sr * PW, P.inner.rows * PW, P.inner.ex + sr);
        if (P.z) {
            const double v = dot64(x0, x1, y0, y1);
            if (lane == 0) P.z[(size_t)k * b + pr0 + r] -= v;
        }
    }
}

// The next diagonal block's update by block j: C -= X X^T (K = 64) for the 16 x 16 sub-blocks of its
// lower triangle, one entry a thread.  grid = (10, problems).
__global__ void __launch_bounds__(256) k_next64(const __grid_constant__ F64Set set, int k, int j)
{
    __shared__ double As[16][65], Bs[16][65];
    const F64Prob &P = set.get(blockIdx.y);
    if (k >= P.tl.T || failed(P.st)) return;
    int bi = 0, bj = (int)blockIdx.x;
    while (bj > bi) bj -= ++bi;
    const int b = P.tl.b;
    double *D = P.tl.t64(k, k) + (size_t)(j + 1) * PW * b;  // the block's rows
    inner16(As, Bs, D + (size_t)bi * 16 * b, D + (size_t)bj * 16 * b, b, j, (j + 1) * PW + bj * 16);
}

// V_k = identity for every tile; grid = (T, b / 64).
__global__ void __launch_bounds__(256) k_identity_tiles(double *__restrict__ V, int b)
{
    double *t = V + (size_t)blockIdx.x * b * b;
    for (int r = (int)blockIdx.y * 64; r < (int)blockIdx.y * 64 + 64; ++r)
        for (int c = threadIdx.x; c < b; c += 256) t[(size_t)r * b + c] = r == c ? 1.0 : 0.0;
}

__device__ __forceinline__ float tf32_rna(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// Rows c0 .. c0 + 7 of W = V_k^T through shared memory (8 columns of V_k, 64-byte segments), one
// warp each: the slices, and the split-TF32 layout if wsp is given.  Shared: 8 (b + 1) doubles.
__global__ void __launch_bounds__(256) k_winv_rows(const __grid_constant__ F64Set set, int k, float *__restrict__ wsp)
{
    extern __shared__ double wrow[];
    const F64Prob &P = set.one;
    if (failed(P.st)) return;
    const int b = P.tl.b, c0 = (int)blockIdx.x * 8, ld = b + 1;
    const double *V = P.vinv + (size_t)k * P.tl.bb();
    for (int e = threadIdx.x; e < 8 * b; e += 256) wrow[(e & 7) * ld + (e >> 3)] = V[(size_t)(e >> 3) * b + c0 + (e & 7)];
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, c = c0 + w;
    const double *row = wrow + w * ld;
    slice7_row(row, b, P.w.sl + (size_t)c * b, (size_t)b * b, P.w.ex + c, P.w.dense + c,
               P.ctr + tc64_dense_slot(b, k));
    if (!wsp) return;
    float *out = wsp + (size_t)c * 2 * b;
    for (int i = lane; i < b; i += 32) {
        const float v = (float)row[i], hi = tf32_rna(v);
        out[i] = hi;
        out[b + i] = tf32_rna(v - hi);
    }
}

// ---- the update -------------------------------------------------------------

struct F64Item {
    int m, n;         // output tile; m < 0 ends
    int rb : 8;       // 128-row block
    int cb : 8;       // 64-column block
    int hold : 8;     // its accumulators are never signalled (failure tests)
    int flush : 8;    // K chunks per accumulator flush
};

// Any of n (64 or 128) rows' marks set.
__device__ __forceinline__ bool any_dense(const uint8_t *rows, int n)
{
    uint4 o = make_uint4(0, 0, 0, 0);
    for (int i = 0; i < n; i += 16) {
        const uint4 v = *reinterpret_cast<const uint4 *>(rows + i);
        o.x |= v.x | v.y;
        o.y |= v.z | v.w;
    }
    return (o.x | o.y) != 0;
}

// F64_TRAIL: output tiles (m, n), n = col0 .. col1 - 1, m = n .. T - 1, visited by blocks of
// kF64Cols columns (the block's triangle, then every lower row), so that the CTAs working side
// by side share the block's B operands in L2.  Operand row r of tile m is slice row
// (m - k - 1) b + r, K = b.
// F64_INNER, inside a panel: the 64-column blocks col0 .. col1 - 1 of tile column k, all rows
// from each block's diagonal down; slice row (m - k) b + r, K = 64.  Tile k + 1 of a diagonal
// tile alone is V_k, its rows below 64 col0 as far as they are nonzero.
// The band solve of a mixed factorisation, X L_kk^T = A for the tiles k + 1 .. col1 - 1 of column k
// with W = L_kk^-1 (B operands the rows of W or L_kk; lower triangular, so column block c needs
// K = 64 (c + 1) only), in three products on those rows' slices:
//   F64_BAND  Y = A W^T;
//   F64_RES   the tiles become R = A - Y L_kk^T;
//   F64_CORR  the tiles become X = Y + R W^T.
// A product with the inverse alone leaves a residual that grows with the condition of L_kk: rms of
// Y L^T - A 4.5 (nu = 1/2, range 0.1), 11 (nu = 1.3, range 0.2) and 58 times (nu = 5/2) a substitution's at
// tile 512, X's 0.46, 0.10 and 0.10 times.  Tile 512: 0.05 ms a step alone, 0.15 with the correction
// (n = 25,600: 63.1 and 68.2 ms; a row substitution took 0.22 ms a step).
enum F64Mode { F64_TRAIL = 0, F64_INNER, F64_BAND, F64_RES, F64_CORR };
constexpr int kF64Cols = 8;
struct F64Work {
    const Tiles &tl;
    int T, k, col0, col1, mode;
    __host__ __device__ int row_blocks() const { return (tl.b + FM - 1) / FM; }
    __host__ __device__ bool band() const { return mode >= F64_BAND; }
    __device__ int kchunks(int cb) const { return mode == F64_INNER ? 1 : (band() ? cb + 1 : tl.b / FKC); }
    __host__ __device__ int64_t items() const
    {
        const int64_t c = col1 - col0;
        if (mode == F64_INNER) return c * row_blocks() * (T - k);
        if (band()) return c * row_blocks() * (tl.b / FN);
        const int64_t h = T - col0;
        return (c * h - c * (c - 1) / 2) * row_blocks() * (tl.b / FN);
    }
    __device__ size_t slice_row(int m) const { return (size_t)(m - k - (mode == F64_INNER ? 0 : 1)) * tl.b; }
    __device__ bool decode(int64_t item, F64Item &w) const
    {
        if (mode == F64_INNER) {
            const int wd = col1 - col0, rbs = row_blocks();
            const int64_t u = item / wd;
            w.m = k + (int)(u / rbs);
            w.n = k;
            w.rb = (int)(u % rbs);
            w.cb = col0 + (int)(item % wd);
            return true;
        }
        const int ncb = tl.b / FN, per = row_blocks() * ncb;
        int64_t t = item / per;
        const int blk = (int)(item % per);
        w.rb = blk / ncb;
        w.cb = blk % ncb;
        if (band()) {
            w.m = col0 + (int)t;
            w.n = k;
            return true;
        }
        int c_lo = col0;
        for (;;) {
            const int wd = min(kF64Cols, col1 - c_lo);
            const int64_t tri = (int64_t)wd * (wd + 1) / 2;
            const int64_t cnt = tri + (int64_t)(T - c_lo - wd) * wd;
            if (t < cnt) {
                if (t < tri) {
                    int ii = 0, u = (int)t;
                    while (u > ii) {
                        u -= ii + 1;
                        ++ii;
                    }
                    w.m = c_lo + ii;
                    w.n = c_lo + u;
                } else {
                    const int64_t u = t - tri;
                    w.m = c_lo + wd + (int)(u / wd);
                    w.n = c_lo + (int)(u % wd);
                }
                return true;
            }
            t -= cnt;
            c_lo += wd;
        }
    }
    // Rows of the item's block that are outputs: r0 <= row < r1 of tile m.  On the diagonal tile
    // from the column block's diagonal down (the factored blocks hold zeros above it).
    // Inside a panel the next diagonal block is k_next64's.
    __device__ int r0(const F64Item &w) const
    {
        return w.m == w.n ? (w.cb + (mode == F64_INNER && w.cb == col0 ? 1 : 0)) * FN : 0;
    }
    __device__ int r1(const F64Item &w, bool solo) const
    {
        return mode == F64_INNER && solo && w.m == k + 1 ? col0 * FN : tl.b;
    }
};

// The level sums v_0 .. v_6 of one flush (v_L a multiple of 2^-8L, |v_0| <= 2^24) as fixed
// point in units of 2^-37, all but the last exactly: the FP64 pipe, at 64 clocks a warp-wide
// instruction, took longer over two additions and the conversions (an epilogue of 250 clocks
// an entry against 75) than the tensor cores over the products.
__device__ __forceinline__ long long fixed_sum7(const float (&v)[kF64Slices])
{
    const int u0 = __float2int_rn(v[0]), u1 = __float2int_rn(v[1] * 0x1p8f), u2 = __float2int_rn(v[2] * 0x1p16f);
    const int u3 = __float2int_rn(v[3] * 0x1p24f), u4 = __float2int_rn(v[4] * 0x1p32f);
    const int w = __float2int_rn(__fadd_rn(v[5], v[6]) * 0x1p37f);
    const long long hi = (long long)u0 * 256 + u1, lo = (long long)u2 * 256 + u3;
    return hi * (1ll << 29) + lo * (1ll << 13) + ((long long)u4 * 32 + w);
}

// f 2^-(37 - up) as a double, rounded once, by integer operations.
__device__ __forceinline__ double fixed_to_f64(long long f, int up)
{
    const unsigned long long m = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    const unsigned long long n = m << lz, r = (n >> 11) + ((n >> 10) & 1);
    const unsigned long long bits = ((unsigned long long)(1022 + 63 - lz - 37 + up) << 52) + r;
    return __longlong_as_double((long long)(bits | (f < 0 ? 1ull << 63 : 0ull)));
}

// 2^s as a double, -1022 <= s <= 1023.
__device__ __forceinline__ double pow2(int s) { return __hiloint2double((s + 1023) << 20, 0); }

// 7 x 16 accumulator columns (levels 64 columns apart) of the calling warp's 32 lanes.
__device__ __forceinline__ void tmem_ld_levels16(uint32_t taddr, float (&v)[kF64Slices][16])
{
    uint32_t r[kF64Slices][16];
#define EGS_LD16(L)                                                                                                  \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "  \
                 "[%16];"                                                                                            \
                 : "=r"(r[L][0]), "=r"(r[L][1]), "=r"(r[L][2]), "=r"(r[L][3]), "=r"(r[L][4]), "=r"(r[L][5]),         \
                   "=r"(r[L][6]), "=r"(r[L][7]), "=r"(r[L][8]), "=r"(r[L][9]), "=r"(r[L][10]), "=r"(r[L][11]),       \
                   "=r"(r[L][12]), "=r"(r[L][13]), "=r"(r[L][14]), "=r"(r[L][15])                                    \
                 : "r"(taddr + (L) * FN))
    EGS_LD16(0);
    EGS_LD16(1);
    EGS_LD16(2);
    EGS_LD16(3);
    EGS_LD16(4);
    EGS_LD16(5);
    EGS_LD16(6);
#undef EGS_LD16
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int L = 0; L < kF64Slices; ++L)
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            // the loads have landed; an empty volatile statement keeps every use behind the wait
            asm volatile("" : "+r"(r[L][j]));
            v[L][j] = __uint_as_float(r[L][j]);
        }
}

__device__ __forceinline__ void tma_load_3d(const CUtensorMap *map, uint64_t *bar, void *dst, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];" ::"r"(tc::smem_u32(dst)),
        "l"((uint64_t)map), "r"(tc::smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// Band: the three products of the band solve, apart from the others (their epilogue's choice of
// sources costs those 0.8%).
template <bool Band>
__global__ void __launch_bounds__(FTHREADS, 1)
k_tc_f64(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
         const __grid_constant__ F64Set set, int k, int c0, int c1, int mode, int slot)
{
    __builtin_assume(Band == (mode >= F64_BAND));
    const F64Prob &P = set.get(blockIdx.y);
    const bool solo = set.solo != 0;
    if (P.tl.T <= k) return;
    const int T = !solo ? P.tl.T : (mode == F64_INNER ? k + 1 + (P.vinv ? 1 : 0) : k + c1);
    // columns k + c0 .. min(k + c1, T) - 1; inside a panel the blocks c0 .. c1 - 1 of column k
    const F64Work work{P.tl, T, k, mode == F64_INNER ? c0 : k + c0, mode == F64_INNER ? c1 : min(k + c1, T), mode};
    if (work.col0 >= work.col1) return;
    const int64_t nitems = work.items();
    if ((int64_t)blockIdx.x >= nitems) return;
    unsigned long long *next = P.ctr + slot;
    DevStatus *st = P.st;
    const F64Rows &rows = mode == F64_INNER ? P.inner : P.panel, &brows = !Band ? rows : (mode == F64_RES ? P.l : P.w);
    const int *__restrict__ ex = rows.ex + rows.row0, *__restrict__ exb = brows.ex + brows.row0;
    const int yrow0 = (int)rows.row0, ybrow0 = (int)brows.row0;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t afull[kF64Slices], aempty[kF64Slices], bfull[2], bempty[2], tfull, tempty;
    __shared__ uint64_t rfull[FRING], rempty[FRING];
    __shared__ F64Item ring[FRING];
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, stop, loaded, hold_first, dense_step;
    __shared__ uint64_t mdone;
    __shared__ unsigned long long limit;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kF64Slices; ++i) {
            tc::mbar_init(&afull[i], 1);
            tc::mbar_init(&aempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&bfull[i], 1);
            tc::mbar_init(&bempty[i], 1);
        }
        tc::mbar_init(&tfull, 1);
        tc::mbar_init(&tempty, 8);
        for (int r = 0; r < FRING; ++r) {
            tc::mbar_init(&rfull[r], 1);
            tc::mbar_init(&rempty[r], 1 + 8);
        }
        tc::mbar_init(&mdone, 1);
        abort_flag = 0;
        loaded = 0;
        limit = set.ctl ? set.ctl->limit_ns : tc::kWaitNs;
        hold_first = mode == F64_TRAIL && set.ctl && set.ctl->prob == (int)blockIdx.y && set.ctl->step == k;
        // the rows' own marks are read only in a step that has one (read for every block they cost
        // the producer 1 us each: n = 51,200, all updates 996 ms against 980)
        dense_step = rows.dense && *(volatile unsigned long long *)(P.ctr + tc64_dense_slot(work.tl.b, k)) != 0;
        stop = failed(st) ? 1 : 0;
        tc::fence_mbar_init();
    }
    __syncthreads();
    if (stop) return;
    if (warp == 0) tc::tmem_alloc(&tmem_base, FTMEM);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = tmem_base;
    const int b = work.tl.b;
    uint8_t *sa = smem, *sb = smem + kF64Slices * FA_SL;

    if (warp == 0) {
        if (lane == 0) {
            tc::prefetch_tmap(&mapA);
            tc::prefetch_tmap(&mapB);
            int g = 0, r = 0;  // chunks loaded, items posted
            int64_t claimed = (int64_t)atomicAdd(next, 1ull);
            while (!abort_flag) {
                F64Item wi;
                const bool valid = claimed < nitems && work.decode(claimed, wi) && wi.rb * FM + FM > work.r0(wi) &&
                                   wi.rb * FM < work.r1(wi, solo);
                if (claimed < nitems && !valid) {
                    claimed = (int64_t)atomicAdd(next, 1ull);
                    continue;
                }
                const int slot = r % FRING;
                if (!tc::mbar_wait(&rempty[slot], ((uint32_t)(r / FRING) & 1u) ^ 1u, &abort_flag, &limit)) break;
                if (!valid) wi.m = -1;
                wi.hold = hold_first && claimed == 0;
                wi.flush = FLUSH;
                if (valid && dense_step && work.kchunks(wi.cb) > FLUSH_DENSE) {
                    // the block's rows of the tile, at most 128
                    const uint8_t *da = rows.dense + yrow0 + work.slice_row(wi.m) + wi.rb * FM;
                    const uint8_t *db = brows.dense + ybrow0 + (Band ? 0 : work.slice_row(wi.n)) + wi.cb * FN;
                    if (any_dense(da, min(FM, b - wi.rb * FM)) || any_dense(db, FN)) wi.flush = FLUSH_DENSE;
                }
                ring[slot] = wi;
                tc::mbar_arrive(&rfull[slot]);
                ++r;
                if (!valid) break;
                claimed = (int64_t)atomicAdd(next, 1ull);  // overlaps the loads below
                const int ya = yrow0 + (int)work.slice_row(wi.m) + wi.rb * FM;
                const int yb = ybrow0 + (Band ? 0 : (int)work.slice_row(wi.n)) + wi.cb * FN;
                const int kchunks = work.kchunks(wi.cb);
                for (int c = 0; c < kchunks && !abort_flag; ++c, ++g) {
                    const int bb = g & 1;
                    if (!tc::mbar_wait(&bempty[bb], ((uint32_t)(g >> 1) & 1u) ^ 1u, &abort_flag, &limit)) break;
                    tc::mbar_arrive_expect_tx(&bfull[bb], FB_BUF);
                    tma_load_3d(&mapB, &bfull[bb], sb + bb * FB_BUF, c * FKC, yb, 0);
                    int i = 0;
                    for (; i < kF64Slices; ++i) {
                        if (!tc::mbar_wait(&aempty[i], ((uint32_t)g & 1u) ^ 1u, &abort_flag, &limit)) break;
                        tc::mbar_arrive_expect_tx(&afull[i], FA_SL);
                        tma_load_3d(&mapA, &afull[i], sa + i * FA_SL, c * FKC, ya, i);
                    }
                    // loads issued so far: chunk g's B box and its first i A boxes
                    loaded = g * 8 + 1 + i;
                    if (i < kF64Slices) break;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int g = 0, r = 0;
            uint32_t f = 0;  // flush groups issued
            while (!abort_flag) {
                const int slot = r % FRING;
                if (!tc::mbar_wait(&rfull[slot], (uint32_t)(r / FRING) & 1u, &abort_flag, &limit)) break;
                const int m = ring[slot].m, kchunks = work.kchunks(ring[slot].cb), hold = ring[slot].hold;
                const int flush = ring[slot].flush;
                tc::mbar_arrive(&rempty[slot]);
                ++r;
                if (m < 0) break;
                for (int c = 0; c < kchunks && !abort_flag; ++c, ++g) {
                    const bool first = (c & (flush - 1)) == 0;
                    if (first) {
                        if (!tc::mbar_wait(&tempty, (f & 1u) ^ 1u, &abort_flag, &limit)) break;
                        tc::tc_fence_after();
                    }
                    const int bb = g & 1;
                    if (!tc::mbar_wait(&bfull[bb], (uint32_t)(g >> 1) & 1u, &abort_flag, &limit)) break;
                    const uint32_t b0 = tc::smem_u32(sb + bb * FB_BUF);
#pragma unroll
                    for (int i = 0; i < kF64Slices; ++i) {
                        if (!tc::mbar_wait(&afull[i], (uint32_t)g & 1u, &abort_flag, &limit)) break;
                        tc::tc_fence_after();
                        const uint32_t a0 = tc::smem_u32(sa + i * FA_SL);
                        const int n = kF64Slices - i;  // B slices 0 .. n - 1
                        const int n0 = n < 4 ? n : 4, n1 = n - n0;
                        const uint32_t id0 = tc::idesc_f32acc(FM, n0 * FN, 1);
                        const uint32_t id1 = tc::idesc_f32acc(FM, (n1 > 0 ? n1 : 1) * FN, 1);
#pragma unroll
                        for (int j = 0; j < FKC / 16; ++j) {
                            // the i = 0 MMAs of a flush group's first K step cover all
                            // seven level blocks and so initialise them
                            const uint32_t acc = (first && i == 0 && j == 0) ? 0u : 1u;
                            const uint64_t ad = tc::desc_sw128(a0 + 32 * j);
                            tc::mma_f16(tbase + (uint32_t)(i * FN), ad, tc::desc_sw128(b0 + 32 * j), id0, acc);
                            if (n1 > 0)
                                tc::mma_f16(tbase + (uint32_t)((i + n0) * FN), ad,
                                            tc::desc_sw128(b0 + n0 * FB_SL + 32 * j), id1, acc);
                        }
                        tc::mma_commit(&aempty[i]);
                    }
                    tc::mma_commit(&bempty[bb]);
                    if ((c & (flush - 1)) == flush - 1 || c == kchunks - 1) {
                        if (!hold) tc::mma_commit(&tfull);
                        ++f;
                    }
                }
            }
            tc::mma_commit(&mdone);  // every MMA issued, whatever way the loop ended
        }
    } else {
        // warp w: TMEM lanes 32 (w % 4) .. + 31 (rows of the block), columns 32 half .. + 31
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t t0 = tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 32);
        uint32_t f = 0;
        int r = 0;
        bool run = true;
        while (run) {
            const int slot = r % FRING;
            const bool got = tc::mbar_wait(&rfull[slot], (uint32_t)(r / FRING) & 1u, &abort_flag, &limit);
            if (!__all_sync(0xffffffffu, got && !abort_flag)) break;
            const F64Item wi = ring[slot];
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&rempty[slot]);
            ++r;
            if (wi.m < 0) break;
            const int kchunks = work.kchunks(wi.cb), nflush = (kchunks + wi.flush - 1) >> (wi.flush == FLUSH ? 2 : 1);
            const int up = kchunks > 2 * FLUSH ? 1 : 0;  // the sum over the flushes stays below 2^63
            long long acc[32];
            for (int fl = 0; fl < nflush; ++fl, ++f) {
                const bool ok = tc::mbar_wait(&tfull, f & 1u, &abort_flag, &limit);
                tc::tc_fence_after();
                if (!__all_sync(0xffffffffu, ok && !abort_flag)) {
                    run = false;
                    break;
                }
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    float v[kF64Slices][16];
                    tmem_ld_levels16(t0 + (uint32_t)(hh * 16), v);
                    if (hh == 1) {
                        tc::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&tempty);  // every level is in registers
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float vj[kF64Slices] = {v[0][j], v[1][j], v[2][j], v[3][j], v[4][j], v[5][j], v[6][j]};
                        const long long d = fixed_sum7(vj) >> up;
                        acc[hh * 16 + j] = fl == 0 ? d : acc[hh * 16 + j] + d;
                    }
                }
            }
            if (!run) break;
            const int row = wi.rb * FM + q * 32 + lane;
            if (row >= work.r0(wi) && row < work.r1(wi, solo)) {
                const int col = wi.cb * FN + half * 32;
                const int ea = ex[work.slice_row(wi.m) + row] - 16;
                const int *eb = exb + (Band ? 0 : work.slice_row(wi.n)) + col;
                double *C = (solo && mode == F64_INNER && wi.m > k ? P.vinv + (size_t)k * work.tl.bb()
                                                                   : work.tl.t64(wi.m, wi.n)) + (size_t)row * b + col;
                const double *Cin = C;  // what the product is added to or subtracted from
                const bool add = Band && mode != F64_RES;
                if (add) {
                    double *y = P.y + (size_t)(wi.m - k - 1) * work.tl.bb() + (size_t)row * b + col;
                    Cin = y;
                    if (mode == F64_BAND) C = y;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    double2 cv[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        cv[j] = Band && mode == F64_BAND ? make_double2(0.0, 0.0)
                                                 : *reinterpret_cast<const double2 *>(Cin + 16 * h + 2 * j);
                    double *cd = reinterpret_cast<double *>(cv);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int s = ea + __ldg(eb + 16 * h + j);
                        const double d = fixed_to_f64(add ? -acc[16 * h + j] : acc[16 * h + j], up);
                        if (s >= -960 && s <= 1000) {
                            cd[j] = fma(-pow2(s), d, cd[j]);
                        } else if (s > 1000) {
                            // an infinity or a NaN in either row reaches every product with it
                            cd[j] = s >= kBadRow / 2 ? __longlong_as_double(0x7ff8000000000000ll)
                                                     : fma(-pow2(s - 100), d * pow2(100), cd[j]);
                        } else {
                            cd[j] = s < -2040 ? cd[j] : fma(-pow2(-600), d * pow2(max(s + 600, -1022)), cd[j]);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) *reinterpret_cast<double2 *>(C + 16 * h + 2 * j) = cv[j];
                }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    if (abort_flag && threadIdx.x == 0) {
        // let every load that was issued land before the CTA exits: chunk g = loaded / 8
        // holds its B box and loaded % 8 - 1 A boxes, the chunks before it are complete
        volatile int dummy = 0;
        const int total = loaded;
        for (int bbi = 0; bbi < 2; ++bbi) {
            int last = (total + 7) / 8 - 1;  // last chunk whose B box was issued
            if (last >= 0 && (last & 1) != bbi) --last;
            if (last >= 0) tc::mbar_wait(&bfull[bbi], (uint32_t)(last >> 1) & 1u, &dummy);
        }
        for (int i = 0; i < kF64Slices; ++i) {
            const int last = (total - 2 - i) >= 0 ? (total - 2 - i) / 8 : -1;
            if (last >= 0) tc::mbar_wait(&afull[i], (uint32_t)last & 1u, &dummy);
        }
        atomicExch(&st->timeout, 1);
        atomicMin(&st->fail_index, 0ull);  // stops the rest of the evaluation
    }
    if (threadIdx.x == 0) {  // and every MMA finish before TMEM goes (long done but after an abort)
        volatile int dummy = 0;
        tc::mbar_wait(&mdone, 0, &dummy);
    }
    tc::tc_fence_after();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, FTMEM);
}

PFN_cuTensorMapEncodeTiled_v12000 f64_encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (PFN_cuTensorMapEncodeTiled_v12000)p;
    }();
    return fn;
}

// 3-D map over the slices (7 x rows x K BF16), box 64 x box_rows x box_slices, 128-byte swizzle.
cudaError_t make_map3(CUtensorMap *m, const void *base, uint64_t rows, uint64_t K, uint32_t box_rows, uint32_t box_sl)
{
    auto fn = f64_encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint64_t dims[3] = {K, rows, (cuuint64_t)kF64Slices};
    cuuint64_t strides[2] = {K * 2, rows * K * 2};
    cuuint32_t box[3] = {(cuuint32_t)FKC, box_rows, box_sl};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

int device_sms()
{
    static const int sms = [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
        return n;
    }();
    return sms;
}

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// Slices and exponents of the panel (K = b) and of its 64-column blocks (K = 64, the
// diagonal tile's rows too), the work counters, the 8 x 8 inverses.
size_t tc64_scratch_bytes(int b, int T)
{
    const size_t R = (size_t)(T - 1) * (size_t)b, R1 = R + b;
    return a256(R * b * kF64Slices * sizeof(uint16_t)) + a256(R * sizeof(int)) + a256(R) +
           a256(R1 * PW * kF64Slices * sizeof(uint16_t)) + a256(R1 * sizeof(int)) +
           a256(tc64_counters(b, T) * sizeof(unsigned long long)) + a256(2 * kWinvDoubles * sizeof(double));
}

F64Prob tc64_problem(void *scratch, const Tiles &tl, DevStatus *st, double *z)
{
    const size_t R = (size_t)(tl.T - 1) * (size_t)tl.b, R1 = R + tl.b;
    char *p = (char *)scratch;
    auto take = [&p](size_t bytes) {
        char *q = p;
        p += a256(bytes);
        return q;
    };
    F64Prob P{};
    P.tl = tl;
    P.st = st;
    P.z = z;
    P.panel.sl = (uint16_t *)take(R * tl.b * kF64Slices * sizeof(uint16_t));
    P.panel.ex = (int *)take(R * sizeof(int));
    P.panel.dense = (uint8_t *)take(R);
    P.panel.rows = R;
    P.inner.sl = (uint16_t *)take(R1 * PW * kF64Slices * sizeof(uint16_t));
    P.inner.ex = (int *)take(R1 * sizeof(int));
    P.inner.rows = R1;
    P.panel.row0 = P.inner.row0 = 0;
    P.ctr = (unsigned long long *)take(tc64_counters(tl.b, tl.T) * sizeof(unsigned long long));
    P.winv = (double *)take(2 * kWinvDoubles * sizeof(double));
    return P;
}

cudaError_t make_f64_maps(const F64Rows &panel, const F64Rows &inner, int b, F64Maps *maps)
{
    cudaError_t e = cudaSuccess;
    if (panel.rows) e = make_map3(&maps->a, panel.sl, panel.rows, (uint64_t)b, FM, 1);
    else maps->a = maps->b = CUtensorMap{};
    if (e == cudaSuccess && panel.rows) e = make_map3(&maps->b, panel.sl, panel.rows, (uint64_t)b, FN, kF64Slices);
    if (e == cudaSuccess) e = make_map3(&maps->ia, inner.sl, inner.rows, PW, FM, 1);
    if (e == cudaSuccess) e = make_map3(&maps->ib, inner.sl, inner.rows, PW, FN, kF64Slices);
    return e;
}

size_t tc64_solo_bytes(int b, int T, int nb)
{
    auto rows = [](size_t n, size_t K) {  // as tc64_solo_problem
        return a256(n * K * kF64Slices * sizeof(uint16_t)) + a256(n * sizeof(int)) + a256(n);
    };
    return rows((size_t)nb * b, b) + rows((size_t)2 * b, PW) + 2 * rows((size_t)b, b) +
           a256((size_t)nb * b * b * sizeof(double)) +
           a256(tc64_counters(b, T) * sizeof(unsigned long long)) + a256(2 * kWinvDoubles * sizeof(double));
}

F64Prob tc64_solo_problem(void *scratch, const Tiles &tl, DevStatus *st, double *vinv, int nb)
{
    const size_t b = (size_t)tl.b;
    char *p = (char *)scratch;
    auto take = [&p](size_t bytes) {
        char *q = p;
        p += a256(bytes);
        return q;
    };
    auto rows = [&](size_t n, size_t K) {
        F64Rows r{};
        r.sl = (uint16_t *)take(n * K * kF64Slices * sizeof(uint16_t));
        r.ex = (int *)take(n * sizeof(int));
        r.dense = (uint8_t *)take(n);
        r.rows = n;
        return r;
    };
    F64Prob P{};
    P.tl = tl;
    P.st = st;
    P.vinv = vinv;
    P.panel = rows((size_t)nb * b, b);
    P.inner = rows(2 * b, PW);
    P.inner.dense = nullptr;  // one chunk: never flushed in between
    P.w = rows(b, b);
    P.l = rows(b, b);
    P.y = (double *)take((size_t)nb * b * b * sizeof(double));
    P.ctr = (unsigned long long *)take(tc64_counters(tl.b, tl.T) * sizeof(unsigned long long));
    P.winv = (double *)take(2 * kWinvDoubles * sizeof(double));
    return P;
}

cudaError_t make_f64_solo_maps(const F64Prob &P, F64Maps *maps)
{
    const uint64_t b = (uint64_t)P.tl.b;
    cudaError_t e = cudaSuccess;
    maps->a = CUtensorMap{};
    if (P.panel.rows) e = make_map3(&maps->a, P.panel.sl, P.panel.rows, b, FM, 1);
    if (e == cudaSuccess && P.panel.rows) e = make_map3(&maps->pb, P.panel.sl, P.panel.rows, b, FN, kF64Slices);
    if (e == cudaSuccess) e = make_map3(&maps->b, P.w.sl, P.w.rows, b, FN, kF64Slices);
    if (e == cudaSuccess) e = make_map3(&maps->lb, P.l.sl, P.l.rows, b, FN, kF64Slices);
    if (e == cudaSuccess) e = make_map3(&maps->ia, P.inner.sl, P.inner.rows, PW, FM, 1);
    if (e == cudaSuccess) e = make_map3(&maps->ib, P.inner.sl, P.inner.rows, PW, FN, kF64Slices);
    return e;
}

// CTAs of a problem's update launch: the whole GPU for one problem, a share for each of many.
static unsigned tc64_ctas(const F64Set &set, int64_t items)
{
    int64_t c = device_sms();
    if (set.count > 1) c = (c * 4 + set.count - 1) / set.count;
    c = items < c ? items : c;
    return (unsigned)(c > 1 ? c : 1);
}

static cudaError_t launch_tc_f64(const CUtensorMap &a, const CUtensorMap &b, const F64Set &set, int k, int c0, int c1,
                                 int mode, int slot, cudaStream_t s, KernelTimer *kt)
{
    auto kernel = mode >= F64_BAND ? k_tc_f64<true> : k_tc_f64<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FSMEM);
    if (e != cudaSuccess) return e;
    // of the largest problem, as in the kernel
    const int T = !set.solo ? set.Tmax : (mode == F64_INNER ? k + 1 + (set.one.vinv ? 1 : 0) : k + c1);
    const Tiles tl{nullptr, nullptr, set.b, T, T};
    const bool in = mode == F64_INNER;
    const F64Work w{tl, T, k, in ? c0 : k + c0, in ? c1 : (k + c1 < T ? k + c1 : T), mode};
    if (w.col0 >= w.col1) return cudaSuccess;
    const dim3 grid(tc64_ctas(set, w.items()), (unsigned)set.count);
    // of a mixed factorisation's diagonal tile: part of its POTRF; its band: the FP64 update class
    const int cls = mode >= F64_BAND ? KC_TRSM : (!set.solo ? KC_UPDATE : (in ? KC_POTRF : KC_UPDATE64));
    EGS_LAUNCH(kt, cls, s,
               kernel<<<grid, FTHREADS, FSMEM, s>>>(a, b, set, k, c0, c1, mode, slot));
    return cudaGetLastError();
}

static cudaError_t launch_diag64(const F64Set &set, int k, int j, cudaStream_t s, KernelTimer *kt)
{
    EGS_LAUNCH(kt, KC_POTRF, s, k_diag64<<<dim3(1, (unsigned)set.count), 256, 0, s>>>(set, k, j));
    return cudaGetLastError();
}

// rows first .. (64 of them if next, else all the others) below block j
static cudaError_t launch_solve64(const F64Set &set, int k, int j, int first, bool next, cudaStream_t s, KernelTimer *kt)
{
    int64_t rows = set.solo && set.one.vinv ? set.b : (int64_t)(set.solo ? 1 : set.Tmax - k) * set.b - (j + 1) * PW;
    rows = next ? PW : rows - first;
    if (rows <= 0) return cudaSuccess;
    if (rows / 16 * set.count <= device_sms())
        EGS_LAUNCH(kt, KC_TRSM, s,
                   k_solve64<16><<<dim3((unsigned)(rows / 16), (unsigned)set.count), 128, 0, s>>>(set, k, j, first));
    else
        EGS_LAUNCH(kt, KC_TRSM, s,
                   k_solve64<32><<<dim3((unsigned)(rows / 32), (unsigned)set.count), 256, 0, s>>>(set, k, j, first));
    return cudaGetLastError();
}

cudaError_t launch_diag_solve64(const F64Set &set, int k, int j, cudaStream_t s, KernelTimer *kt)
{
    cudaError_t e = launch_diag64(set, k, j, s, kt);
    return e == cudaSuccess ? launch_solve64(set, k, j, 0, false, s, kt) : e;
}

cudaError_t F64Fork::create(cudaStream_t s, bool high_priority)
{
    cudaError_t e = aux.create(s, high_priority);
    for (cudaEvent_t *ev : {&diag, &next})
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    return e;
}

F64Fork::~F64Fork()
{
    for (cudaEvent_t ev : {diag, next})
        if (ev) cudaEventDestroy(ev);
}

F64Prob dfma_problem(double *winv, const Tiles &tl, DevStatus *st, double *z)
{
    F64Prob P{};
    P.tl = tl;
    P.st = st;
    P.z = z;
    P.winv = winv;
    return P;
}

// With a fork, what the next diagonal block waits for (its rows' solve, its own update) goes ahead
// on s, and the other rows and columns follow beside it on the second stream (evaluations of
// n = 16,900: 75.7 -> 70.4 ms, n = 5,000: 9.8 -> 9.0 ms).
cudaError_t launch_panel64(const F64Maps &maps, const F64Set &set, int k, F64Fork *fork, cudaStream_t s, KernelTimer *kt)
{
    const int nj = set.b / PW;
    if (kt && kt->on) fork = nullptr;  // per-launch times and traces: one stream, launches in order
    cudaStream_t bs = fork ? fork->aux.st : s;
    cudaError_t e = cudaSuccess;
    if (fork) fork->aux.open = true;  // until s waits for it below; otherwise its owner does at the end
    for (int j = 0; j < nj && e == cudaSuccess; ++j) {
        const bool more = j + 1 < nj;
        e = launch_diag64(set, k, j, s, kt);
        if (!fork) {
            if (e == cudaSuccess) e = launch_solve64(set, k, j, 0, false, s, kt);
        } else {
            if (e == cudaSuccess) e = cudaEventRecord(fork->diag, s);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(bs, fork->diag, 0);
            if (e == cudaSuccess && more) {
                // the next block's rows carry block j - 1's update of column j
                if (j > 0) e = cudaStreamWaitEvent(s, fork->aux.done, 0);
                if (e == cudaSuccess) e = launch_solve64(set, k, j, 0, true, s, kt);
                if (e == cudaSuccess) e = cudaEventRecord(fork->next, s);
            }
            if (e == cudaSuccess) e = launch_solve64(set, k, j, more ? PW : 0, false, bs, kt);
        }
        if (e != cudaSuccess) break;
        if (more) {
            EGS_LAUNCH(kt, set.solo ? KC_POTRF : KC_UPDATE, s,
                       k_next64<<<dim3(10, (unsigned)set.count), 256, 0, s>>>(set, k, j));
            e = cudaGetLastError();
            if (fork && e == cudaSuccess) e = cudaStreamWaitEvent(bs, fork->next, 0);
            if (e == cudaSuccess)
                e = launch_tc_f64(maps.ia, maps.ib, set, k, j + 1, nj, F64_INNER,
                                  tc64_slot(set.b, k, 4 + j), bs, kt);
        }
        if (fork && e == cudaSuccess) e = cudaEventRecord(fork->aux.done, bs);
    }
    if (fork && e == cudaSuccess) e = cudaStreamWaitEvent(s, fork->aux.done, 0);
    if (fork && e == cudaSuccess) fork->aux.open = false;
    return e;
}

cudaError_t launch_slice_panel64(const F64Set &set, int k, cudaStream_t s, KernelTimer *kt)
{
    if (k + 1 >= set.Tmax) return cudaSuccess;
    EGS_LAUNCH(kt, KC_TRSM, s,
               k_slice_panel64<<<dim3((unsigned)((size_t)(set.Tmax - k - 1) * set.b / 8), (unsigned)set.count), 256, 0,
                                 s>>>(set, k, 0));
    return cudaGetLastError();
}

cudaError_t launch_update_tc64(const F64Maps &maps, const F64Set &set, int k, cudaStream_t s, KernelTimer *kt)
{
    return launch_tc_f64(maps.a, maps.b, set, k, 1, set.Tmax, F64_TRAIL, tc64_slot(set.b, k, 0), s, kt);
}

cudaError_t launch_solo_init(const F64Set &set, cudaStream_t s, KernelTimer *kt)
{
    cudaError_t e = cudaMemsetAsync(set.one.ctr, 0, tc64_counters(set.b, set.Tmax) * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    EGS_LAUNCH(kt, KC_OTHER, s,
               k_identity_tiles<<<dim3((unsigned)set.Tmax, (unsigned)(set.b / 64)), 256, 0, s>>>(set.one.vinv, set.b));
    return cudaGetLastError();
}

static cudaError_t launch_slice_band(const F64Set &set, int k, int rows, int src, cudaStream_t s, KernelTimer *kt)
{
    EGS_LAUNCH(kt, KC_TRSM, s, k_slice_panel64<<<dim3((unsigned)(rows / 8), 1), 256, 0, s>>>(set, k, src));
    return cudaGetLastError();
}

cudaError_t launch_winv(const F64Set &set, int k, float *wsp, cudaStream_t s, KernelTimer *kt)
{
    const size_t sm = (size_t)8 * (set.b + 1) * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_winv_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * 1025 * sizeof(double));
    if (e != cudaSuccess) return e;
    EGS_LAUNCH(kt, KC_TRSM, s, k_winv_rows<<<(unsigned)(set.b / 8), 256, sm, s>>>(set, k, wsp));
    e = cudaGetLastError();
    return e == cudaSuccess ? launch_slice_band(set, k, set.b, 2, s, kt) : e;
}

cudaError_t launch_band_solve(const F64Maps &maps, const F64Set &set, int k, int nb, cudaStream_t s, KernelTimer *kt)
{
    if (nb <= 0) return cudaSuccess;
    const int rows = nb * set.b;
    cudaError_t e = launch_slice_band(set, k, rows, 0, s, kt);
    if (e == cudaSuccess) e = launch_tc_f64(maps.a, maps.b, set, k, 1, 1 + nb, F64_BAND, tc64_slot(set.b, k, 1), s, kt);
    if (e == cudaSuccess) e = launch_slice_band(set, k, rows, 1, s, kt);
    if (e == cudaSuccess) e = launch_tc_f64(maps.a, maps.lb, set, k, 1, 1 + nb, F64_RES, tc64_slot(set.b, k, 2), s, kt);
    if (e == cudaSuccess) e = launch_slice_band(set, k, rows, 0, s, kt);
    if (e == cudaSuccess) e = launch_tc_f64(maps.a, maps.b, set, k, 1, 1 + nb, F64_CORR, tc64_slot(set.b, k, 3), s, kt);
    return e;
}

cudaError_t launch_band_update(const F64Maps &maps, const F64Set &set, int k, int nb, cudaStream_t s, KernelTimer *kt)
{
    if (nb <= 0) return cudaSuccess;
    cudaError_t e = launch_slice_band(set, k, nb * set.b, 0, s, kt);
    if (e != cudaSuccess) return e;
    return launch_tc_f64(maps.a, maps.pb, set, k, 1, 1 + nb, F64_TRAIL, tc64_slot(set.b, k, 0), s, kt);
}

}  // namespace egs
