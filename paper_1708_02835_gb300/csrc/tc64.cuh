// Host interface of the FP64 factorisation on the tensor cores (tc64.cu).
#pragma once
#include "blocks.cuh"
#include "egs_internal.cuh"
#include "side_stream.cuh"

namespace egs {

constexpr int kF64Slices = 7;
constexpr int kF64Panel = 64;  // width of the blocks a tile column is factored in

// FP64 factorisations take the tensor cores above this many rows.  The line is the persistent
// batch's: it runs the DFMA routines and equals single evaluations bit for bit.  The tensor cores
// alone would win from about 700 rows on (evaluations by DFMA / by slice products, default tile:
// n = 500 0.88 / 0.89 ms, 777 1.58 / 1.44, 1,600 3.67 / 2.55, 2,048 5.42 / 3.16, 2,049 6.11 / 3.36,
// 4,096 25.3 / 7.05).
constexpr int64_t kTc64MinRows = 2049;
// They also need memory that starts on a 16-byte boundary (tc64_aligned: TMA boxes, pairs of doubles
// in the update's epilogue); a caller's tiles or workspace without that take the DFMA update.
inline bool tc64_aligned(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
inline bool tc64_applies(int64_t n, int b, int T) { return n >= kTc64MinRows && T > 1 && b % 64 == 0; }

// Work counters of a problem, per step: the trailing update (a mixed factorisation: the band update),
// the three products of a mixed factorisation's band solve, then each 64-column block's inner update
// but the last one's, whose place holds whether any row sliced in the step is dense.
__host__ __device__ inline int tc64_slot(int b, int k, int i) { return k * (4 + b / kF64Panel) + i; }
__host__ __device__ inline int tc64_dense_slot(int b, int k) { return tc64_slot(b, k + 1, -1); }
inline size_t tc64_counters(int b, int T) { return (size_t)tc64_slot(b, T, 0); }

// Slices of operand rows (slice i of row r at sl[(i rows + r) K ..], K = b or 64) and the
// rows' exponents; several problems share one array, each from its own row0 on.
struct F64Rows {
    uint16_t *sl;
    int *ex;
    size_t rows, row0;
    uint8_t *dense;  // K = b: 1 for a row whose level sums need the short flush (tc64.cu); NULL for K = 64
};

// One problem as the kernels see it.
struct F64Prob {
    Tiles tl;
    DevStatus *st;
    double *z;                // T b: the right-hand side, solved along (L^-1 z); NULL: none
    double *vinv;             // diagonal tiles alone: V_k = L_kk^-T (T b x b, identities before), or NULL
    F64Rows panel;            // K = b: row r of tile m at row0 + (m - k - 1) b + r
    F64Rows inner;            // K = 64, the current 64-column block: row0 + (m - k) b + r; sl NULL: no slices
    F64Rows w, l;             // diagonal tiles alone: K = b, the rows of L_kk^-1 and of L_kk
    double *y;                // diagonal tiles alone: the band rows' first solution, nb b x b
    unsigned long long *ctr;  // tc64_counters(b, T) zeroed work counters
    double *winv;             // inverses of the block's eight 8 x 8 diagonal blocks, two of kWinvDoubles (j & 1)
};

// Failure detection of a batch (egs_batch_set_wait_limit): the bound of k_tc_f64's waits, and the
// problem and step whose trailing update never signals its first output block (-1: none).
struct F64Ctl {
    unsigned long long limit_ns;
    int prob, step;
};

// The problems of a launch (one per grid row): one, or count of them in device memory with
// Tmax tiles at most.
struct F64Set {
    const F64Prob *arr;
    F64Prob one;
    int count, b, Tmax;
    int solo;  // 1: the diagonal tile of a step alone (launch_panel64 is its POTRF and, with vinv, its
               // inverse: V_k as further rows of the panel, row r at inner slice row b + r)
    const F64Ctl *ctl;  // in device memory, or NULL: 2 s, none
    __device__ const F64Prob &get(int i) const { return arr ? arr[i] : one; }
};


struct F64Maps {
    CUtensorMap a, b, ia, ib;  // panel slices, inner slices; diagonal tiles alone: b is W's, pb the panel's, lb L_kk's
    CUtensorMap pb, lb;
};
// Over slice arrays of rows (K = b) and irows (K = 64) rows.
cudaError_t make_f64_maps(const F64Rows &panel, const F64Rows &inner, int b, F64Maps *maps);

// Device scratch of one tensor-core FP64 factorisation, and the problem on it.
size_t tc64_scratch_bytes(int b, int T);
F64Prob tc64_problem(void *scratch, const Tiles &tl, DevStatus *st, double *z);

// The same for the diagonal tiles of a mixed factorisation and the solves of nb tiles below
// each (the FP64 band): launch_solo_init once, then per step launch_panel64, launch_winv and
// launch_band_solve.
size_t tc64_solo_bytes(int b, int T, int nb);
F64Prob tc64_solo_problem(void *scratch, const Tiles &tl, DevStatus *st, double *vinv, int nb);
cudaError_t make_f64_solo_maps(const F64Prob &p, F64Maps *maps);
// Identities into V, the counters.
cudaError_t launch_solo_init(const F64Set &set, cudaStream_t s, KernelTimer *kt);
// The rows of W = L_kk^-1 = V_k^T and of L_kk: slices, and (wsp not NULL) the split-TF32 layout of
// the off-band solve, row c: [hi | lo] of (float)W[c][.].
cudaError_t launch_winv(const F64Set &set, int k, float *wsp, cudaStream_t s, KernelTimer *kt);
// Tiles (k + 1 .. k + nb, k): X L_kk^T = A, in place, by products with W and one correction.
cudaError_t launch_band_solve(const F64Maps &maps, const F64Set &set, int k, int nb, cudaStream_t s, KernelTimer *kt);

// The same without slices, for the DFMA updates; winv: 2 kWinvDoubles of scratch.
F64Prob dfma_problem(double *winv, const Tiles &tl, DevStatus *st, double *z);
// Diagonal block j of step k; the solves of the rows below it (launch_panel64's first two parts).
cudaError_t launch_diag_solve64(const F64Set &set, int k, int j, cudaStream_t s, KernelTimer *kt);

// A second stream for the panels of one factorisation on stream s.
struct F64Fork {
    SideStream aux;  // aux.done: the panel's bulk
    cudaEvent_t diag = nullptr, next = nullptr;
    cudaError_t create(cudaStream_t s, bool high_priority);
    ~F64Fork();
};

// POTRF of tile (k, k) and the solves of every tile below it, in 64-column blocks; fork may be NULL.
cudaError_t launch_panel64(const F64Maps &maps, const F64Set &set, int k, F64Fork *fork, cudaStream_t s,
                           KernelTimer *kt);
// C_mn -= X_m X_n^T for the FP64 band tiles k < n <= m <= k + nb, from the solved band rows.
cudaError_t launch_band_update(const F64Maps &maps, const F64Set &set, int k, int nb, cudaStream_t s, KernelTimer *kt);
// Slices of the solved panel tiles (k + 1 .. T - 1, k).
cudaError_t launch_slice_panel64(const F64Set &set, int k, cudaStream_t s, KernelTimer *kt);
// C_mn -= P_m P_n^T for k < n <= m < T.
cudaError_t launch_update_tc64(const F64Maps &maps, const F64Set &set, int k, cudaStream_t s, KernelTimer *kt);

}  // namespace egs
