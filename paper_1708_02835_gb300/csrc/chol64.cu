// FP64 tile Cholesky (Algorithm 2, dpotrf) by the right-looking tile algorithm
// of Section 5.2: for k = 0..T-1
//   POTRF  L_kk = chol(A_kk)
//   TRSM   A_mk <- A_mk L_kk^-T            (m > k)
//   SYRK   A_mm <- A_mm - A_mk A_mk^T       (m > k)
//   GEMM   A_mn <- A_mn - A_mk A_nk^T       (m > n > k)
// SYRK and GEMM share one kernel (a diagonal output tile skips its upper
// sub-blocks).  POTRF and TRSM run together over the whole tile column, in
// 64-column blocks (tc64.cu): the 64 x 64 Cholesky on one SM, the solve of every
// row below, the update of the column's other blocks.
//
// GB300's FP64 rate is 2 DFMA per clock per SM (about 1.2 TFLOP/s for the
// chip), so the DFMA kernels here are FP64-pipe bound whatever their memory
// traffic; they serve problems whose time the chain of diagonal blocks sets
// (tc64_applies).  Every output element is updated by exactly one thread in a
// fixed order, so results are bitwise reproducible, and the persistent batch
// (batched_dag.cu) runs the same operations on every element.  n = 777 (tile
// 128): 4.51 ms with 32 x 32 task-graph POTRFs and whole-tile solves, 1.60 ms now;
// n = 1,600 (tile 320): 7.44 and 3.37 ms.
#include "blocks.cuh"
#include "tc64.cuh"

namespace egs {

// ---- kernels --------------------------------------------------------------

// Trailing update at step k for the first gridDim.x tiles of the trailing
// triangle (enumerated row by row: (k+1,k+1), (k+2,k+1), (k+2,k+2), ...):
// C_mn -= A_mk A_nk^T in 64 x 64 sub-blocks.  grid = (tiles, (b/64)^2).
__global__ void __launch_bounds__(256) k_update_f64(Tiles tl, int k, DevStatus *st)
{
    if (failed(st)) return;
    const int b = tl.b;
    int mm, nn;
    tri_decode((int64_t)blockIdx.x, mm, nn);
    const int m = k + 1 + mm, nc = k + 1 + nn;
    const int nsub = b >> 6;
    const int sr = (int)blockIdx.y / nsub, sc = (int)blockIdx.y % nsub;
    if (m == nc && sc > sr) return;
    gemm_sub64(tl.t64(m, k) + (size_t)sr * 64 * b, b, tl.t64(nc, k) + (size_t)sc * 64 * b, b, b,
               tl.t64(m, nc) + (size_t)sr * 64 * b + sc * 64, b);
}

// The update inside a panel by its 64-column block j for the rows and columns of tile column k
// right of and below the block, one 16 x 16 sub-block per CTA (blocks on the diagonal or below
// it).  grid = (row sub-blocks, column sub-blocks).
__global__ void __launch_bounds__(256) k_inner_f64(Tiles tl, int k, int j, const DevStatus *st)
{
    if (failed(st)) return;
    __shared__ double As[16][65], Bs[16][65];
    const int b = tl.b, c0 = (j + 1) * 64 + (int)blockIdx.y * 16, pr0 = (j + 1) * 64 + (int)blockIdx.x * 16;
    if (pr0 < c0) return;
    inner16(As, Bs, tl.t64(k + pr0 / b, k) + (size_t)(pr0 % b) * b, tl.t64(k, k) + (size_t)c0 * b, b, j, c0);
}

// The same update in 32 x 32 sub-blocks, for launches too small to fill the
// GPU with 64 x 64 blocks.
__global__ void __launch_bounds__(256) k_update_f64_32(Tiles tl, int k, DevStatus *st)
{
    if (failed(st)) return;
    const int b = tl.b;
    int mm, nn;
    tri_decode((int64_t)blockIdx.x, mm, nn);
    const int m = k + 1 + mm, nc = k + 1 + nn;
    const int nsub = b >> 5;
    const int sr = (int)blockIdx.y / nsub, sc = (int)blockIdx.y % nsub;
    if (m == nc && sc > sr) return;
    gemm_sub32(tl.t64(m, k) + (size_t)sr * 32 * b, b, tl.t64(nc, k) + (size_t)sc * 32 * b, b, b,
               tl.t64(m, nc) + (size_t)sr * 32 * b + sc * 32, b);
}

static cudaError_t launch_update_f64(const Tiles &tl, int k, int64_t ntri, DevStatus *st, cudaStream_t s,
                                     KernelTimer *kt)
{
    if (ntri <= 0) return cudaSuccess;
    const int nsub = tl.b / 64;
    if (ntri * nsub * (nsub + 1) / 2 < 304) {
        const int n32 = tl.b / 32;
        EGS_LAUNCH(kt, KC_UPDATE, s, k_update_f64_32<<<dim3((unsigned)ntri, (unsigned)(n32 * n32)), 256, 0, s>>>(tl, k, st));
    } else {
        EGS_LAUNCH(kt, KC_UPDATE, s, k_update_f64<<<dim3((unsigned)ntri, (unsigned)(nsub * nsub)), 256, 0, s>>>(tl, k, st));
    }
    return cudaGetLastError();
}

cudaError_t launch_potrf_tiles_f64(double *tiles, const TileGeom &g, DevStatus *st, cudaStream_t s, KernelTimer *kt,
                                   double *winv, void *tc_scratch, double *z)
{
    const int T = g.T, nj = g.b / kF64Panel;
    const Tiles tl{tiles, nullptr, g.b, T, T};
    cudaError_t e = cudaSuccess;
    if (tc_scratch) {
        const F64Set set{nullptr, tc64_problem(tc_scratch, tl, st, z), 1, g.b, T, 0};
        F64Maps maps;
        e = make_f64_maps(set.one.panel, set.one.inner, g.b, &maps);
        F64Fork fork;
        if (e == cudaSuccess) e = fork.create(s, false);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(set.one.ctr, 0, tc64_counters(g.b, T) * sizeof(unsigned long long), s);
        for (int k = 0; k < T && e == cudaSuccess; ++k) {
            if (kt) kt->step = k;
            e = launch_panel64(maps, set, k, &fork, s, kt);
            if (e == cudaSuccess) e = launch_slice_panel64(set, k, s, kt);
            if (e == cudaSuccess) e = launch_update_tc64(maps, set, k, s, kt);
        }
    } else {
        const F64Set set{nullptr, dfma_problem(winv, tl, st, z), 1, g.b, T, 0};
        for (int k = 0; k < T && e == cudaSuccess; ++k) {
            if (kt) kt->step = k;
            for (int j = 0; j < nj && e == cudaSuccess; ++j) {
                e = launch_diag_solve64(set, k, j, s, kt);
                const unsigned cols = (unsigned)(4 * (nj - 1 - j)), rows = (unsigned)(4 * ((T - k) * nj - 1 - j));
                if (e == cudaSuccess && cols > 0) {
                    EGS_LAUNCH(kt, KC_UPDATE, s, k_inner_f64<<<dim3(rows, cols), 256, 0, s>>>(tl, k, j, st));
                    e = cudaGetLastError();
                }
            }
            if (e == cudaSuccess) e = launch_update_f64(tl, k, (int64_t)(T - k - 1) * (T - k) / 2, st, s, kt);
        }
    }
    if (e != cudaSuccess) return e;
    if (kt) kt->step = -1;
    return cudaGetLastError();
}

}  // namespace egs
