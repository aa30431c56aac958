// Persistent batched scheduler for FP64 batches: every problem's tile
// algorithm (Algorithm 2: Matern generation, the tile Cholesky of Section 5.2,
// the forward solve with the log-determinant and the dot product, Eq. 1) is
// expanded into one list of tile tasks, and ONE kernel launch executes the
// whole list.  Each CTA repeatedly claims the next task from a global counter
// and, before running it, waits until the tile counters it depends on have
// reached the values the task needs:
//
//   GEN(i, j)       tile (i, j) of Sigma; GEN(i, i) also copies z block i
//   POTRF(k)        needs the k updates of tile (k, k); also solves z block k and
//                   forms the tile's log-determinant and dot product
//   TRSM(m, k)      needs POTRF(k), the k updates of tile (m, k) and GEN(m, m) (z
//                   block m); also takes tile (m, k)'s product with y_k off z block m
//   UPDATE(m, n, k) needs TRSM(m, k), TRSM(n, k) and updates 0..k-1 of (m, n)
//                   (so the updates of a tile are applied in step order)
//   FINAL           needs POTRF(T - 1); assembles l (Eq. 1)
//
// Tile counter (i, j) counts 1 for its generation, 1 per update applied and 1
// when it is final (after POTRF or TRSM).  The products into z block m need no
// counter: TRSM(m, k + 1) waits for an update that waits for TRSM(m, k).
//
// The list is built on the host in a topological order (checked on the host
// by replaying it sequentially), so the lowest unfinished task always has its
// dependencies done: a CTA only waits for tasks that running CTAs have
// already claimed, and the schedule cannot deadlock however many CTAs are
// resident.  Problems are aligned at their last step (problem p's step k sits
// at position k + Tmax - T_p), so the largest problems start first and all
// finish together.  Every wait is bounded by %globaltimer; an expired wait
// sets an abort flag that makes every CTA stop claiming tasks, and the run
// reports EGS_ERR_TIMEOUT.  A problem whose Cholesky fails still signals all
// its counters (without doing the work), so the others are not held up.
//
// The tile routines are the ones of the step-synchronous batch and of the
// single-problem FP64 path, applied in the same order to each tile, so every
// l is bitwise equal to the corresponding egs_loglik_ex result.
#include <algorithm>
#include <vector>

#include "batched.cuh"
#include "batched_dag.cuh"
#include "blocks.cuh"
#include "matern.cuh"

namespace egs {

namespace {

enum DagType { D_GEN = 0, D_POTRF, D_TRSM, D_UPDATE, D_FINAL };

// The tasks' shared memory, overlaid: one task runs at a time in a CTA.
struct GenSmem {
    egs_matern_params P;
    double T[EGS_MT_INTS];
};

union DagSmem {
    Chol64Smem chol;
    Solve64Smem<32> solve;
    GemmSmem<double> gemm;
    GenSmem gen;
    double vec[256];
};

struct DagArgs {
    const int4 *tasks;  // x = problem, y = type | (i << 16), z = j | (k << 16), w = unused
    long long ntasks;
    const BatchProblem *probs;
    DagCtl *ctl;
    int b;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Thread 0 of a CTA: wait until *c >= target.  False if the batch aborted
// (this wait or another one ran out of time).
__device__ bool dag_wait(const unsigned *c, unsigned target, DagCtl *ctl)
{
    if (ld_acquire(c) >= target) return true;
    const unsigned long long t0 = global_ns();
    const unsigned long long limit = *(volatile unsigned long long *)&ctl->limit_ns;
    for (;;) {
        __nanosleep(100);
        if (ld_acquire(c) >= target) return true;
        if (*(volatile unsigned *)&ctl->abort) return false;
        if (global_ns() - t0 > limit) {
            atomicAdd(&ctl->timeouts, 1u);
            atomicExch(&ctl->abort, 1u);
            return false;
        }
    }
}

__device__ __forceinline__ unsigned *tile_cnt(const BatchProblem &p, int i, int j)
{
    return p.cnt + tile_linear(i, j);
}

__device__ void task_gen(GenSmem &gs, const BatchProblem &pr, int b, int ti, int tj)
{
    egs_matern_params &Ps = gs.P;
    {
        const double *s = reinterpret_cast<const double *>(pr.P);
        double *d = reinterpret_cast<double *>(&Ps);
        for (int i = threadIdx.x; i < (int)(sizeof(egs_matern_params) / sizeof(double)); i += blockDim.x) d[i] = s[i];
        __syncthreads();
    }
    const double *Tab = stage_table(&Ps, pr.mtab, gs.T);
    __syncthreads();
    const int nsub = b >> 6, tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int64_t n = pr.n;
    double *tile = pr.tiles + (size_t)tile_linear(ti, tj) * b * b;
    for (int sub = 0; sub < nsub * nsub; ++sub) {
        const int sr = sub / nsub, sc = sub % nsub;
        const int64_t gj = (int64_t)tj * b + sc * 64 + tx;
        const double xj = gj < n ? pr.X[gj] : 0.0, yj = gj < n ? pr.Y[gj] : 0.0;
        for (int rr = 0; rr < 16; ++rr) {
            const int r = sr * 64 + ty + 4 * rr;
            const int64_t gi = (int64_t)ti * b + r;
            double v;
            if (gi >= n || gj >= n) v = (gi == gj) ? 1.0 : 0.0;
            else if (gi == gj) v = Ps.th1;
            else v = matern_pair(&Ps, Tab, pr.X[gi], pr.Y[gi], xj, yj);
            tile[(size_t)r * b + sc * 64 + tx] = v;
        }
    }
    if (ti == tj)
        for (int r = threadIdx.x; r < b; r += blockDim.x) {
            const int64_t i = (int64_t)ti * b + r;
            pr.zpad[i] = i < n ? pr.z[i] : 0.0;
        }
}

// The rows below a 64-column block j of tile column k in one tile, 32 at a time: X and the
// products with y off z (the block of z those rows belong to), as k_solve64.
__device__ __forceinline__ void solve_tile_rows(Solve64Smem<32> &sm, const BatchProblem &pr, double *tile, int b, int k,
                                                int j, int row0, double *z)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const double *L = pr.tiles + (size_t)tile_linear(k, k) * b * b + (size_t)j * 64 * (b + 1);
    const double *y = pr.zpad + (size_t)k * b + j * 64;
    __syncthreads();
    solve64_stage(sm, L, b, pr.winv + ((size_t)k * (b / 64) + j) * kWinvDoubles);
    const double y0 = y[2 * lane], y1 = y[2 * lane + 1];
    for (int r0 = row0; r0 < b; r0 += 32) {
        double *X = tile + (size_t)r0 * b + j * 64;
        for (int e = tid; e < 32 * 64; e += 256) sm.Xs[e >> 6][e & 63] = X[(size_t)(e >> 6) * b + (e & 63)];
        __syncthreads();
        solve64_rows(sm);
        __syncthreads();
        for (int r = tid >> 5; r < 32; r += 8) {
            const double x0 = sm.Xs[r][2 * lane], x1 = sm.Xs[r][2 * lane + 1];
            X[(size_t)r * b + 2 * lane] = x0;
            X[(size_t)r * b + 2 * lane + 1] = x1;
            const double v = dot64(x0, x1, y0, y1);
            if (lane == 0) z[r0 + r] -= v;
        }
        __syncthreads();
    }
}

// The update of a tile's columns right of block j by its solved columns (K = 64), as
// k_inner_f64; diag: the diagonal tile itself, blocks from its diagonal down.
__device__ __forceinline__ void inner_update(GemmSmem<double> &sm, double *tile, const double *diag_tile, int b, int j,
                                             bool diag)
{
    const int nj = b >> 6;
    for (int c = j + 1; c < nj; ++c)
        for (int r = diag ? c : 0; r < nj; ++r)
            gemm_sub64_s(sm, tile + (size_t)r * 64 * b + j * 64, b, diag_tile + (size_t)c * 64 * b + j * 64, b, 64,
                         tile + (size_t)r * 64 * b + c * 64, b);
    __syncthreads();
}

// POTRF of diagonal tile k in one CTA, by the single evaluation's 64-column blocks: the same
// operations on every element in the same order, so factors are equal bit for bit.
__device__ void task_potrf(DagSmem &sm, const BatchProblem &pr, int b, int k)
{
    double *A = pr.tiles + (size_t)tile_linear(k, k) * b * b, *z = pr.zpad + (size_t)k * b;
    for (int j = 0; j < b / 64; ++j) {
        if (!diag64_block(sm.chol, A + (size_t)j * 64 * (b + 1), b, b - (j + 1) * 64, z + j * 64,
                          pr.winv + ((size_t)k * (b / 64) + j) * kWinvDoubles, (int64_t)k * b + j * 64, pr.st))
            return;
        __syncthreads();
        if ((j + 1) * 64 < b) {
            solve_tile_rows(sm.solve, pr, A, b, k, j, (j + 1) * 64, z);
            inner_update(sm.gemm, A, A, b, j, true);
        }
    }
    __syncthreads();
    logdet_quad_tile(A, b, z, sm.vec, pr.partials + k, (size_t)pr.T);
}

__device__ void task_trsm(DagSmem &sm, const BatchProblem &pr, int b, int m, int k)
{
    const double *Lkk = pr.tiles + (size_t)tile_linear(k, k) * b * b;
    double *X = pr.tiles + (size_t)tile_linear(m, k) * b * b;
    for (int j = 0; j < b / 64; ++j) {
        solve_tile_rows(sm.solve, pr, X, b, k, j, 0, pr.zpad + (size_t)m * b);
        inner_update(sm.gemm, X, Lkk, b, j, false);
    }
}

__device__ void task_update(DagSmem &sm, const BatchProblem &pr, int b, int m, int nc, int k)
{
    const size_t bb = (size_t)b * b;
    const double *Am = pr.tiles + (size_t)tile_linear(m, k) * bb;
    const double *An = pr.tiles + (size_t)tile_linear(nc, k) * bb;
    double *C = pr.tiles + (size_t)tile_linear(m, nc) * bb;
    const int nsub = b >> 6;
    for (int sr = 0; sr < nsub; ++sr)
        for (int sc = 0; sc < nsub; ++sc) {
            if (m == nc && sc > sr) continue;
            gemm_sub64_s(sm.gemm, Am + (size_t)sr * 64 * b, b, An + (size_t)sc * 64 * b, b, b,
                         C + (size_t)sr * 64 * b + sc * 64, b);
        }
}

// l from the log-det and dot partials (as k_finalize / kb_finalize).
__device__ void task_final(DagSmem &sm, const BatchProblem &pr)
{
    double *red = sm.vec;
    double s = 0.0, q = 0.0;
    for (int t = threadIdx.x; t < pr.T; t += 256) {
        s += pr.partials[t];
        q += pr.partials[pr.T + t];
    }
    const double lsum = block_sum(s, red);
    __syncthreads();
    const double qsum = block_sum(q, red);
    if (threadIdx.x == 0) {
        DevStatus *st = pr.st;
        if (failed(st)) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            st->result[0] = st->result[1] = st->result[2] = nan;
        } else {
            const double logdet = 2.0 * lsum;
            st->result[0] = -0.5 * qsum - 0.5 * logdet - 0.5 * (double)pr.n * 1.8378770664093454836;
            st->result[1] = logdet;
            st->result[2] = qsum;
        }
    }
}

// Thread 0: the waits of one task.
__device__ bool task_wait(int type, int i, int j, int k, const BatchProblem &pr, DagCtl *ctl)
{
    switch (type) {
    case D_POTRF: return dag_wait(tile_cnt(pr, k, k), (unsigned)k + 1, ctl);
    case D_TRSM:  // (i, i) generated: z block i is there
        return dag_wait(tile_cnt(pr, k, k), (unsigned)k + 2, ctl) && dag_wait(tile_cnt(pr, i, k), (unsigned)k + 1, ctl) &&
               dag_wait(tile_cnt(pr, i, i), 1u, ctl);
    case D_UPDATE:
        return dag_wait(tile_cnt(pr, i, k), (unsigned)k + 2, ctl) && dag_wait(tile_cnt(pr, j, k), (unsigned)k + 2, ctl) &&
               dag_wait(tile_cnt(pr, i, j), (unsigned)k + 1, ctl);
    case D_FINAL: return dag_wait(tile_cnt(pr, pr.T - 1, pr.T - 1), (unsigned)pr.T + 1, ctl);
    default: return true;  // D_GEN
    }
}

// Thread 0, after the task's work: release its counter(s).
__device__ void task_signal(int type, int i, int j, int k, const BatchProblem &pr)
{
    __threadfence();
    switch (type) {
    case D_GEN: atomicAdd(tile_cnt(pr, i, j), 1u); break;
    case D_POTRF: atomicAdd(tile_cnt(pr, k, k), 1u); break;
    case D_TRSM: atomicAdd(tile_cnt(pr, i, k), 1u); break;
    case D_UPDATE: atomicAdd(tile_cnt(pr, i, j), 1u); break;
    default: break;
    }
}

__global__ void __launch_bounds__(256, 2) kb_dag(DagArgs a)
{
    __shared__ int4 s_task;
    __shared__ long long s_idx;
    __shared__ int s_go, s_skip;
    __shared__ DagSmem sm;
    for (;;) {
        if (threadIdx.x == 0) {
            int go = 0;
            if (!*(volatile unsigned *)&a.ctl->abort) {
                const long long t = (long long)atomicAdd(&a.ctl->next, 1ull);
                if (t < a.ntasks) {
                    s_task = a.tasks[t];
                    s_idx = t;
                    go = 1;
                }
            }
            s_go = go;
        }
        __syncthreads();
        if (!s_go) return;
        const int4 tk = s_task;
        const long long idx = s_idx;
        const BatchProblem &pr = a.probs[tk.x];
        const int type = tk.y & 0xFFFF, i = tk.y >> 16, j = tk.z & 0xFFFF, k = tk.z >> 16;
        if (threadIdx.x == 0) {
            s_go = task_wait(type, i, j, k, pr, a.ctl) ? 1 : 0;
            s_skip = failed(pr.st) ? 1 : 0;
        }
        __syncthreads();
        if (!s_go) return;
        if (!s_skip || type == D_FINAL) {
            switch (type) {
            case D_GEN: task_gen(sm.gen, pr, a.b, i, j); break;
            case D_POTRF: task_potrf(sm, pr, a.b, k); break;
            case D_TRSM: task_trsm(sm, pr, a.b, i, k); break;
            case D_UPDATE: task_update(sm, pr, a.b, i, j, k); break;
            case D_FINAL: task_final(sm, pr); break;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && idx != *(volatile long long *)&a.ctl->withhold) task_signal(type, i, j, k, pr);
    }
}

inline int4 pack(int prob, int type, int i, int j, int k) { return make_int4(prob, type | (i << 16), j | (k << 16), 0); }

}  // namespace

egs_status dag_plan(const std::vector<int> &T, int b, std::vector<int4> &tasks, std::vector<size_t> &cnt_off,
                    size_t &ncounters)
{
    const int np = (int)T.size();
    if (b > 256 || b % 64) return set_error(EGS_ERR_ARG, "persistent batch: tile %d must be 64, 128, 192 or 256", b);
    int Tmax = 0;
    cnt_off.resize(np);
    ncounters = 0;
    for (int p = 0; p < np; ++p) {
        if (T[p] > 32767) return set_error(EGS_ERR_ARG, "persistent batch: %d tiles per side is too many", T[p]);
        Tmax = std::max(Tmax, T[p]);
        cnt_off[p] = ncounters;
        ncounters += (size_t)T[p] * (T[p] + 1) / 2;
    }
    tasks.clear();
    // position key = k + Tmax - T_p; generation at key - 1.  Within a key:
    // POTRF, TRSM, UPDATE, FINAL, each over all problems.
    for (int key = -1; key < Tmax; ++key) {
        for (int p = 0; p < np; ++p) {
            const int k = key - (Tmax - T[p]) + 1;  // generation precedes step 0
            if (k == 0)
                for (int i = 0; i < T[p]; ++i)
                    for (int j = 0; j <= i; ++j) tasks.push_back(pack(p, D_GEN, i, j, 0));
        }
        for (int rank = 0; rank < 4; ++rank)
            for (int p = 0; p < np; ++p) {
                const int k = key - (Tmax - T[p]);
                if (k < 0 || k >= T[p]) continue;
                const int Tp = T[p];
                switch (rank) {
                case 0: tasks.push_back(pack(p, D_POTRF, k, k, k)); break;
                case 1:
                    for (int m = k + 1; m < Tp; ++m) tasks.push_back(pack(p, D_TRSM, m, k, k));
                    break;
                case 2:
                    for (int m = k + 1; m < Tp; ++m)
                        for (int n = k + 1; n <= m; ++n) tasks.push_back(pack(p, D_UPDATE, m, n, k));
                    break;
                case 3:
                    if (k == Tp - 1) tasks.push_back(pack(p, D_FINAL, 0, 0, 0));
                    break;
                }
            }
    }
    // Replay the list sequentially: every wait must already hold from the
    // tasks before it (so the ordered claiming cannot deadlock), and every
    // counter must end at its final value.
    std::vector<unsigned> c(ncounters, 0);
    auto tc = [&](int p, int i, int j) -> unsigned & { return c[cnt_off[p] + (size_t)i * (i + 1) / 2 + j]; };
    for (size_t t = 0; t < tasks.size(); ++t) {
        const int4 tk = tasks[t];
        const int p = tk.x, type = tk.y & 0xFFFF, i = tk.y >> 16, j = tk.z & 0xFFFF, k = tk.z >> 16;
        const unsigned uk = (unsigned)k;
        bool ok = true;
        switch (type) {
        case D_GEN: ++tc(p, i, j); break;
        case D_POTRF: ok = tc(p, k, k) >= uk + 1; ++tc(p, k, k); break;
        case D_TRSM:
            ok = tc(p, k, k) >= uk + 2 && tc(p, i, k) >= uk + 1 && tc(p, i, i) >= 1;
            ++tc(p, i, k);
            break;
        case D_UPDATE:
            ok = tc(p, i, k) >= uk + 2 && tc(p, j, k) >= uk + 2 && tc(p, i, j) >= uk + 1;
            ++tc(p, i, j);
            break;
        case D_FINAL: ok = tc(p, T[p] - 1, T[p] - 1) >= (unsigned)T[p] + 1; break;
        }
        if (!ok) return set_error(EGS_ERR_ARG, "persistent batch: task %zu of the plan is not in dependency order", t);
    }
    for (int p = 0; p < np; ++p)
        for (int i = 0; i < T[p]; ++i)
            for (int j = 0; j <= i; ++j)
                if (tc(p, i, j) != (unsigned)j + 2) return set_error(EGS_ERR_ARG, "persistent batch: incomplete plan");
    return EGS_OK;
}

int dag_grid()
{
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kb_dag, 256, 0) != cudaSuccess || per < 1) per = 1;
    return sms * per;
}

cudaError_t dag_enqueue(const int4 *d_tasks, long long ntasks, const BatchProblem *d_probs, DagCtl *d_ctl, int b,
                        int grid, cudaStream_t s)
{
    DagArgs a{d_tasks, ntasks, d_probs, d_ctl, b};
    kb_dag<<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace egs
