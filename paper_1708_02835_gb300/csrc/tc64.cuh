// Host interface of the FP64 trailing update on the tensor cores (tc64.cu).
#pragma once
#include "egs_internal.cuh"

namespace egs {

constexpr int kF64Slices = 7;

// The sliced panel of one step: slice i of panel row r (row r of tiles k + 1 .. T - 1, in
// order) at slices[(i R + r) b ..], R = (T - 1) b, and the row's exponent.
struct F64Panel {
    uint16_t *slices;
    int *exps;
};
struct F64Maps {
    CUtensorMap a, b;
};

// FP64 factorisations take the tensor cores above this many rows.  Below it the chain of
// diagonal tiles sets the time (n = 1,600: update 1.1 of 6.2 ms), and the persistent batch,
// which runs the DFMA routines, stays bit for bit equal to a single evaluation; above it the
// update does (n = 5,000: 36.4 of 57 ms with DFMA, 1.6 here).
constexpr int64_t kTc64MinRows = 2049;
inline bool tc64_applies(int64_t n, int b, int T) { return n >= kTc64MinRows && T > 1 && b % 64 == 0; }

// Device scratch of one tensor-core FP64 factorisation.
size_t tc64_scratch_bytes(int b, int T);
struct F64Scratch {
    F64Panel panel;
    unsigned long long *counters;  // one work counter per launch
};
F64Scratch tc64_scratch(void *base, int b, int T);

cudaError_t make_f64_maps(const F64Panel &p, int b, int T, F64Maps *maps);
// Slices of the solved panel tiles (m0 .. T - 1, k).
cudaError_t launch_slice_panel64(const Tiles &tl, int k, int m0, const F64Panel &p, const DevStatus *st, cudaStream_t s,
                                 KernelTimer *kt);
// C_mn -= P_m P_n^T for n = col0 .. col1 - 1, m = n .. T - 1.  counter: a zeroed word;
// reserve: SMs left to other streams.
cudaError_t launch_update_tc64(const F64Maps &maps, const Tiles &tl, int k, int col0, int col1, const F64Panel &p,
                               unsigned long long *counter, int reserve, DevStatus *st, cudaStream_t s, KernelTimer *kt);

}  // namespace egs
