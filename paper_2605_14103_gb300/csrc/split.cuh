// FP64 contraction of the plain method on the tensor cores (split.cu): the
// operands as exact sums of seven 8-bit slices held in FP16.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "zbus_internal.cuh"

namespace zbus {

constexpr int SPLIT_S = 7;                        // slices of 8 bits
constexpr int SPLIT_PLANES = 3 * SPLIT_S + 1;     // Re, Im, Re + Im; magnitudes
constexpr int SPLIT_BITS = 55;                    // |fixed-point Re, Im| <= 2^55
// Padded unknowns the path takes.  Below, k_solve_fused_f64 runs a whole small
// solve in one launch.  From there on the path is the faster one at every
// batch (solves of 99 unknowns in us, FP64 contraction / this path: one
// scenario 461 / 272, 64 2354 / 306, 4096 6477 / 1551; 597 unknowns: 1175 /
// 411, 7733 / 467; 1197: 2079 / 683, 12867 / 717).  Above, a partial product's
// sum could leave 32 bits.
constexpr int SPLIT_MIN_NPAD = FUSED_MAX_NPAD + 1;
constexpr int SPLIT_MAX_NPAD = 12288;

inline int split_kpad(int n) { return round_up(n, 64); }
inline int split_ld(int n) { return round_up(n, 8); }   // rows of the partial products
inline bool split_size_ok(int n_pad) {
  return n_pad >= SPLIT_MIN_NPAD && n_pad <= SPLIT_MAX_NPAD;
}

inline size_t split_ops_bytes(int n) {
  return (size_t)SPLIT_PLANES * n * split_kpad(n) * 2 + (size_t)n * sizeof(double);
}

// The independent parts of a network (unknowns that its admittances join; Z is
// zero between two parts), from the sparse rows of Y_LL (host): the unknowns
// part by part, and each unknown's range of that list.
zbus_status split_parts(zbus_network net, const std::vector<int32_t>& ptr,
                        const std::vector<int32_t>& col, cudaStream_t st);

size_t split_scratch_bytes(int n, int64_t rows);
zbus_status split_scratch_bind(SplitScratch* s, void* base, int n, int64_t rows);

// The slices of a matrix given by its 3M copies (row-major [n_pad][n_pad],
// read by the sweeps too) and its parts (split_parts).
zbus_status split_pack(SplitOps* ops, const double* Zr, const double* Zi, int n, int n_pad,
                       const int2* part, const int32_t* part_col, cudaStream_t st);
void split_release(SplitOps* ops);

// The checked build's wait limit (zbus_checked_set_wait).
cudaError_t split_set_wait(uint64_t wait_ns);

// First operand of a solve (after k_init / k_adj_init wrote the context, its
// list and the start), and one sweep of up to `batch` scenarios: contraction,
// then update, stop test, active list and the next operand.  adjoint: the
// operand is conj(lambda) of the load gradient and the no-load term is zero.
void split_fill_ctx(SolveCtx* h, const SplitScratch& s);
void launch_split_first(SolveCtx* ctx, int n, int64_t batch, int64_t rows, bool adjoint,
                        cudaStream_t st);
zbus_status launch_split_gemm(SolveCtx* ctx, const SplitScratch& s, const SplitOps& ops, int n,
                              int64_t batch, cudaStream_t st);
void launch_split_step(SolveCtx* ctx, const SplitOps& ops, const double2* w, int n, int64_t batch,
                       int64_t rows, bool adjoint, cudaGraphConditionalHandle h, bool use_handle,
                       cudaStream_t st);

}  // namespace zbus
