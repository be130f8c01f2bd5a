// Internal: projections of a few rows (gemm_skinny_sm100.cu): 128 weight rows against all rows of x per thread-block
// cluster, K split over the cluster's blocks, partial tiles summed through distributed shared memory.
#pragma once
#include "common.cuh"
#include "gemm_skinny_layout.cuh"

namespace relaxkv {

// Where the features of y = x W^T go: segment i takes features [col0[i], col0[i + 1]) and is a row-major matrix of that
// width of its own (+ an optional residual of the same shape).  Segment widths are multiples of 8.
struct SkinnyOut {
  uint16_t* y[3];
  const uint16_t* residual[3];
  int col0[4];
  int n;
};

// x [n_rows <= 128, n_in], weight [n_out, n_in].  swiglu != 0: weight is the gate/up-tiled matrix of relaxkv_linear_swiglu
// (n_out = 2 x inter rows) and the one output is [n_rows, n_out / 2].  Arguments are validated by the caller.
relaxkv_status launch_gemm_skinny(const void* x, const void* weight, const SkinnyOut& outs, int n_rows, int n_out, int n_in,
                                  int swiglu, cudaStream_t stream);

}  // namespace relaxkv
