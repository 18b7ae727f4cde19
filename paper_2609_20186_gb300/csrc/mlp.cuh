// mlp.cuh -- host interface of the tensor-core two-layer probe (mlp.cu), used by the step entry points.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace switchsd {

constexpr int kMaxMlpSplit = 16;    // parts of K
constexpr int kMaxMlpChunks = 8;    // 64-element K chunks staged per CTA: d <= 16 * 8 * 64 = 8192
constexpr int kMaxMlpHidden = 1024; // H1
constexpr int kMlpNMin = 64;        // hidden units of the smaller tile (the larger has twice as many)

// Parts of K for hidden size d: the most partial sums per (row, unit).
int mlp_split(int d);
// CTAs per tile of 128 rows x 64 or 128 units, each with an equal share of the parts: the partial sums per (row,
// unit) of a launch.  A power of two, at most mlp_split(d).
int mlp_ctas_per_tile(int B, int d, int H1, int sms);
// Chunks a CTA stages at once when the rescan kernel runs beside the launch with `beside` bytes of shared memory an SM
// (0: all of them).
int mlp_stages_beside(int B, int d, int H1, int S, int sms, size_t beside);
// Whether (d, H1) is within the kernel's limits.
bool mlp_shape_ok(int d, int H1);
// H1 rounded up to the smaller tile's 64 units: the row stride of the partial sums.
int mlp_hidden_padded(int H1);
// part [S][B][mlp_hidden_padded(H1)] <- split-K partial sums of W1 h (fp32; units >= H1 are zero), S =
// mlp_ctas_per_tile(...).  Launched with programmatic stream serialization; prefetch: the hidden states and W1 may be
// read (and the MMAs run) before the preceding kernel finishes (the caller's guarantee,
// SWITCHSD_PREFETCH_PROBE), and the next kernel is released at once; the stores wait.  stages:
// operand chunks staged at once per CTA (0 or >= the CTA's chunks: all of them; fewer leave shared memory
// to a kernel that runs beside this one).
cudaError_t launch_mlp_tc(const uint16_t *hidden, const uint16_t *W1, float *part, int B, int d, int H1, int S,
                          bool prefetch, cudaStream_t stream, int stages = 0);

}  // namespace switchsd
