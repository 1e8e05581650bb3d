// Delta-encoded host batches: each request's prompt is its base request's prompt followed
// by its own delta tokens (an agentic turn extends the session's previous turn; the
// samples of a prompt group repeat one prompt).  After the deltas have been copied to the
// device, this kernel rebuilds the full token array of the batch, so the routing kernels
// see exactly the batch the encoding describes.  No counterpart in the paper: an input
// encoding of the host path.
//
// A CTA per request: one thread walks the chain r -> base(r) -> ... -> root (its depth is
// checked on the host); then the warps copy the deltas in pieces of 512 tokens, which are all
// independent (the host computed the full offsets, and where a delta begins in the prompt is the
// length of its base's prompt).  Copies start at any word on both sides, so they are 4-byte loads, 16 a
// lane in flight; with one in flight, a warp per request, the longest prompts of an 8,192-request
// batch (17K tokens) took 172 us, beside the route of the batch before.
#include "common.cuh"
#include "kernels.h"

namespace misat {

namespace {
constexpr int kExpandWarps = 4;
constexpr int kExpandPer = 16;  // tokens per lane and piece
}  // namespace

__global__ void __launch_bounds__(32 * kExpandWarps) k_delta_expand(DeltaArgs a) {
  __shared__ int32_t s_chain[kDeltaMaxDepth], s_at[kDeltaMaxDepth], s_depth;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int r = blockIdx.x; r < a.n; r += gridDim.x) {
    __syncthreads();  // the last request's chain has been read
    if (threadIdx.x == 0) {
      int depth = 0;
      for (int e = r; e >= 0 && depth < kDeltaMaxDepth; ++depth) {
        const int b = a.base[e];
        s_chain[depth] = e;
        s_at[depth] = b >= 0 ? (int32_t)(a.tok_off[b + 1] - a.tok_off[b]) : 0;
        e = b;
      }
      s_depth = depth;
    }
    __syncthreads();
    int32_t* out = a.tokens + a.tok_off[r];
    const int len = (int)(a.tok_off[r + 1] - a.tok_off[r]);
    const int depth = s_depth;
    for (int i = 0; i < depth; ++i) {
      const int e = s_chain[i], at = s_at[i];
      const int64_t d0 = a.doff[e];
      int d = (int)(a.doff[e + 1] - d0);
      if (at + d > len) d = len - at;  // never for a well-formed encoding (host-checked)
      const int32_t* src = a.dtok + d0;
      // the pieces of a prompt's deltas go round the warps
      for (int j0 = 32 * kExpandPer * ((wid + i) % kExpandWarps); j0 < d; j0 += 32 * kExpandPer * kExpandWarps) {
        int32_t v[kExpandPer];
#pragma unroll
        for (int u = 0; u < kExpandPer; ++u) {
          const int j = j0 + 32 * u + lane;
          v[u] = j < d ? src[j] : 0;
        }
#pragma unroll
        for (int u = 0; u < kExpandPer; ++u) {
          const int j = j0 + 32 * u + lane;
          if (j < d) out[at + j] = v[u];
        }
      }
    }
  }
}

void launch_delta_expand(const DeltaArgs& a, int num_sms, cudaStream_t st) {
  if (a.n <= 0) return;
  const int grid = a.n < num_sms * 16 ? a.n : num_sms * 16;
  k_delta_expand<<<grid, 32 * kExpandWarps, 0, st>>>(a);
}

}  // namespace misat
