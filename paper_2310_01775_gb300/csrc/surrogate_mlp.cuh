// One-launch surrogate rollout and its reverse sweep (surrogate_mlp.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "mlp.cuh"
#include "stamp_internal.cuh"

namespace stamp {
namespace mlp {

struct SurArgs {
    const float* theta;              // N x D
    int N, n_tiles;                  // n_tiles = ceil(N / 128)
    uint64_t seed;
    int iter;                        // < 0: no Gumbel noise
    const unsigned char *w_tiled, *wt_tiled;
    const float* bias;
    // H x N x 3 n_blocks: q_k, all of them when zsave is given, else q_{H-1} only
    float* pose;
    float* y;                        // N x 3 n_blocks: the last push's pose change
    float* relax;                    // N x H x (M + 2): all when zsave is given, else the sigmoids only
    unsigned char* zsave;            // pre-activation tiles of push k at k n_tiles + tile, or NULL
    int tile_cap;
    const float* apose;              // reverse: dC/dq_H, N x 3 n_blocks
    float* grad;                     // reverse: N x D
    int* err;
};
cudaError_t surrogate_pass(const SimConst& sc, const SurArgs& a, bool reverse, int sms, cudaStream_t st);

// An MLP's buffers.
struct View {
    const unsigned char *w_tiled, *wt_tiled;
    const float* bias;
    unsigned char* zsave;
    int tile_cap, sm_count;
    int* err;
};
View view(const stamp_mlp* m);

}  // namespace mlp
}  // namespace stamp
