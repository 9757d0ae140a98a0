// sgtv_rules.h -- dispatch rules over sizes alone, plain C++ (no CUDA), so that
// they can be checked on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SGTV_RULE __host__ __device__ constexpr
#else
#define SGTV_RULE constexpr
#endif

namespace sgtv {

// Pieces that a plane (sample, channel) of n elements is cut into for the loss
// head: one where the planes alone fill `blocks` blocks, else enough to, of at
// least 1024 elements (four a thread). A sample of one channel, 256 x 256: 87 us with
// one block, 5.8 with 64; 16 channels 89 and 10.9; 8 samples of 320 channels, 64 x
// 64, one piece a plane either way.
SGTV_RULE int64_t mse_pieces(int64_t planes, int64_t n, int64_t blocks)
{
    const int64_t want = (blocks + planes - 1) / planes, most = (n + 1023) / 1024;
    return want < most ? want : most;
}

}  // namespace sgtv
