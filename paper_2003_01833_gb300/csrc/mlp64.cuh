// Parameter order of the H = 64 warm-start network and the order of a
// gradient partial row of its kernels (mlp64.cu), for the kernel that sums the
// rows (mlp.cu).
#pragma once

namespace tagi {
namespace mlp64 {

constexpr int kF = 8, kH = 64;
// parameters: W1 (H x F), b1, W2 (H x H), b2, W3, b3
constexpr int oW1 = 0, oB1 = kH * kF, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + kH;
constexpr int kParams = oB3 + 1;  // 4801

// A partial row has its own order, so that the folds' reads and writes are
// coalesced (lane r of TMEM, one column after another): W2[r][c] at c * 64 + r,
// then b2, W1[r][f] at f * 64 + r, b1, W3, b3 and the loss.
constexpr int pW2 = 0, pB2 = kH * kH, pW1 = pB2 + kH, pB1 = pW1 + kH * kF, pW3 = pB1 + kH, pB3 = pW3 + kH,
              pLoss = pB3 + 1;
static_assert(pLoss == kParams, "the same entries, then the loss");

// entry of the row that holds parameter e (e = kParams: the loss)
__device__ __forceinline__ int slot(int e)
{
    if (e < oB1) return pW1 + (e % kF) * kH + e / kF;
    if (e < oW2) return pB1 + e - oB1;
    if (e < oB2) return pW2 + ((e - oW2) % kH) * kH + (e - oW2) / kH;
    if (e < oW3) return pB2 + e - oB2;
    if (e < oB3) return pW3 + e - oW3;
    return e == oB3 ? pB3 : pLoss;
}

}  // namespace mlp64
}  // namespace tagi
