// One-time derived tables of a block: per-output-channel step-size products and zero-point corrections of
// every (linear layer, branch) pair, and the relative-position bias expanded to the attention kernel's fragment order.
#include "kernels.h"
#include <cfloat>

namespace mixaq {

// one warp per output channel: mult[n] = s_a * s_w[n];
// pre[n] = 0x4B400000 - z_a * sum_k w[n][k], what the GEMM's epilogue adds to the raw sums (see acc_to_float2);
// bound[n]: no dequantized sum |mult * acc| exceeds its magnitude; negative where |acc| could reach the 2^22 that `pre` leaves
// room for.  The codes lie in 0 .. qmax, so acc = sum_k w (a - z) is largest with a = qmax where w > 0 and a = 0 elsewhere, and
// smallest the other way round: half of qmax * sum |w| for a zero point in the middle of the range or weights of either sign alike.
__global__ void __launch_bounds__(256) k_prepare_linear(const int8_t* __restrict__ w, const float* __restrict__ sw,
                                                        int N, int K, float sa, int za, int qmax, float* mult, int32_t* pre,
                                                        float* bound) {
  int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (n >= N) return;
  int up = 0, down = 0;                                     // sum of the positive weights, of the negative ones
  for (int k = lane; k < K; k += 32) { const int c = (int)w[(long)n * K + k]; up += c > 0 ? c : 0; down += c < 0 ? -c : 0; }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    up += __shfl_xor_sync(0xffffffffu, up, off);
    down += __shfl_xor_sync(0xffffffffu, down, off);
  }
  if (lane == 0) {
    pre[n] = (int32_t)(kMagicBits - (uint32_t)(za * (up - down)));
    mult[n] = __fmul_rn(sa, sw[n]);
    const long hi = (long)up * (qmax - za) + (long)down * za, lo = (long)up * za + (long)down * (qmax - za), most = hi > lo ? hi : lo;
    const float limit = fabsf(mult[n]) * (float)most * 1.0001f;
    // (a step that is no number leaves no bound: its column takes the contract's own operations either way)
    bound[n] = most < (1L << 22) - 16 ? limit : limit > 0.0f ? -limit : limit == limit ? -FLT_MIN : -INFINITY;
  }
}

// Relative-position bias in the order the attention kernel's accumulator fragments want it:
// out[(((h*4 + mt)*7 + nt)*2 + r)*32 + lane] = float2 of bias[h][i][j] at (i, j) = (16mt+g+8r, 8nt+2t), (16mt+g+8r, 8nt+2t+1)
// with g = lane/4, t = lane%4, so that a warp reads a row half of a tile as 256 consecutive bytes; 0 outside the 49 x 49
// table, where
// bias[h][i][j] = table[((yi - yj + 6) * 13 + (xi - xj + 6)) * heads + h].
__global__ void k_prepare_relbias(const float* __restrict__ table, int heads, float* out) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= heads * 4 * 7 * 32 * 4) return;
  const int comp = (idx & 1) | ((idx >> 6 & 1) << 1), lane = (idx >> 1) & 31;
  const int tile = idx >> 7;                       // (h*4 + mt)*7 + nt
  const int nt = tile % 7, mt = (tile / 7) & 3, h = tile / 28;
  const int i = 16 * mt + (lane >> 2) + 8 * (comp >> 1);
  const int j = 8 * nt + 2 * (lane & 3) + (comp & 1);
  float v = 0.0f;
  if (i < WT && j < WT) {
    int dy = i / WS - j / WS + (WS - 1), dx = i % WS - j % WS + (WS - 1);
    v = table[(dy * (2 * WS - 1) + dx) * heads + h];
  }
  out[idx] = v;
}

void launch_prepare_linear(const int8_t* w, const float* sw, int N, int K, float sa, int za, int bits, float* mult,
                           int32_t* pre, float* bound, cudaStream_t st) {
  k_prepare_linear<<<(N + 7) / 8, 256, 0, st>>>(w, sw, N, K, sa, za, (1 << bits) - 1, mult, pre, bound);
  ++g_launches;
}

void launch_prepare_relbias(const float* table, int heads, float* out, cudaStream_t st) {
  int n = heads * 4 * 7 * 32 * 4;
  k_prepare_relbias<<<(n + 255) / 256, 256, 0, st>>>(table, heads, out);
  ++g_launches;
}

}  // namespace mixaq
