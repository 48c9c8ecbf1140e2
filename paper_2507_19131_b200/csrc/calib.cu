// Calibration of the activation quantizers (MixA-Q Section 4.3, post-training flow: one calibration sample, and the
// FULL feature map -- every window, not the windows a branch will later see -- initialises the step sizes of both
// branches).  The kernels below run the floating-point Two-Branch block (all quantizers off, weights = code x step)
// through ONE branch's LayerNorm parameters and biases and record the minimum and maximum of what each of the seven
// quantizer sites would see.  Arithmetic: LayerNorm, softmax and GELU exactly as in the quantized path (the same
// device functions); matrix products on the integer tensor cores, to binary64 accuracy.
#include "kernels.h"
#include "tc_ptx.cuh"

namespace mixaq {

namespace {

// order-preserving map float -> unsigned, so that integer atomics give the float minimum / maximum
__device__ __forceinline__ uint32_t ordered_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
// obs[2*site] holds the key of the minimum (starts at 0xFFFFFFFF), obs[2*site+1] that of the maximum (starts at 0)
__device__ __forceinline__ void observe_warp(uint32_t* obs, int site, float lo, float hi) {
  uint32_t klo = ordered_key(lo), khi = ordered_key(hi);
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    klo = min(klo, __shfl_xor_sync(0xffffffffu, klo, off));
    khi = max(khi, __shfl_xor_sync(0xffffffffu, khi, off));
  }
  // most warps do not move the extremes: a plain read (possibly stale, which only costs an atomic) spares the
  // serialised atomics on one address (stage-1 LayerNorm of a 200 x 334 map: 68 208 warps)
  if ((threadIdx.x & 31) == 0) {
    const uint2 seen = __ldcg(reinterpret_cast<const uint2*>(obs) + site);
    if (klo < seen.x) atomicMin(obs + 2 * site, klo);
    if (khi > seen.y) atomicMax(obs + 2 * site + 1, khi);
  }
}

__device__ __forceinline__ int cal_window_src(int b, int H, int W, int Hp, int Wp, int shift, int nwx, int w, int t) {
  const int wy = w / nwx, wx = w - wy * nwx;
  const int i = t / WS, j = t - i * WS;
  int y = wy * WS + i + shift; if (y >= Hp) y -= Hp;
  int x = wx * WS + j + shift; if (x >= Wp) x -= Wp;
  if (y >= H || x >= W) return -1;
  return (b * H + y) * W + x;
}

// Row m of the window batch (all windows of all images in natural order, 49 rows each): source token, LayerNorm of the
// real tokens, zeros for pad tokens.  rowsrc == NULL on input means "rows are already a [M][C] matrix" (LN2).
template <int NPL>
__global__ void __launch_bounds__(256) k_cal_ln(const float* __restrict__ src, int32_t* __restrict__ rowsrc_out,
                                                const float* __restrict__ gamma, const float* __restrict__ beta,
                                                float* __restrict__ out, long M, int gather, int H, int W, int shift,
                                                int nwx, int nW, uint32_t* obs, int site, int site_in) {
  constexpr int C = NPL * 32;
  const long m = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= M) return;
  long s = m;
  if (gather) {
    const int Hp = (H + WS - 1) / WS * WS, Wp = (W + WS - 1) / WS * WS;
    const long slot = m / WT;
    const int t = (int)(m - slot * WT), b = (int)(slot / nW), w = (int)(slot - (long)b * nW);
    s = cal_window_src(b, H, W, Hp, Wp, shift, nwx, w, t);
    if (lane == 0) rowsrc_out[m] = (int32_t)s;
  }
  float v[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) v[i] = s < 0 ? 0.0f : __ldg(src + s * C + lane + 32 * i);
  if (site_in >= 0) {                      // the raw input values of the real tokens (each token sits in one window)
    float ilo = INFINITY, ihi = -INFINITY;
    if (s >= 0) {
#pragma unroll
      for (int i = 0; i < NPL; ++i) { ilo = fminf(ilo, v[i]); ihi = fmaxf(ihi, v[i]); }
    }
    observe_warp(obs, site_in, ilo, ihi);
  }
  float mean, rstd;
  ln_stats<NPL>(v, (float)C, mean, rstd);
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int c = lane + 32 * i;
    const float y = s < 0 ? 0.0f : ln_apply(v[i], mean, rstd, __ldg(gamma + c), __ldg(beta + c));
    out[m * C + c] = y;
    lo = fminf(lo, y); hi = fmaxf(hi, y);
  }
  observe_warp(obs, site, lo, hi);
}

// patch-merging rows: 2x2 neighbours concatenated (zeros outside the map), LayerNorm over 4C
template <int NPL>
__global__ void __launch_bounds__(256) k_cal_merge_ln(const float* __restrict__ x, const float* __restrict__ gamma,
                                                      const float* __restrict__ beta, float* __restrict__ out,
                                                      int B, int H, int W, uint32_t* obs) {
  constexpr int K = NPL * 32, C = K / 4;
  const int H2 = (H + 1) / 2, W2 = (W + 1) / 2;
  const long tok = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (tok >= (long)B * H2 * W2) return;
  const int b = (int)(tok / ((long)H2 * W2)), r = (int)(tok - (long)b * H2 * W2);
  const int y2 = r / W2, x2 = r - y2 * W2;
  float v[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int c = lane + 32 * i, g = c / C, cc = c - g * C;
    const int yy = 2 * y2 + (g & 1), xx = 2 * x2 + (g >> 1);
    v[i] = (yy < H && xx < W) ? __ldg(x + (((long)b * H + yy) * W + xx) * C + cc) : 0.0f;
  }
  float mean, rstd;
  ln_stats<NPL>(v, (float)K, mean, rstd);
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int c = lane + 32 * i;
    const float y = ln_apply(v[i], mean, rstd, __ldg(gamma + c), __ldg(beta + c));
    out[tok * K + c] = y;
    lo = fminf(lo, y); hi = fmaxf(hi, y);
  }
  observe_warp(obs, 0, lo, hi);
}

// ---- matrix products ----------------------------------------------------------------------------------------------------
// out[m][n] = (float)( sum_k a[m][k] * w[n][k] * sw[n]  + bias[n] ) with the sum to binary64 accuracy, then per mode:
enum CalMode { CAL_QKV = 0, CAL_PROJ = 1, CAL_FC1 = 2, CAL_FC2 = 3, CAL_PLAIN = 4 };
struct CalLinearArgs {
  const float* a; const int8_t* w; const float* sw; const float* bias;   // bias nullable
  float* out;                 // QKV, FC1, PLAIN: [M][N];  PROJ: x1 [M][N];  FC2: the output feature map
  const float* res;           // PROJ: input feature map (gathered through rowsrc);  FC2: x1 [M][N]
  const int32_t* rowsrc;      // PROJ, FC2
  uint8_t* slices; int32_t* expo;   // workspace: [CAL_SLICES][M][K] bytes of the fixed-point rows, [M] their exponents or CAL_PLAIN_ROW
  long M; int N, K, C;        // C: width of one q/k/v section (QKV)
  uint32_t* obs;
  int* status;
};
// The weights are whole numbers times a step per output channel, so the product runs on the integer tensor cores, by exact integer
// slices of the operands (the Ozaki scheme): every row of `a` becomes 56-bit fixed point with the row's largest exponent, cut into
// seven bytes, the top one signed.  Each byte plane times the weight codes is an exact int32 sum; the seven sums are put together in
// integers and three binary64 values, a handful of binary64 roundings where the plain binary64 sum has one or two per product.
// The 56 bits hold every bit of a value whose exponent is at most 31 below the row's largest.  A row with a smaller value (it would
// lose bits, which are all that counts where the large ones meet weights of zero), or with an infinity or a NaN, is summed in
// binary64 instead: k_cal_split knows it, and puts its sums where the product's epilogue then reads them.
// A Swin-T calibration on a 200 x 334 map: 23.4 ms of products on the binary64 pipe (8.5 T products/s, about half of its rate),
// 5.8 ms here and 1.35 ms for the byte planes.  One block of C = 96 on that map: 0.76 ms with usual rows, 1.8 with the rows of both
// LayerNorms summed in binary64, 2.0 with all rows (20.7 with a serial loop per output in the product's epilogue).
constexpr int CAL_PLAIN_ROW = 0;         // in place of the exponent (at least 1) of a row that is summed in binary64

// The sums of a CTA's plain rows (bit r of `todo`: row first + r), before residual and GELU, into their places of the output.
// A thread has a column and four rows at a time, so that a weight is fetched and converted once for four products; a product of 24
// and 8 bits is exact in binary64, and the sums run over k in ascending order.  All threads of the CTA come here together.
constexpr int CAL_PLAIN_ROWS = 4, CAL_PLAIN_K = 128;
__device__ __noinline__ void cal_plain_rows(const CalLinearArgs& p, bool scatter, long first, uint32_t todo, double (*sa)[CAL_PLAIN_K]) {
  const int tid = threadIdx.x;
  while (todo) {
    long row[CAL_PLAIN_ROWS];
    int rows = 0;
#pragma unroll
    for (int r = 0; r < CAL_PLAIN_ROWS; ++r) {
      row[r] = todo ? first + __ffs(todo) - 1 : row[0];
      rows += todo ? 1 : 0;
      todo &= todo - 1u;                                                      // (stays 0)
    }
    for (int n0 = 0; n0 < p.N; n0 += (int)blockDim.x) {
      const int n = n0 + tid;
      const int8_t* w = p.w + (long)(n < p.N ? n : 0) * p.K;
      double s[CAL_PLAIN_ROWS] = {};
      for (int k0 = 0; k0 < p.K; k0 += CAL_PLAIN_K) {                         // K is a multiple of 32
        const int kn = min(CAL_PLAIN_K, p.K - k0);
        __syncthreads();
        if (tid < kn) {
#pragma unroll
          for (int r = 0; r < CAL_PLAIN_ROWS; ++r) sa[r][tid] = (double)__ldg(p.a + row[r] * p.K + k0 + tid);
        }
        __syncthreads();
        for (int k = 0; k < kn; k += 16) {
          const int4 w16 = __ldg(reinterpret_cast<const int4*>(w + k0 + k));
          const int w4[4] = {w16.x, w16.y, w16.z, w16.w};
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const double c = (double)(int)(int8_t)(w4[j >> 2] >> (8 * (j & 3)));
#pragma unroll
            for (int r = 0; r < CAL_PLAIN_ROWS; ++r) s[r] = __fma_rn(sa[r][k + j], c, s[r]);
          }
        }
      }
      if (n >= p.N) continue;
      const double step = (double)__ldg(p.sw + n), bias = p.bias ? (double)__ldg(p.bias + n) : 0.0;
#pragma unroll
      for (int r = 0; r < CAL_PLAIN_ROWS; ++r) {
        const long dst = scatter ? (long)__ldg(p.rowsrc + row[r]) : row[r];
        if (r < rows && dst >= 0) p.out[dst * p.N + n] = (float)__dadd_rn(__dmul_rn(s[r], step), bias);
      }
    }
  }
}

// One warp per row: the largest exponent, then the byte planes (a row of one plane is K bytes).  scatter: row m of the output is
// row rowsrc[m] (fc2).
constexpr int CAL_SPLIT_WARPS = 8;
__global__ void __launch_bounds__(32 * CAL_SPLIT_WARPS, 6) k_cal_split(const __grid_constant__ CalLinearArgs p, int scatter) {
  __shared__ double sa[CAL_PLAIN_ROWS][CAL_PLAIN_K];
  __shared__ uint32_t plain_rows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K = p.K;
  const long first = (long)blockIdx.x * CAL_SPLIT_WARPS, m = first + warp;
  if (threadIdx.x == 0) plain_rows = 0;
  __syncthreads();
  bool plain = false;
  if (m < p.M) {
    const uint4* row = reinterpret_cast<const uint4*>(p.a + m * K);
    uint32_t top = 0, low = 0xFFFFFFFFu;                      // largest magnitude; smallest but zero, minus 1
    for (int i = lane; i < K / 4; i += 32) {
      const uint4 v = __ldg(row + i);
      const uint32_t x = v.x & 0x7FFFFFFFu, y = v.y & 0x7FFFFFFFu, z = v.z & 0x7FFFFFFFu, w = v.w & 0x7FFFFFFFu;
      top = max(max(top, max(x, y)), max(z, w));
      low = min(min(low, min(x - 1u, y - 1u)), min(z - 1u, w - 1u));
    }
    const int E = max(1, (int)(__reduce_max_sync(0xffffffffu, top) >> 23));
    const uint32_t least = __reduce_min_sync(0xffffffffu, low);
    plain = E == 255 || (least != 0xFFFFFFFFu && max(1, (int)((least + 1u) >> 23)) < E - 31);
    if (lane == 0) {
      p.expo[m] = plain ? CAL_PLAIN_ROW : E;
      if (plain) atomicOr(&plain_rows, 1u << warp);
    }
    for (int i = plain ? K : lane; i < K / 4; i += 32) {      // (what the planes of a plain row hold does not matter)
      const uint4 v = __ldg(row + i);
      const uint32_t in[4] = {v.x, v.y, v.z, v.w};
      uint32_t lo[4], hi[4];                                  // 56-bit two's complement: bytes 0-3 and 4-6
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int e = (in[j] >> 23) & 255;
        const long long f = (in[j] & 0x7FFFFFu) | (e ? 0x800000u : 0u);
        long long q = f << max((e ? e : 1) - E + 31, 0);      // 0 ... 31; below 0 for zeros only
        if (in[j] >> 31) q = -q;
        lo[j] = (uint32_t)q; hi[j] = (uint32_t)(q >> 32);
      }
#pragma unroll
      for (int s = 0; s < CAL_SLICES; ++s) {
        const uint32_t* x = s < 4 ? lo : hi;
        const uint32_t sel = (uint32_t)(s & 3) | (uint32_t)((s & 3) + 4) << 4;
        reinterpret_cast<uint32_t*>(p.slices + ((long)s * p.M + m) * K)[i] =
            __byte_perm(__byte_perm(x[0], x[1], sel), __byte_perm(x[2], x[3], sel), 0x5410);
      }
    }
  }
  if (__syncthreads_or(plain)) cal_plain_rows(p, scatter != 0, first, plain_rows, sa);
}

// Persistent, one CTA per SM: warp 0 TMA, warp 1 MMA, sixteen epilogue warps (a lane quarter and 16 columns each).
// A 128 x 64 tile has seven accumulators of 64 TMEM columns, one per byte plane.  Per 128 codes of k the weight tile is loaded
// once and met by the seven activation tiles, which are what the loads are made of (16 KB each against 140 cycles of MMA): the
// width of 64 is the largest with which seven accumulators fit.  What bounds it up to K = 384 is the epilogue (seven TMEM loads,
// eight binary64 operations and two conversions an output: 16 warps 5.8 ms, 8 warps with the loop unrolled 7.9), then the loads.
// Sums of more than CAL_KCHUNK products, which int32 might not hold, are drained in parts.
constexpr int CG_BM = 128, CG_BN = 64, CG_BK = 128, CG_A_RING = 8, CG_B_RING = 4, CAL_KCHUNK = 32768;
constexpr int CG_A_BYTES = CG_BM * CG_BK, CG_B_BYTES = CG_BN * CG_BK, CG_EPI_WARPS = 16, CG_THREADS = 32 * (2 + CG_EPI_WARPS);
constexpr int CG_EPI_COLS = CG_BN / (CG_EPI_WARPS / 4);
constexpr int CG_BARS = 2 * CG_A_RING + 2 * CG_B_RING + 3;
constexpr int CG_COLS_OFF = CG_A_RING * CG_A_BYTES + CG_B_RING * CG_B_BYTES;             // constants of the epilogue warps' columns
constexpr int CG_BARS_OFF = CG_COLS_OFF + CG_EPI_WARPS * CG_EPI_COLS * 16;
constexpr int CG_SMEM = CG_BARS_OFF + CG_BARS * 8 + 16 + 1024;

template <int MODE>
__global__ void __launch_bounds__(CG_THREADS, 1) k_cal_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                            const __grid_constant__ CalLinearArgs p, int n_tiles, int tiles) {
  extern __shared__ uint8_t cg_raw[];
  const uint32_t raw = smem_u32(cg_raw), base = (raw + 1023u) & ~1023u;
  const uint32_t b_ring = base + CG_A_RING * CG_A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(cg_raw + (base - raw) + CG_BARS_OFF);
  const uint32_t a_full = smem_u32(bars), a_empty = a_full + 8u * CG_A_RING, b_full = a_empty + 8u * CG_A_RING;
  const uint32_t b_empty = b_full + 8u * CG_B_RING, acc_full = b_empty + 8u * CG_B_RING, acc_empty = acc_full + 8u, drained = acc_full + 16u;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + CG_BARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t a_used = 0, a_phase = 0, b_used = 0, b_phase = 0;     // TMA thread: filled slots and the parity of their last fill
  if (tid == 0) {
    for (int i = 0; i < CG_BARS; ++i) {
      const uint32_t bar = a_full + 8u * i;
      mbar_init(bar, bar == acc_empty ? (uint32_t)CG_EPI_WARPS : 1u);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_holder;
  const int K = p.K, n_chunks = (K + CAL_KCHUNK - 1) / CAL_KCHUNK;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int as = 0, bs = 0;
      uint32_t ap = 0, bp = 0;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int m0 = t / n_tiles * CG_BM, n0 = t % n_tiles * CG_BN;
        for (int k0 = 0; k0 < K && ok; k0 += CG_BK) {
          if ((b_used >> bs & 1u) && !mbar_wait(b_empty + 8u * bs, bp ^ 1u, abort_flag)) { ok = false; break; }
          b_used |= 1u << bs; b_phase = (b_phase & ~(1u << bs)) | bp << bs;
          mbar_arrive_expect_tx(b_full + 8u * bs, CG_B_BYTES);
          tma_load_2d(b_ring + (uint32_t)(bs * CG_B_BYTES), &tmB, k0, n0, b_full + 8u * bs);
          if (++bs == CG_B_RING) { bs = 0; bp ^= 1u; }
          for (int s = 0; s < CAL_SLICES; ++s) {
            if ((a_used >> as & 1u) && !mbar_wait(a_empty + 8u * as, ap ^ 1u, abort_flag)) { ok = false; break; }
            a_used |= 1u << as; a_phase = (a_phase & ~(1u << as)) | ap << as;
            mbar_arrive_expect_tx(a_full + 8u * as, CG_A_BYTES);
            tma_load_2d(base + (uint32_t)(as * CG_A_BYTES), &tmA, k0, (int)(s * p.M) + m0, a_full + 8u * as);
            if (++as == CG_A_RING) { as = 0; ap ^= 1u; }
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint64_t adesc0 = smem_desc_sw128(base), bdesc0 = smem_desc_sw128(b_ring);
      bool ok = true, first = true;
      int as = 0, bs = 0;
      uint32_t ap = 0, bp = 0, ep = 0;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        for (int kc = 0; kc < K && ok; kc += CAL_KCHUNK) {
          if (!first) { if (!mbar_wait(acc_empty, ep, abort_flag)) { ok = false; break; } ep ^= 1u; }
          first = false;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int k_end = min(K, kc + CAL_KCHUNK);
          for (int k0 = kc; k0 < k_end && ok; k0 += CG_BK) {
            if (!mbar_wait<true>(b_full + 8u * bs, bp, abort_flag)) { ok = false; break; }
            const int steps = min(CG_BK, k_end - k0) / 32;
            const uint64_t bdesc = bdesc0 + (uint64_t)(bs * (CG_B_BYTES >> 4));
            for (int s = 0; s < CAL_SLICES; ++s) {
              if (!mbar_wait<true>(a_full + 8u * as, ap, abort_flag)) { ok = false; break; }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              // s32 += (byte plane: u8, the top one s8) x s8
              const uint32_t idesc = (2u << 4) | ((s == CAL_SLICES - 1 ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(CG_BN >> 3) << 17) | ((uint32_t)(CG_BM >> 4) << 24);
              const uint64_t adesc = adesc0 + (uint64_t)(as * (CG_A_BYTES >> 4));
              for (int kk = 0; kk < steps; ++kk)
                mma_i8(tmem_base + (uint32_t)(s * CG_BN), adesc + (uint64_t)(2 * kk), bdesc + (uint64_t)(2 * kk), idesc, (uint32_t)(k0 > kc || kk > 0));
              mma_commit(a_empty + 8u * as);
              if (++as == CG_A_RING) { as = 0; ap ^= 1u; }
            }
            if (!ok) break;
            mma_commit(b_empty + 8u * bs);
            if (++bs == CG_B_RING) { bs = 0; bp ^= 1u; }
          }
          if (ok) mma_commit(acc_full);
        }
      }
    }
    __syncwarp();
  } else {
    // the warp's lane quarter (four consecutive warps cover the four) and CG_EPI_COLS columns
    const int q = warp & 3, col0 = (warp - 2) / 4 * CG_EPI_COLS;
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
    double2* cols = reinterpret_cast<double2*>(cg_raw + (base - raw) + CG_COLS_OFF) + (warp - 2) * CG_EPI_COLS;   // (step, bias)
    double part[CG_EPI_COLS];                                     // more than one chunk of k: the sums so far
    uint32_t fp = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const long m = (long)(t / n_tiles) * CG_BM + q * 32 + lane;
      const int n0 = t % n_tiles * CG_BN + col0;
      const bool row_ok = m < p.M;
      const int E = row_ok ? __ldg(p.expo + m) : 1;
      long src = -1, dst = m;
      if (MODE == CAL_PROJ || MODE == CAL_FC2) src = row_ok ? (long)__ldg(p.rowsrc + m) : -1;
      if (MODE == CAL_FC2) dst = src;
      const long rr = MODE == CAL_PROJ ? src : m;                 // row of the residual, < 0: zero
      const bool store = row_ok && (MODE != CAL_FC2 || src >= 0);
      const double unit = __longlong_as_double((long long)(E - 181 + 1023) << 52);      // value of the lowest bit of the row
      __syncwarp();
      if (lane < CG_EPI_COLS) {
        const int n = n0 + lane < p.N ? n0 + lane : 0;
        cols[lane] = make_double2((double)__ldg(p.sw + n), p.bias ? (double)__ldg(p.bias + n) : 0.0);
      }
      __syncwarp();
      float lo = INFINITY, hi = -INFINITY;
      for (int c = 0; c < n_chunks; ++c) {
        if (!mbar_wait_warp(acc_full, fp, abort_flag)) { ok = false; break; }
        fp ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
        for (int g = 0; g < CG_EPI_COLS; g += 8) {
          int32_t S[CAL_SLICES][8];
          __syncwarp();                                           // rows that are not stored left the pass before early
#pragma unroll
          for (int s = 0; s < CAL_SLICES; ++s) tmem_ld(taddr + (uint32_t)(s * CG_BN + g), S[s]);
#pragma unroll
          for (int s = 0; s < CAL_SLICES; ++s) tmem_ld_wait(S[s]);
          if (g + 8 == CG_EPI_COLS) {                             // the accumulators are read: the next tile may start
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty);
          }
          float v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            // whole numbers below 2^51 become binary64 through the bit pattern of 1.5 * 2^52
            constexpr long long kMagic64 = 0x4338000000000000LL;
            const double h = __dadd_rn(__longlong_as_double((long long)S[6][j] * 65536 + ((long long)S[5][j] * 256 + (S[4][j] + kMagic64))), -6755399441055744.0);
            const double mid = __dadd_rn(__longlong_as_double((long long)S[3][j] * 256 + (S[2][j] + kMagic64)), -6755399441055744.0);
            const double l = __dadd_rn(__longlong_as_double((long long)S[1][j] * 256 + (S[0][j] + kMagic64)), -6755399441055744.0);
            double d = __fma_rn(h, 4294967296.0, __fma_rn(mid, 65536.0, l));
            if (n_chunks > 1) {
              if (c > 0) d = __dadd_rn(d, part[g + j]);
              part[g + j] = d;
            }
            const double2 cb = cols[g + j];
            v[j] = (float)__dadd_rn(__dmul_rn(__dmul_rn(d, unit), cb.x), cb.y);
          }
          if (c + 1 < n_chunks) continue;
          const int n = n0 + g;
          if (E == CAL_PLAIN_ROW && store) {                      // k_cal_split has put this row's sums where the results go
#pragma unroll
            for (int j = 0; j < 8; ++j) if (n + j < p.N) v[j] = p.out[dst * p.N + n + j];
          }
          if (MODE == CAL_FC1) {
#pragma unroll
            for (int j = 0; j < 8; j += 2) { const float2 a = gelu_f2(make_float2(v[j], v[j + 1])); v[j] = a.x; v[j + 1] = a.y; }
          }
          if ((MODE == CAL_QKV || MODE == CAL_FC1) && row_ok && n < p.N) {
#pragma unroll
            for (int j = 0; j < 8; ++j) { lo = fminf(lo, v[j]); hi = fmaxf(hi, v[j]); }
          }
          if (!store || n >= p.N) continue;
          float* out = p.out + dst * p.N + n;
          if (MODE == CAL_PLAIN && p.N % 8) {                     // only a merge may have a ragged width
#pragma unroll
            for (int j = 0; j < 8; ++j) if (n + j < p.N) out[j] = v[j];
            continue;
          }
          if ((MODE == CAL_PROJ || MODE == CAL_FC2) && rr >= 0) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(p.res + rr * p.N + n)), b = __ldg(reinterpret_cast<const float4*>(p.res + rr * p.N + n) + 1);
            v[0] = __fadd_rn(a.x, v[0]); v[1] = __fadd_rn(a.y, v[1]); v[2] = __fadd_rn(a.z, v[2]); v[3] = __fadd_rn(a.w, v[3]);
            v[4] = __fadd_rn(b.x, v[4]); v[5] = __fadd_rn(b.y, v[5]); v[6] = __fadd_rn(b.z, v[6]); v[7] = __fadd_rn(b.w, v[7]);
          } else if (MODE == CAL_PROJ || MODE == CAL_FC2) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __fadd_rn(0.0f, v[j]);
          }
          reinterpret_cast<float4*>(out)[0] = make_float4(v[0], v[1], v[2], v[3]);
          reinterpret_cast<float4*>(out)[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
      }
      if (!ok) break;
      // a warp's columns lie in one q/k/v section (sections are multiples of 32 channels)
      if (MODE == CAL_QKV) { if (n0 < p.N) observe_warp(p.obs, 1 + n0 / p.C, lo, hi); }
      else if (MODE == CAL_FC1) { if (n0 < p.N) observe_warp(p.obs, 6, lo, hi); }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag) {
    // a wait ran out: the copies and MMAs already issued have to end (bounded) before the CTA may exit
    if (tid == 32) mma_commit(drained);
    if (tid == 0) {
      atomicExch(p.status, 1);
      p.obs[CAL_STATUS] = 1;
      auto drain = [](uint32_t bar, uint32_t parity) {
        for (uint32_t it = 0; it < (1u << 20); ++it) if (mbar_try_wait(bar, parity)) return;
      };
      for (int s = 0; s < CG_A_RING; ++s) if (a_used >> s & 1u) drain(a_full + 8u * s, a_phase >> s & 1u);
      for (int s = 0; s < CG_B_RING; ++s) if (b_used >> s & 1u) drain(b_full + 8u * s, b_phase >> s & 1u);
      drain(drained, 0u);
    }
    __syncthreads();
  }
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

// softmax of the numeric contract over 49 logits: exact maximum, exponentials through 2^t, four interleaved partial
// sums (column j of the 8-wide group j/8 goes to partial (j mod 8)/2, in increasing j), (p0+p1)+(p2+p3), one division
__device__ __forceinline__ void softmax49(float (&s)[WT]) {
  float mx = s[0];
#pragma unroll
  for (int j = 1; j < WT; ++j) mx = fmaxf(mx, s[j]);
#pragma unroll
  for (int j = 0; j < WT; ++j) {
    const float t = fmaxf(__fmul_rn(__fsub_rn(s[j], mx), 1.44269504088896340736f), -125.0f);
    s[j] = exp2_core2(make_float2(t, t)).x;
  }
  float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int grp = 0; grp * 8 < WT; ++grp)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int j = grp * 8 + 2 * t + u;
        if (j < WT) part[t] = __fadd_rn(part[t], s[j]);
      }
  const float inv = __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(part[0], part[1]), __fadd_rn(part[2], part[3])));
#pragma unroll
  for (int j = 0; j < WT; ++j) s[j] = __fmul_rn(s[j], inv);
}

// One CTA of 64 threads per (window slot, head): q, k, v staged in shared memory as binary64, logits as 7 x 7 register
// tiles (thread (i/7, j/7)), one thread per row for the softmax of the contract, P.V as 7 rows x 4 channels per thread.
// The products of binary32 values are exact in binary64 (48 bits), so a fused multiply-add rounds like multiply-then-add;
// the sums run in index order.  Bound by the binary64 pipe and the conversions of the operands (once per CTA).
struct CalAttnArgs {
  const float* qkv; const float* relpos; float* o;
  long slots; int C, heads, shift, Hp, Wp, nwx, nW;
  uint32_t* obs;
};
struct CalAttnSmem {
  double q[HEAD_DIM][WT + 1], k[HEAD_DIM][WT + 1];   // [channel][token]
  double v[WT][HEAD_DIM + 2];
  float s[WT][WT];
  uint8_t region[WT + 7];
};
__global__ void __launch_bounds__(64) k_cal_attention(CalAttnArgs a) {
  extern __shared__ __align__(16) uint8_t cal_smem[];
  CalAttnSmem& sm = *reinterpret_cast<CalAttnSmem*>(cal_smem);
  double (*pd)[WT + 1] = reinterpret_cast<double (*)[WT + 1]>(&sm.q[0][0]);   // P in binary64 over the dead q and k
  static_assert(sizeof(double) * WT * (WT + 1) <= 2 * sizeof(double) * HEAD_DIM * (WT + 1), "P does not fit over q and k");
  const int tid = threadIdx.x;
  const long slot = (long)blockIdx.x / a.heads;
  const int h = (int)((long)blockIdx.x - slot * a.heads), C = a.C;
  const float* base = a.qkv + slot * WT * 3 * C + h * HEAD_DIM;
  const int w = (int)(slot % a.nW), wy = w / a.nwx, wx = w - wy * a.nwx;
  auto region = [&](int pos, int L) { return pos < L - WS ? 0 : (pos < L - a.shift ? 1 : 2); };
  for (int item = tid; item < WT * HEAD_DIM; item += 64) {
    const int r = item >> 5, e = item & 31;
    const float* row = base + (long)r * 3 * C + e;
    sm.q[e][r] = (double)__ldg(row); sm.k[e][r] = (double)__ldg(row + C); sm.v[r][e] = (double)__ldg(row + 2 * C);
  }
  if (tid < WT) sm.region[tid] = (uint8_t)(region(wy * WS + tid / WS, a.Hp) * 3 + region(wx * WS + tid % WS, a.Wp));
  __syncthreads();
  if (tid < 49) {
    const int i0 = (tid / 7) * 7, j0 = (tid % 7) * 7;
    double d[7][7];
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
      for (int j = 0; j < 7; ++j) d[i][j] = 0.0;
    for (int e = 0; e < HEAD_DIM; ++e) {
      double qv[7], kv[7];
#pragma unroll
      for (int i = 0; i < 7; ++i) { qv[i] = sm.q[e][i0 + i]; kv[i] = sm.k[e][j0 + i]; }
#pragma unroll
      for (int i = 0; i < 7; ++i)
#pragma unroll
        for (int j = 0; j < 7; ++j) d[i][j] = __fma_rn(qv[i], kv[j], d[i][j]);
    }
    const double rs = 1.0 / sqrt((double)HEAD_DIM);
    // row i0 + i is token (tid / 7, i) of the window, column j0 + j token (tid % 7, j)
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        const int ridx = (tid / 7 - tid % 7 + WS - 1) * (2 * WS - 1) + (i - j + WS - 1);
        const double maskv = a.shift > 0 && sm.region[i0 + i] != sm.region[j0 + j] ? -100.0 : 0.0;
        sm.s[i0 + i][j0 + j] = (float)__dadd_rn(__dadd_rn(__dmul_rn(d[i][j], rs), (double)__ldg(a.relpos + (long)ridx * a.heads + h)), maskv);
      }
  }
  __syncthreads();
  if (tid < WT) {
    float s[WT];
#pragma unroll
    for (int j = 0; j < WT; ++j) s[j] = sm.s[tid][j];
    softmax49(s);
#pragma unroll
    for (int j = 0; j < WT; ++j) pd[tid][j] = (double)s[j];
  }
  __syncthreads();
  float lo = INFINITY, hi = -INFINITY;
  if (tid < 56) {
    const int i0 = (tid >> 3) * 7, e0 = (tid & 7) * 4;
    double o[7][4];
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[i][e] = 0.0;
    for (int j = 0; j < WT; ++j) {
      double vv[4];
#pragma unroll
      for (int e = 0; e < 4; e += 2) *reinterpret_cast<double2*>(&vv[e]) = *reinterpret_cast<const double2*>(&sm.v[j][e0 + e]);
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        const double pv = pd[i0 + i][j];
#pragma unroll
        for (int e = 0; e < 4; ++e) o[i][e] = __fma_rn(pv, vv[e], o[i][e]);
      }
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      const float4 f = make_float4((float)o[i][0], (float)o[i][1], (float)o[i][2], (float)o[i][3]);
      *reinterpret_cast<float4*>(a.o + (slot * WT + i0 + i) * C + h * HEAD_DIM + e0) = f;
      lo = fminf(fminf(lo, fminf(f.x, f.y)), fminf(f.z, f.w));
      hi = fmaxf(fmaxf(hi, fmaxf(f.x, f.y)), fmaxf(f.z, f.w));
    }
  }
  observe_warp(a.obs, 4, lo, hi);
}

__global__ void k_cal_obs_init(uint32_t* obs, int sites) {
  const int i = threadIdx.x;
  if (i < 2 * sites) obs[i] = (i & 1) ? 0u : 0xFFFFFFFFu;
  if (i == CAL_STATUS) obs[i] = 0u;
}

template <int MODE>
bool launch_cal_linear(const CalLinearArgs& p, cudaStream_t st) {
  if (p.M == 0) return true;
  if (cudaFuncSetAttribute(k_cal_gemm<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, CG_SMEM) != cudaSuccess) return false;
  CUtensorMap mA, mB;
  if (!make_map(&mA, p.slices, (uint64_t)CAL_SLICES * p.M, (uint64_t)p.K, CG_BM) || !make_map(&mB, p.w, (uint64_t)p.N, (uint64_t)p.K, CG_BN)) return false;
  k_cal_split<<<(unsigned)((p.M + CAL_SPLIT_WARPS - 1) / CAL_SPLIT_WARPS), 32 * CAL_SPLIT_WARPS, 0, st>>>(p, MODE == CAL_FC2);
  const int n_tiles = (p.N + CG_BN - 1) / CG_BN;
  const int tiles = (int)((p.M + CG_BM - 1) / CG_BM) * n_tiles, sms = sm_count();
  k_cal_gemm<MODE><<<tiles < sms ? tiles : sms, CG_THREADS, CG_SMEM, st>>>(mA, mB, p, n_tiles, tiles);
  g_launches += 2;
  return true;
}

}  // namespace

// keys written by the observers -> floats (host side)
float cal_key_to_float(uint32_t key) {
  const uint32_t u = (key & 0x80000000u) ? (key & 0x7FFFFFFFu) : ~key;
  float f;
  memcpy(&f, &u, 4);
  return f;
}

#define MIXAQ_CAL_LN_CASE(n) case n: k_cal_ln<n><<<grid, 256, 0, st>>>(src, rowsrc_out, gamma, beta, out, M, gather, H, W, shift, nwx, nW, obs, site, site_in); break;
static bool launch_cal_ln(const float* src, int32_t* rowsrc_out, const float* gamma, const float* beta, float* out, long M,
                          int C, int gather, int H, int W, int shift, int nwx, int nW, uint32_t* obs, int site, int site_in, cudaStream_t st) {
  const unsigned grid = (unsigned)((M + 7) / 8);
  switch (C / 32) {
    MIXAQ_CAL_LN_CASE(1) MIXAQ_CAL_LN_CASE(2) MIXAQ_CAL_LN_CASE(3) MIXAQ_CAL_LN_CASE(4) MIXAQ_CAL_LN_CASE(6) MIXAQ_CAL_LN_CASE(8)
    MIXAQ_CAL_LN_CASE(12) MIXAQ_CAL_LN_CASE(16) MIXAQ_CAL_LN_CASE(24) MIXAQ_CAL_LN_CASE(32)
    default: return false;
  }
  ++g_launches;
  return true;
}

// The floating-point block through one branch.  Workspace (floats unless noted): rowsrc int32[M], ln [M][C],
// qkv [M][3C], o [M][C], x1 [M][C], h [M][hidden], slices, expo; obs: keys of the seven sites and the block's input map, status.
bool launch_calibrate_block(const CalBlockArgs& c, cudaStream_t st) {
  const int C = c.C, Hd = c.hidden;
  const int Hp = (c.H + WS - 1) / WS * WS, Wp = (c.W + WS - 1) / WS * WS, nwx = Wp / WS, nW = (Hp / WS) * nwx;
  const long slots = (long)c.B * nW, M = slots * WT;
  k_cal_obs_init<<<1, 32, 0, st>>>(c.obs, 8);
  ++g_launches;
  if (!launch_cal_ln(c.x, c.rowsrc, c.ln1_g, c.ln1_b, c.ln, M, C, 1, c.H, c.W, c.shift, nwx, nW, c.obs, 0, 7, st)) return false;
  CalLinearArgs l;
  l.obs = c.obs; l.status = c.status; l.slices = c.slices; l.expo = c.expo; l.M = M; l.C = C; l.rowsrc = c.rowsrc;
  l.a = c.ln; l.w = c.w_qkv; l.sw = c.s_qkv; l.bias = c.b_qkv; l.out = c.qkv; l.res = nullptr; l.N = 3 * C; l.K = C;
  if (!launch_cal_linear<CAL_QKV>(l, st)) return false;
  CalAttnArgs a;
  a.qkv = c.qkv; a.relpos = c.relpos; a.o = c.o; a.slots = slots; a.C = C; a.heads = c.heads; a.shift = c.shift;
  a.Hp = Hp; a.Wp = Wp; a.nwx = nwx; a.nW = nW; a.obs = c.obs;
  if (cudaFuncSetAttribute(k_cal_attention, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CalAttnSmem)) != cudaSuccess) return false;
  k_cal_attention<<<(unsigned)(slots * c.heads), 64, sizeof(CalAttnSmem), st>>>(a);
  ++g_launches;
  l.a = c.o; l.w = c.w_proj; l.sw = c.s_proj; l.bias = c.b_proj; l.out = c.x1; l.res = c.x; l.N = C; l.K = C;
  if (!launch_cal_linear<CAL_PROJ>(l, st)) return false;
  if (!launch_cal_ln(c.x1, nullptr, c.ln2_g, c.ln2_b, c.ln, M, C, 0, c.H, c.W, c.shift, nwx, nW, c.obs, 5, -1, st)) return false;
  l.a = c.ln; l.w = c.w_fc1; l.sw = c.s_fc1; l.bias = c.b_fc1; l.out = c.h; l.res = nullptr; l.N = Hd; l.K = C;
  if (!launch_cal_linear<CAL_FC1>(l, st)) return false;
  l.a = c.h; l.w = c.w_fc2; l.sw = c.s_fc2; l.bias = c.b_fc2; l.out = c.y; l.res = c.x1; l.N = C; l.K = Hd; l.slices = c.slices_fc2;
  if (!launch_cal_linear<CAL_FC2>(l, st)) return false;
  return true;
}

#define MIXAQ_CAL_MERGE_CASE(n) case n: k_cal_merge_ln<n><<<grid, 256, 0, st>>>(c.x, c.ln_g, c.ln_b, c.ln, c.B, c.H, c.W, c.obs); break;
bool launch_calibrate_merge(const CalMergeArgs& c, cudaStream_t st) {
  const long M = (long)c.B * ((c.H + 1) / 2) * ((c.W + 1) / 2);
  k_cal_obs_init<<<1, 32, 0, st>>>(c.obs, 1);
  ++g_launches;
  const unsigned grid = (unsigned)((M + 7) / 8);
  switch (4 * c.C / 32) {
    MIXAQ_CAL_MERGE_CASE(4) MIXAQ_CAL_MERGE_CASE(8) MIXAQ_CAL_MERGE_CASE(12) MIXAQ_CAL_MERGE_CASE(16) MIXAQ_CAL_MERGE_CASE(24)
    MIXAQ_CAL_MERGE_CASE(32) MIXAQ_CAL_MERGE_CASE(48) MIXAQ_CAL_MERGE_CASE(64)
    default: return false;
  }
  ++g_launches;
  CalLinearArgs l;
  l.obs = c.obs; l.status = c.status; l.slices = c.slices; l.expo = c.expo; l.M = M; l.C = c.N; l.rowsrc = nullptr; l.res = nullptr;
  l.a = c.ln; l.w = c.w; l.sw = c.sw; l.bias = nullptr; l.out = c.y; l.N = c.N; l.K = 4 * c.C;
  if (!launch_cal_linear<CAL_PLAIN>(l, st)) return false;
  return true;
}

}  // namespace mixaq
