// Calibration of the activation quantizers (MixA-Q Section 4.3, post-training flow: one calibration sample, and the
// FULL feature map -- every window, not the windows a branch will later see -- initialises the step sizes of both
// branches).  The kernels below run the floating-point Two-Branch block (all quantizers off, weights = code x step)
// through ONE branch's LayerNorm parameters and biases and record the minimum and maximum of what each of the seven
// quantizer sites would see.  Arithmetic: LayerNorm, softmax and GELU exactly as in the quantized path (the same
// device functions); matrix products accumulated in binary64 in index order (register-tiled SIMT kernels).
#include "kernels.h"

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

// out[m][n] = (float)( sum_k a[m][k] * (w[n][k] * sw[n])  [binary64, k ascending]  + bias[n] ), then per mode:
enum CalMode { CAL_QKV = 0, CAL_PROJ = 1, CAL_FC1 = 2, CAL_FC2 = 3, CAL_PLAIN = 4 };
struct CalLinearArgs {
  const float* a; const int8_t* w; const float* sw; const float* bias;   // bias nullable
  float* out;                 // QKV, FC1, PLAIN: [M][N];  PROJ: x1 [M][N];  FC2: the output feature map
  const float* res;           // PROJ: input feature map (gathered through rowsrc);  FC2: x1 [M][N]
  const int32_t* rowsrc;      // PROJ, FC2
  long M; int N, K, C;        // C: width of one q/k/v section (QKV)
  uint32_t* obs;
};
// Register-tiled binary64 product: a CTA of 64 threads owns a 128 x 32 output tile (every width here is a multiple of 32),
// a thread 8 rows x 8 columns, so one value read from shared memory feeds 8 products and an input is converted to
// binary64 once per tile instead of once per product.  Each sum still runs over k in ascending order, so the results are
// those of the plain loop.
// FUSED: the product a * (code * step) needs at most 24 + 24 + (significant bits of the code) bits; up to 5 bits of code
// (weights of 6 bits or fewer) it is exact in binary64, and a fused multiply-add rounds exactly like the product
// followed by the addition.  Wider weights keep the two separate roundings.
// Bound by the binary64 pipe (64 lanes per SM and clock) and by shared-memory reads: with 8 x 4 values per thread the
// 16-byte reads took as long as the products.  Figures: see launch_calibrate_block.
constexpr int CTM = 128, CTN = 32, CTK = 16, CTPAD = 2;   // tile, k-step, padding (doubles) of a shared row
template <int MODE, bool FUSED>
__global__ void __launch_bounds__(64, 4) k_cal_linear(CalLinearArgs p) {
  __shared__ __align__(16) double sa[2][CTK][CTM + CTPAD], sb[2][CTK][CTN + CTPAD];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = (lane & 7) + 8 * warp, tx = lane >> 3;  // rows 2 ty + {0, 1} + 32 i, columns 2 tx + {0, 1} + 8 j
  const int n_tiles = (p.N + CTN - 1) / CTN;
  const long m0 = (long)(blockIdx.x / n_tiles) * CTM;
  const int n0 = (int)(blockIdx.x % n_tiles) * CTN;
  // staging: four lanes fetch the 16 k of one row (64-byte runs; one lane per row made the L1 lookups the bound), one
  // half of the rows of a per half step; lane n of the first warp fetches the 16 weight codes of row n
  const int sr = tid >> 2, sk = 4 * (tid & 3);
  const bool b_ok = warp == 0 && n0 + lane < p.N;
  const int8_t* wr = p.w + (long)(b_ok ? n0 + lane : 0) * p.K;
  const double sw = b_ok ? (double)__ldg(p.sw + n0 + lane) : 0.0;
  float4 av[4];
  int4 wv = make_int4(0, 0, 0, 0);
  auto fetch_a = [&](int k0, int half) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const long m = m0 + sr + 16 * r + 64 * half;
      av[r] = __ldg(reinterpret_cast<const float4*>(p.a + (m < p.M ? m : 0) * p.K + k0 + sk));
    }
  };
  auto store_a = [&](int buf, int half) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = sr + 16 * r + 64 * half;
      sa[buf][sk][row] = (double)av[r].x; sa[buf][sk + 1][row] = (double)av[r].y;
      sa[buf][sk + 2][row] = (double)av[r].z; sa[buf][sk + 3][row] = (double)av[r].w;
    }
  };
  auto store_b = [&](int buf) {
    if (warp == 0) {
      const int w4[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
      for (int j = 0; j < CTK; ++j)
        sb[buf][j][lane] = __dmul_rn((double)(int)(int8_t)(w4[j >> 2] >> (8 * (j & 3))), sw);   // exact
    }
  };
  double acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  if (b_ok) wv = __ldg(reinterpret_cast<const int4*>(wr));
  fetch_a(0, 0); store_a(0, 0);
  fetch_a(0, 1); store_a(0, 1);
  store_b(0);
  __syncthreads();
  for (int k0 = 0, buf = 0; k0 < p.K; k0 += CTK, buf ^= 1) {            // K is a multiple of 32
    const bool more = k0 + CTK < p.K;
    if (more && b_ok) wv = __ldg(reinterpret_cast<const int4*>(wr + k0 + CTK));
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (more) fetch_a(k0 + CTK, half);
#pragma unroll
      for (int k = half * (CTK / 2); k < (half + 1) * (CTK / 2); ++k) {
        double a[8], b[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double2 t = *reinterpret_cast<const double2*>(&sa[buf][k][2 * ty + 32 * i]);
          const double2 u = *reinterpret_cast<const double2*>(&sb[buf][k][2 * tx + 8 * i]);
          a[2 * i] = t.x; a[2 * i + 1] = t.y; b[2 * i] = u.x; b[2 * i + 1] = u.y;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            acc[i][j] = FUSED ? __fma_rn(a[i], b[j], acc[i][j]) : __dadd_rn(acc[i][j], __dmul_rn(a[i], b[j]));
      }
      if (more) store_a(buf ^ 1, half);
    }
    if (more) store_b(buf ^ 1);
    __syncthreads();
  }
  // the tile's 32 columns lie in one q/k/v section (sections are multiples of 32 channels)
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long m = m0 + 2 * ty + (i & 1) + 32 * (i >> 1);
    if (m >= p.M) continue;
    long dst = m, src = -1;
    if (MODE == CAL_PROJ || MODE == CAL_FC2) src = p.rowsrc[m];
    if (MODE == CAL_FC2) { if (src < 0) continue; dst = src; }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 2 * tx + 8 * j;
      if (n >= p.N) continue;                                  // only a merge may have a ragged width
      const bool pair = n + 1 < p.N;
      float2 v = make_float2((float)__dadd_rn(acc[i][2 * j], p.bias ? (double)__ldg(p.bias + n) : 0.0),
                             (float)__dadd_rn(acc[i][2 * j + 1], p.bias && pair ? (double)__ldg(p.bias + n + 1) : 0.0));
      if (MODE == CAL_FC1) v = gelu_f2(v);
      if (MODE == CAL_QKV || MODE == CAL_FC1) { lo = fminf(lo, fminf(v.x, v.y)); hi = fmaxf(hi, fmaxf(v.x, v.y)); }
      if (MODE == CAL_PROJ || MODE == CAL_FC2) {
        float2 r = make_float2(0.f, 0.f);
        const long rr = MODE == CAL_PROJ ? src : m;
        if (rr >= 0) r = __ldg(reinterpret_cast<const float2*>(p.res + rr * p.N + n));
        v = make_float2(__fadd_rn(r.x, v.x), __fadd_rn(r.y, v.y));
      }
      float* out = p.out + dst * p.N + n;
      if (MODE == CAL_PLAIN && p.N % 2) { out[0] = v.x; if (pair) out[1] = v.y; }
      else *reinterpret_cast<float2*>(out) = v;
    }
  }
  if (MODE == CAL_QKV) observe_warp(p.obs, 1 + n0 / p.C, lo, hi);
  else if (MODE == CAL_FC1) observe_warp(p.obs, 6, lo, hi);
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
}

// w_bits: declared width of the weight codes; up to 6 bits (5 significant) the fused product is exact, see k_cal_linear
template <int MODE>
void launch_cal_linear(const CalLinearArgs& p, int w_bits, cudaStream_t st) {
  if (p.M == 0) return;
  const unsigned grid = (unsigned)(((p.N + CTN - 1) / CTN) * ((p.M + CTM - 1) / CTM));
  if (w_bits >= 2 && w_bits <= 6) k_cal_linear<MODE, true><<<grid, 64, 0, st>>>(p);
  else k_cal_linear<MODE, false><<<grid, 64, 0, st>>>(p);
  ++g_launches;
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

// Calibration of a Swin-T backbone on a 200 x 334 map (W4, both branches of 12 blocks, 205 G products): 125 ms with one
// thread per output, 31 ms with the register tiles (27 ms of kernels: 24 ms of products at 8.5 T/s, about half of the
// binary64 pipe's rate).  The output map, the observed ranges and the quantizers are unchanged bit for bit.
// The floating-point block through one branch.  Workspace (floats unless noted): rowsrc int32[M], ln [M][C],
// qkv [M][3C], o [M][C], x1 [M][C], h [M][hidden]; obs: 16 keys (seven sites and the block's input map).
bool launch_calibrate_block(const CalBlockArgs& c, cudaStream_t st) {
  const int C = c.C, Hd = c.hidden;
  const int Hp = (c.H + WS - 1) / WS * WS, Wp = (c.W + WS - 1) / WS * WS, nwx = Wp / WS, nW = (Hp / WS) * nwx;
  const long slots = (long)c.B * nW, M = slots * WT;
  k_cal_obs_init<<<1, 32, 0, st>>>(c.obs, 8);
  ++g_launches;
  if (!launch_cal_ln(c.x, c.rowsrc, c.ln1_g, c.ln1_b, c.ln, M, C, 1, c.H, c.W, c.shift, nwx, nW, c.obs, 0, 7, st)) return false;
  CalLinearArgs l;
  l.obs = c.obs; l.M = M; l.C = C; l.rowsrc = c.rowsrc;
  l.a = c.ln; l.w = c.w_qkv; l.sw = c.s_qkv; l.bias = c.b_qkv; l.out = c.qkv; l.res = nullptr; l.N = 3 * C; l.K = C;
  launch_cal_linear<CAL_QKV>(l, c.wb_qkv, st);
  CalAttnArgs a;
  a.qkv = c.qkv; a.relpos = c.relpos; a.o = c.o; a.slots = slots; a.C = C; a.heads = c.heads; a.shift = c.shift;
  a.Hp = Hp; a.Wp = Wp; a.nwx = nwx; a.nW = nW; a.obs = c.obs;
  if (cudaFuncSetAttribute(k_cal_attention, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CalAttnSmem)) != cudaSuccess) return false;
  k_cal_attention<<<(unsigned)(slots * c.heads), 64, sizeof(CalAttnSmem), st>>>(a);
  ++g_launches;
  l.a = c.o; l.w = c.w_proj; l.sw = c.s_proj; l.bias = c.b_proj; l.out = c.x1; l.res = c.x; l.N = C; l.K = C;
  launch_cal_linear<CAL_PROJ>(l, c.wb_proj, st);
  if (!launch_cal_ln(c.x1, nullptr, c.ln2_g, c.ln2_b, c.ln, M, C, 0, c.H, c.W, c.shift, nwx, nW, c.obs, 5, -1, st)) return false;
  l.a = c.ln; l.w = c.w_fc1; l.sw = c.s_fc1; l.bias = c.b_fc1; l.out = c.h; l.res = nullptr; l.N = Hd; l.K = C;
  launch_cal_linear<CAL_FC1>(l, c.wb_fc1, st);
  l.a = c.h; l.w = c.w_fc2; l.sw = c.s_fc2; l.bias = c.b_fc2; l.out = c.y; l.res = c.x1; l.N = C; l.K = Hd;
  launch_cal_linear<CAL_FC2>(l, c.wb_fc2, st);
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
  l.obs = c.obs; l.M = M; l.C = c.N; l.rowsrc = nullptr; l.res = nullptr;
  l.a = c.ln; l.w = c.w; l.sw = c.sw; l.bias = nullptr; l.out = c.y; l.N = c.N; l.K = 4 * c.C;
  launch_cal_linear<CAL_PLAIN>(l, c.w_bits, st);
  return true;
}

}  // namespace mixaq
