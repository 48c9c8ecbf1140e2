// Window importance scoring and ratio-driven selection (MixA-Q Section 3.2; pruned class: Section 3.4).
// Integer work throughout: int8 score codes, int32 token energies, int64 window scores, ranks by counting.
#include "kernels.h"
#include <climits>

namespace mixaq {

// energy[token] = sum_c clamp(rne(x*inv), -127, 127)^2.  Integer sums are exact in any order, so the loads are
// laid out for the memory system only: a group of G = 8 lanes owns one token and walks its channels with
// 16-byte loads (C is a multiple of 32), four tokens per warp.
__device__ __forceinline__ int score_code_sq(float v, float inv) {
  // clamp before rounding (the bounds are integers), then round to nearest-even by the 1.5*2^23 addition
  float t = fminf(fmaxf(__fmul_rn(v, inv), -127.0f), 127.0f);
  int code = (int)(__float_as_uint(__fadd_rn(t, 12582912.0f)) - kMagicBits);
  return code * code;
}
__global__ void __launch_bounds__(256) k_energy(const float* __restrict__ x, int32_t* __restrict__ energy,
                                                long ntok, int C, float inv) {
  griddep_wait();
  griddep_launch();
  const long tok = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const int sub = threadIdx.x & 7;
  int e = 0;
  if (tok < ntok) {
    const float4* row = reinterpret_cast<const float4*>(x + tok * C);
    for (int c0 = sub; c0 < C / 4; c0 += 32) {          // four loads in flight per lane
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = c0 + 8 * u < C / 4 ? __ldg(row + c0 + 8 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        e += score_code_sq(v[u].x, inv) + score_code_sq(v[u].y, inv) + score_code_sq(v[u].z, inv) + score_code_sq(v[u].w, inv);
    }
  }
#pragma unroll
  for (int off = 4; off >= 1; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
  if (sub == 0 && tok < ntok) energy[tok] = e;
}

__device__ __forceinline__ int window_src(int b, int H, int W, int Hp, int Wp, int shift, int nwx, int w, int t) {
  int wy = w / nwx, wx = w - wy * nwx;
  int i = t / WS, j = t - i * WS;
  int y = wy * WS + i + shift; if (y >= Hp) y -= Hp;
  int x = wx * WS + j + shift; if (x >= Wp) x -= Wp;
  if (y >= H || x >= W) return -1;
  return (b * H + y) * W + x;
}

// One warp per (image, window): score = sum of the energies of the window's real tokens under this
// block's own (possibly shifted, cyclically wrapped) partition.
constexpr int MAX_SELECT_BATCH = 24;
struct SelectBatch { SelectArgs a[MAX_SELECT_BATCH]; };

__global__ void __launch_bounds__(256) k_window_score(const __grid_constant__ SelectBatch batch) {
  griddep_wait();
  griddep_launch();
  const SelectArgs& a = batch.a[blockIdx.y];
  int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (gw >= a.B * a.nW) return;
  int b = gw / a.nW, w = gw - b * a.nW;
  int Hp = (a.H + WS - 1) / WS * WS, Wp = (a.W + WS - 1) / WS * WS;
  long long s = 0;
  for (int t = lane; t < WT; t += 32) {
    int src = window_src(b, a.H, a.W, Hp, Wp, a.shift, a.nwx, w, t);
    if (src >= 0) s += a.energy[src];
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) a.score[gw] = s;
}

// How many windows of an image precede window w in (score descending, index ascending), by one warp.  key: the scores in shared
// memory (negated for the ascending order), n4 groups of four, padded with the lowest value.  Windows before w precede it with an
// equal score too; a lane compares four per load.
template <class Key>
__device__ __forceinline__ int count_preceding(const Key* key, int n4, int w, int lane) {
  struct alignas(4 * sizeof(Key)) Four { Key k[4]; };
  const Four* four = reinterpret_cast<const Four*>(key);
  const Key mine = key[w];
  int cnt = 0;
  for (int i = lane; i < n4; i += 32) {
    const Four o = four[i];
    // (the group that holds w: those from w on have to exceed it)
    const Key at_least = 4 * i + 3 < w ? mine : mine + 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) cnt += o.k[j] >= at_least ? 1 : 0;
    if (i == w >> 2)
      for (int j = 0; j < 4; ++j) cnt += 4 * i + j < w && o.k[j] == mine ? 1 : 0;
  }
  return __reduce_add_sync(0xffffffffu, cnt);
}

// The bookkeeping of the slot that window w takes with its rank (by one warp)
__device__ __forceinline__ void emit_window(const SelectArgs& a, int b, int w, int rank, int lane, int Hp, int Wp) {
  const int c = rank < a.n_hi ? 0 : (rank < a.n_hi + a.n_lo ? 1 : 2);
  int32_t* dst; long slot;
  if (c == 0)      { slot = (long)b * a.n_hi + rank;                     dst = a.rowsrc_hi; }
  else if (c == 1) { slot = (long)b * a.n_lo + (rank - a.n_hi);          dst = a.rowsrc_lo; }
  else             { slot = (long)b * a.n_pr + (rank - a.n_hi - a.n_lo); dst = a.rowsrc_pr; }
  if (lane == 0) {
    a.order[(long)b * a.nW + rank] = w;
    a.cls[(long)b * a.nW + w] = (uint8_t)c;
    if (c == 0) a.win_hi[slot] = w;
    else if (c == 1) a.win_lo[slot] = w;
  }
  for (int t = lane; t < WT; t += 32) dst[slot * WT + t] = window_src(b, a.H, a.W, Hp, Wp, a.shift, a.nwx, w, t);
}

// Rank by counting: ranks are a permutation.  One warp per window: the lanes split the windows to compare against, and then
// write the batch bookkeeping of the window's slot (49 source-token indices) together.  Bound by the comparisons (n^2 per image),
// so scores that fit are compared as 32-bit numbers: every score made of the library's own energies does (at most
// 49 x 1024 x 127^2); a caller's energies may not.
constexpr int RANK_WARPS = 8;
__global__ void __launch_bounds__(RANK_WARPS * 32) k_rank_emit(const __grid_constant__ SelectBatch batch) {
  griddep_launch();
  griddep_wait();
  extern __shared__ __align__(32) unsigned char s_keys[];
  const SelectArgs& a = batch.a[blockIdx.z];
  const int b = blockIdx.y, n4 = (a.nW + 3) / 4;
  const int64_t* sc = a.score + (long)b * a.nW;
  const int lane = threadIdx.x & 31, w = blockIdx.x * RANK_WARPS + (threadIdx.x >> 5);
  const int Hp = (a.H + WS - 1) / WS * WS, Wp = (a.W + WS - 1) / WS * WS;
  auto rank_with = [&](auto* key, auto lowest) {
    for (int i = threadIdx.x; i < 4 * n4; i += blockDim.x)
      key[i] = i < a.nW ? (decltype(lowest))(a.reverse ? -sc[i] : sc[i]) : lowest;
    __syncthreads();
    if (w < a.nW) emit_window(a, b, w, count_preceding(key, n4, w, lane), lane, Hp, Wp);
  };
  if (a.narrow) rank_with(reinterpret_cast<int*>(s_keys), (int)INT_MIN);
  else rank_with(reinterpret_cast<long long*>(s_keys), (long long)LLONG_MIN);
}

// Score, rank and bookkeeping of one (image, block) in one CTA with a warp per window, for images of at most 32 windows:
// there the two kernels above are launch latency, and one CTA needs no exchange through global memory.  A whole block call
// with one against two launches (us): 43.9 and 45.5 at 4 windows, 37.1 and 37.9 at 16, 36.2 and 36.9 at 25; with two windows
// per warp it is the other way round, 38.9 and 37.4 at 36, 39.7 and 38.1 at 49, 41.1 and 39.0 at 64 windows.  (Only for 16
// images and the 18 blocks of a deep stage in one launch is the single kernel still 2 us faster up to 64 windows.)
constexpr int SMALL_WINDOWS = 32;
__global__ void __launch_bounds__(SMALL_WINDOWS * 32) k_select_small(const __grid_constant__ SelectBatch batch) {
  __shared__ __align__(32) long long s_score[SMALL_WINDOWS];
  griddep_wait();
  griddep_launch();
  const SelectArgs& a = batch.a[blockIdx.y];
  const int b = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int Hp = (a.H + WS - 1) / WS * WS, Wp = (a.W + WS - 1) / WS * WS;
  if (w < a.nW) {
    long long s = 0;
    for (int t = lane; t < WT; t += 32) {
      const int src = window_src(b, a.H, a.W, Hp, Wp, a.shift, a.nwx, w, t);
      if (src >= 0) s += a.energy[src];
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) { s_score[w] = a.reverse ? -s : s; a.score[(long)b * a.nW + w] = s; }
  } else if (lane == 0) {
    s_score[w] = LLONG_MIN;
  }
  __syncthreads();
  if (w < a.nW) emit_window(a, b, w, count_preceding(s_score, SMALL_WINDOWS / 4, w, lane), lane, Hp, Wp);
}

// One CTA per image: every warp takes a run of windows, counts the members of the three classes in it, and writes them behind those
// of the warps before it (order-preserving compaction by ballot).  One warp per class took 25 us at 3 025 windows.
constexpr int LIST_WARPS = 32;
struct ClassListArgs { const uint8_t* cls; int32_t* out[3]; int count[3]; int B, nW; };
__global__ void __launch_bounds__(LIST_WARPS * 32) k_class_lists(ClassListArgs a) {
  __shared__ int s_count[3][LIST_WARPS];
  griddep_launch();
  griddep_wait();
  const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint8_t* cls = a.cls + (long)b * a.nW;
  const int per = ((a.nW + LIST_WARPS - 1) / LIST_WARPS + 31) / 32 * 32, first = warp * per, end = min(a.nW, first + per);
  int base[3] = {0, 0, 0};
  for (int w0 = first; w0 < end; w0 += 32) {
    const int c = w0 + lane < end ? cls[w0 + lane] : 3;
#pragma unroll
    for (int k = 0; k < 3; ++k) base[k] += __popc(__ballot_sync(0xffffffffu, c == k));
  }
  if (lane < 3) s_count[lane][warp] = lane == 0 ? base[0] : lane == 1 ? base[1] : base[2];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 3; ++k) base[k] = __reduce_add_sync(0xffffffffu, lane < warp ? s_count[k][lane] : 0);
  for (int w0 = first; w0 < end; w0 += 32) {
    const int c = w0 + lane < end ? cls[w0 + lane] : 3;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, c == k);
      if (c == k && a.out[k]) a.out[k][(long)b * a.count[k] + base[k] + __popc(m & ((1u << lane) - 1u))] = w0 + lane;
      base[k] += __popc(m);
    }
  }
}

void launch_class_lists(const uint8_t* cls, int B, int nW, int32_t* const out[3], const int count[3], cudaStream_t st) {
  ClassListArgs a;
  a.cls = cls; a.B = B; a.nW = nW;
  for (int c = 0; c < 3; ++c) { a.out[c] = out[c]; a.count[c] = count[c]; }
  launch_pdl(k_class_lists, dim3(B), LIST_WARPS * 32, 0, st, a);
  ++g_launches;
}

void launch_energy(const float* x, int32_t* energy, long ntok, int C, float inv_scale, cudaStream_t st) {
  launch_pdl(k_energy, dim3((unsigned)((ntok * 8 + 255) / 256)), 256, 0, st, x, energy, ntok, C, inv_scale);
  ++g_launches;
}

void launch_select(const SelectArgs* args, int count, cudaStream_t st) {
  // all entries share B, H, W (one stage); shift, ratios and output buffers differ
  for (int first = 0; first < count; first += MAX_SELECT_BATCH) {
    const int n = count - first < MAX_SELECT_BATCH ? count - first : MAX_SELECT_BATCH;
    SelectBatch batch;
    for (int i = 0; i < n; ++i) batch.a[i] = args[first + i];
    for (int i = n; i < MAX_SELECT_BATCH; ++i) batch.a[i] = args[first];
    const SelectArgs& a = args[first];
    if (a.nW <= SMALL_WINDOWS) {
      launch_pdl(k_select_small, dim3(a.B, n), SMALL_WINDOWS * 32, 0, st, batch);
      ++g_launches;
      continue;
    }
    const int nwin = a.B * a.nW;
    launch_pdl(k_window_score, dim3((nwin + 7) / 8, n), 256, 0, st, batch);
    ++g_launches;
    dim3 grid((a.nW + RANK_WARPS - 1) / RANK_WARPS, a.B, n);
    launch_pdl(k_rank_emit, grid, RANK_WARPS * 32, (size_t)(a.nW + 3) / 4 * 4 * sizeof(long long), st, batch);
    ++g_launches;
  }
}

// ---- guard zones ---------------------------------------------------------------------------------------
namespace {
constexpr int GUARD_BATCH = 48;
constexpr uint32_t GUARD_PATTERN = 0xA5C3E1B7u;
struct GuardList { uint32_t* zone[GUARD_BATCH]; };
template <bool FILL>
__global__ void k_guards(GuardList g, int* status) {
  uint32_t* z = g.zone[blockIdx.x];
  const int i = threadIdx.x;                               // GUARD_BYTES / 4 threads
  if (FILL) z[i] = GUARD_PATTERN ^ (uint32_t)i;
  else if (z[i] != (GUARD_PATTERN ^ (uint32_t)i)) atomicOr(status, 2);
}
}  // namespace

void launch_guards(void* const* zones, int count, bool fill, int* status, cudaStream_t st) {
  for (int first = 0; first < count; first += GUARD_BATCH) {
    const int n = count - first < GUARD_BATCH ? count - first : GUARD_BATCH;
    GuardList g;
    for (int i = 0; i < GUARD_BATCH; ++i) g.zone[i] = (uint32_t*)zones[first + (i < n ? i : 0)];
    if (fill) k_guards<true><<<n, GUARD_BYTES / 4, 0, st>>>(g, status);
    else k_guards<false><<<n, GUARD_BYTES / 4, 0, st>>>(g, status);
  }
}

}  // namespace mixaq
