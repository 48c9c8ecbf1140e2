// Fused epilogues of the integer GEMMs (MixA-Q Section 3.2: shared integer weights, per-branch step sizes,
// zero points and biases).  One epilogue warp owns 32 rows (one TMEM lane quarter) and every c_step-th chunk of the tile, 32
// columns wide for the code outputs and 16 for the binary32 outputs (the warps of a group that share a lane quarter deal the
// chunks round-robin).  A quad of lanes holds a row of a chunk, lane t of it 8 (4) consecutive channels, of rows l / 4 + 0, 8, 16,
// 24: the accumulator is read in the layout of tmem_ld_quads and the weights arrive with their rows in the matching order
// (make_quad_map).
//   raw[n] = sum_k a[m][k] * w[n][k]                   with UNSIGNED activation codes a;
//   acc[n] = raw[n] - z_a * sum_k w[n][k]              (zero-point correction, exact in int32)
//   v[n]       = fma((float)acc[n], s_a*s_w[n], bias[n])
// The per-column constants (pre, mult, bias) sit in shared memory.  With a row per lane every warp read all of a chunk's constants in
// every lane, 12 bytes a value through a 128-byte path: a quarter of the fc1 epilogue's time and half of the QKV epilogue's.  Now a
// value read serves four rows, and the binary32 outputs need no transposition through shared memory.  B200, 294 912 rows of 128
// channels, before and after: QKV 58.4 -> 49.0 us, proj 60.1 -> 55.1, fc1 137.5 -> 137.2, fc2 76.1 -> 76.1; 18 432 rows of 512: QKV
// 23.4 -> 20.4, proj 23.0 -> 20.9, fc1 46.4 -> 45.0, fc2 33.1 -> 33.8.  Since the warp number comes through a shuffle (gemm_tc.cu):
// 47.7, 54.0, 120.1, 74.8 and 20.4, 20.1, 40.1, 34.0.
#pragma once
#include "kernels.h"
#include "tc_ptx.cuh"
#include <type_traits>

namespace mixaq {

constexpr int CODE_NC = 32, F32_NC = 16;               // columns per chunk of the code and of the binary32 epilogues
constexpr int EPI_CHUNK_FLOATS = 32 * F32_NC;          // a residual chunk of the binary32 epilogues

struct ColConsts {                                     // shared-memory arrays indexed by the column within the tile
  const int32_t* pre; const float* mult; const float* bias;
};

// asynchronous 16-byte copy global -> shared (no register staging); groups complete in order
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int RES_SLOTS = 4;                           // residual chunks a warp keeps in flight (32 x 16 floats each)

// raw + pre[n] is 0x4B400000 + acc: the zero point is taken out, and while |acc| < 2^22 (NARROW) those bits ARE the
// binary32 number 1.5 * 2^23 + acc, so one packed subtraction converts two of them.
template <bool NARROW>
__device__ __forceinline__ float2 acc_to_float2(int32_t a, int32_t b) {
  if (NARROW) return __fadd2_rn(make_float2(__int_as_float(a), __int_as_float(b)), f2(-12582912.0f));
  return make_float2(__int2float_rn(a - (int32_t)kMagicBits), __int2float_rn(b - (int32_t)kMagicBits));
}
// the constants of four columns
struct Consts4 {
  int4 pre; float4 mult, bias;
  template <bool BIAS> __device__ __forceinline__ void load(const ColConsts& cc, int lc) {
    pre = *reinterpret_cast<const int4*>(cc.pre + lc);
    mult = *reinterpret_cast<const float4*>(cc.mult + lc);
    bias = BIAS ? *reinterpret_cast<const float4*>(cc.bias + lc) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};
// Dequantization of four columns of a row, two per packed instruction (each lane rounds like the scalar fma / mul).
// tap: where the accumulators of these columns go, or nullptr
template <int MODE, bool TAPS, bool NARROW>
__device__ __forceinline__ void dequant4(const Consts4& k, int32_t a0, int32_t a1, int32_t a2, int32_t a3, int32_t* tap, float2& lo, float2& hi) {
  if (TAPS && tap) {
    tap[0] = a0 + k.pre.x - (int32_t)kMagicBits; tap[1] = a1 + k.pre.y - (int32_t)kMagicBits;
    tap[2] = a2 + k.pre.z - (int32_t)kMagicBits; tap[3] = a3 + k.pre.w - (int32_t)kMagicBits;
  }
  const float2 f0 = acc_to_float2<NARROW>(a0 + k.pre.x, a1 + k.pre.y), f1 = acc_to_float2<NARROW>(a2 + k.pre.z, a3 + k.pre.w);
  if (MODE == EPI_MERGE) {
    lo = __fmul2_rn(f0, make_float2(k.mult.x, k.mult.y)); hi = __fmul2_rn(f1, make_float2(k.mult.z, k.mult.w));
  } else {
    lo = __ffma2_rn(f0, make_float2(k.mult.x, k.mult.y), make_float2(k.bias.x, k.bias.y));
    hi = __ffma2_rn(f1, make_float2(k.mult.z, k.mult.w), make_float2(k.bias.z, k.bias.w));
  }
}

// ---- quantizers of the code outputs ------------------------------------------------------------------------------------
// Both leave rne(x * inv_scale) (FC1: + zp) in the low 16 bits of every pattern, unclamped; clamp_pack4 adds, clamps and
// packs.  They need |x * inv_scale| < 2^15, which `in_range` of the caller guarantees (the channel's bound + |bias|, times
// inv_scale); launches for which that cannot be shown take the exact functions with their binary32 clamps.
constexpr float kPatternRange = 30000.0f;

// QKV: t = x * inv_scale rounded, then the rounding add.  A packed multiply feeding a packed add would be contracted into
// one rounding; the multiply is therefore written as fma(x, inv_scale, -0) (same value) with a -0 the compiler cannot see.
__device__ __forceinline__ void quant_pattern2(float2 x, float inv_scale, float neg_zero, uint32_t& m0, uint32_t& m1) {
  const float2 t = __fadd2_rn(__ffma2_rn(x, f2(inv_scale), f2(neg_zero)), f2(12582912.0f));
  m0 = __float_as_uint(t.x); m1 = __float_as_uint(t.y);
}
// FC1: code of GELU(v) from a polynomial of degree 6 and the special-function exponential instead of the contract's two polynomials
// (a third of the packed operations).  The value can differ from the contract's in the last bits, so `dist` collects the largest distance
// to the nearest integer; where it comes within the error bound of one half (see gelu_threshold) the caller recomputes.
// The zero point is part of the rounding constant; at exact ties that changes the parity rule, and ties are recomputed.
__device__ __forceinline__ void gelu_pattern2(float2 v, float inv_scale, float magic_zp, float& dist, uint32_t& m0, uint32_t& m1) {
  const float2 a = make_float2(fmaxf(-fabsf(v.x), -5.0f), fmaxf(-fabsf(v.y), -5.0f));        // minus the contract's a
  const float2 q = gelu_log2_tail_neg2(a);
  const float2 g = __ffma2_rn(a, make_float2(ex2_approx(q.x), ex2_approx(q.y)), make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f)));
  const float2 r = __ffma2_rn(g, f2(inv_scale), f2(magic_zp));
  const float2 n = __fadd2_rn(f2(magic_zp), make_float2(-r.x, -r.y));          // minus the rounded value, exactly
  const float2 d = __ffma2_rn(g, f2(inv_scale), n);
  asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(dist) : "f"(d.x), "f"(d.y));
  m0 = __float_as_uint(r.x); m1 = __float_as_uint(r.y);
}
// Distance of g * inv_scale from the contract's t: the polynomials change h = a 2^q <= 0.17 by at most 6.4e-8, both exponentials are
// within 2^-22 of theirs, so h differs by at most 6.4e-8 + 0.17 * 2^-21 + one rounding < 1.7e-7; g is rounded in both evaluations
// and t in the contract's, which adds |t| * 3 * 2^-24, and |t| <= max(code, zp) + 1 for every t that is not clamped anyway; the
// distance itself is rounded by 2^-26.
// maxf: at least the codes in question and the zero point
__device__ __forceinline__ float gelu_threshold(float inv_scale, float maxf) {
  return 0.5f - __fmaf_rn(inv_scale, 1.9e-7f, (maxf + 2.0f) * 1.8e-7f);
}

// Four columns of two of the lane's rows by the contract's own operations, read again from tensor memory.  A function of its own: its
// twenty constants and its temporaries would otherwise take registers of the loop that hardly ever comes here.
template <int MODE>
__device__ __noinline__ uint2 codes_exact8(uint32_t taddr, ColConsts cc, int lc, float inv_scale, float zpf, float qmaxf) {
  int32_t a[8];
  tmem_ld_quads(taddr, a);
  Consts4 k;
  k.load<true>(cc, lc);
  tmem_ld_wait(a);
  const uint32_t zp2 = (uint32_t)zpf * 0x10001u, qmax2 = (uint32_t)qmaxf * 0x10001u;
  uint32_t w[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    float2 v0, v1;
    uint32_t c[4];
    dequant4<MODE, false, false>(k, a[2 * j], a[2 * j + 1], a[2 * j + 4], a[2 * j + 5], nullptr, v0, v1);
    quant_magic2(MODE == EPI_FC1 ? gelu_f2(v0) : v0, inv_scale, -zpf, qmaxf - zpf, c[0], c[1]);
    quant_magic2(MODE == EPI_FC1 ? gelu_f2(v1) : v1, inv_scale, -zpf, qmaxf - zpf, c[2], c[3]);
    w[j] = clamp_pack4<true>(c[0], c[1], c[2], c[3], zp2, qmax2);
  }
  return make_uint2(w[0], w[1]);
}

// What a warp's epilogue needs of its branch, read once per branch (the parameters sit in constant memory, and a tile used
// to read them again field by field).
struct EpiBranch {
  int M, cbits;                                            // code outputs: bits a stored code takes
  uint8_t* out_codes; float* out_f; const float* res; const int32_t* rowsrc;
  long row_bytes;                                          // code outputs: bytes of an output row
  float qmaxf;                                             // largest code
  __device__ __forceinline__ EpiBranch(const GemmBranch& b, int N)
      : M(b.M), cbits(b.out_bits), out_codes(b.out_codes), out_f(b.out_f), res(b.res), rowsrc(b.rowsrc),
        row_bytes((long)N * b.out_bits / 8), qmaxf(b.q0.qmaxf) {}
};

// The warp's part of one output tile.  taddr: TMEM address of (the warp's lane quarter, the tile's first column);
// n_tile0: global index of that column; the warp owns the tile's chunks c_first, c_first + c_step, ... < c_total
// cc: the constants of the tile's columns;
// narrow: no sum of the tile's columns reaches 2^22 (see acc_to_float2);
// in_range: the code outputs of the tile's columns cannot leave the pattern's range (see quant_pattern2);
// acc_ready(): waits (bounded) for the tile's accumulator, false when the CTA is giving up.
template <int MODE, bool TAPS, class WaitFn>
__device__ __forceinline__ bool epilogue_warp_tile(const GemmBranch& br, const EpiBranch& eb, int N, int C, long row0, int lane, int n_tile0,
                                                   int c_first, int c_step, int c_total, const ColConsts& cc,
                                                   uint32_t taddr_tile, bool narrow, bool in_range, float neg_zero, WaitFn acc_ready,
                                                   float* res_ring = nullptr /* per warp: RES_SLOTS x 32 x 16 floats */) {
  // this lane's rows: row0 + 8 i + rsub, i = 0 ... 3; rows_left: how many of the warp's rows exist
  const int cj = lane & 3, rsub = lane >> 2;
  const int rows_left = row0 + 32 <= eb.M ? 32 : (int)(eb.M - row0);
  constexpr int NC = MODE == EPI_QKV || MODE == EPI_FC1 ? CODE_NC : F32_NC;
  constexpr int LANE_COLS = NC / 4;                        // consecutive columns of a lane
  const int n_chunks = c_first < c_total ? (c_total - c_first + c_step - 1) / c_step : 0;
  const int n_first = n_tile0 + c_first * NC + LANE_COLS * cj;   // global column of this lane's first one
  const int lc_first = c_first * NC + LANE_COLS * cj;            // and within the tile
  const int col_step = c_step * NC;                        // distance between consecutive chunks of the warp
  const uint32_t taddr = taddr_tile + (uint32_t)(c_first * NC);
  auto tap_at = [&](int i, int col) -> int32_t* {          // the accumulator tap of this lane's i-th row, tile column col
    return TAPS && br.tap_acc && 8 * i + rsub < rows_left ? br.tap_acc + (row0 + 8 * i + rsub) * N + n_tile0 + col : nullptr;
  };

  if (MODE == EPI_QKV || MODE == EPI_FC1) {
    // ---- code outputs: a thread quantizes and packs 8 codes of each of its four rows; a quad stores 32 codes side by side ----
    // a tile lies within one of the q, k, v sections (its width divides a section's), so its quantizer is the tile's
    const AQ& q = MODE == EPI_FC1 || n_tile0 < C ? br.q0 : (n_tile0 < 2 * C ? br.q1 : br.q2);
    const float inv_scale = q.inv_scale, zpf = q.zpf;
    const int cbits = eb.cbits;
    const uint32_t zp2 = (uint32_t)q.zp * 0x10001u, qmax2 = (uint32_t)eb.qmaxf * 0x10001u;
    const float magic_zp = 12582912.0f + zpf;                              // FC1
    const float thr = gelu_threshold(inv_scale, eb.qmaxf);                 // FC1
    // this thread's output position in its first row of the warp's first chunk, and the distance of its rows
    uint8_t* out_ptr = eb.out_codes + (row0 + rsub) * eb.row_bytes + n_first * cbits / 8;
    const int row_step = 8 * (int)eb.row_bytes;
    const int out_step = col_step * cbits / 8;
    if (!acc_ready()) return false;
    // 32 columns at a time, without a branch between them: the dependent chain of a value is about twenty operations
    // long, and with three warps per scheduler only independent values hide its latency.  The accumulator comes in halves of 16
    // columns (four of this lane's in each of its rows), each requested a half ahead, the first one of the next chunk behind the
    // second one of this.
    int32_t first[16], second[16];
    if (n_chunks > 0) tmem_ld_quads32(taddr, first);
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ++ch) {
      const uint32_t ta = taddr + (uint32_t)(ch * col_step);
      const int lc = lc_first + ch * col_step;
      uint32_t w[4][2];                                                    // [row][half of the columns]
      float dist[4];                                                       // [2 * half of the columns + half of the rows]
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h == 0) { tmem_ld_wait(first); tmem_ld_quads32(ta + 16u, second); }
        else        { tmem_ld_wait(second); if (ch + 1 < n_chunks) tmem_ld_quads32(ta + (uint32_t)col_step, first); }
        const int32_t (&a)[16] = h == 0 ? first : second;
        Consts4 k;
        k.load<true>(cc, lc + 4 * h);
        dist[2 * h] = 0.0f; dist[2 * h + 1] = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int o = 8 * (i >> 1) + 2 * (i & 1);
          float2 v0, v1;
          uint32_t c[4];
          dequant4<MODE, TAPS, false>(k, a[o], a[o + 1], a[o + 4], a[o + 5], tap_at(i, lc + 4 * h), v0, v1);
          if (MODE == EPI_FC1) {
            float& d = dist[2 * h + (i >> 1)];
            gelu_pattern2(v0, inv_scale, magic_zp, d, c[0], c[1]); gelu_pattern2(v1, inv_scale, magic_zp, d, c[2], c[3]);
          } else {
            quant_pattern2(v0, inv_scale, neg_zero, c[0], c[1]); quant_pattern2(v1, inv_scale, neg_zero, c[2], c[3]);
          }
          w[i][h] = clamp_pack4<MODE != EPI_FC1>(c[0], c[1], c[2], c[3], zp2, qmax2);
        }
        if (TAPS) __syncwarp();                              // (rows that exist were tapped)
      }
      // Half of the columns of half of the rows again by the contract's own operations: where some value of the warp is too close
      // to a rounding boundary, and all of them where the patterns above do not hold.  A sixth of the chunks at A8 has a value
      // within the bound for the largest code; with the bound for the lane's own codes, which are mostly small, few of them are left.
      const bool near = MODE == EPI_FC1 && fmaxf(fmaxf(dist[0], dist[1]), fmaxf(dist[2], dist[3])) >= thr;
      if (!in_range || (MODE == EPI_FC1 && __any_sync(0xffffffffu, near))) {
        tmem_ld_wait(first);                                 // nothing may be on its way into registers across a call
        uint32_t todo = 0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t any = w[2 * (g & 1)][g >> 1] | w[2 * (g & 1) + 1][g >> 1];      // no code is above the bits of all of them
          any |= any >> 16; any |= any >> 8;
          const float t = gelu_threshold(inv_scale, fmaxf((float)(any & 0xFFu), zpf));
          if (!in_range || __any_sync(0xffffffffu, dist[g] >= t)) todo |= 1u << g;
        }
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
          if (!(todo >> g & 1u)) continue;
          const int h = g >> 1, i0 = 2 * (g & 1);
          const uint2 pk = codes_exact8<MODE>(ta + ((uint32_t)(8 * i0) << 16) + (uint32_t)(16 * h), cc, lc + 4 * h, inv_scale, zpf, eb.qmaxf);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) w[i][hh] = g == 2 * hh + (i >> 1) ? ((i & 1) ? pk.y : pk.x) : w[i][hh];
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (8 * i + rsub < rows_left) store_codes8(out_ptr + i * (long)row_step + ch * out_step, w[i][0], w[i][1], cbits);
      __syncwarp();                                          // tensor memory is read by all lanes at once
    }
    return true;
  }

  // ---- binary32 outputs (proj: x1 = x_window + out; fc2: y = x1 + out scattered to the token's own position;
  //      merge: out).  A lane holds 16 bytes of a row, so global accesses are 64-byte runs (4 lanes per row, 8 rows per instruction)
  //      and the constants are those of 4 columns. ----
  int src_mine = -1;
  if (MODE != EPI_MERGE && lane < rows_left) src_mine = eb.rowsrc[row0 + lane];
  // this lane's four pieces of the warp's first chunk: residual source and output, NULL: none
  const float* res_ptr[4];
  float* dst_ptr[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 8 * i + rsub;
    const long mr = row0 + r;
    const long s = __shfl_sync(0xffffffffu, src_mine, r);
    const bool ok = r < rows_left;
    long res_row, dst_row;               // row offsets (in elements), -1: none
    if (MODE == EPI_PROJ)     { res_row = (ok && s >= 0) ? s * N : -1;  dst_row = ok ? mr * N : -1; }
    else if (MODE == EPI_FC2) { res_row = (ok && s >= 0) ? mr * N : -1; dst_row = (ok && s >= 0) ? s * N : -1; }
    else                      { res_row = -1;                            dst_row = ok ? mr * N : -1; }
    res_ptr[i] = (MODE != EPI_MERGE && res_row >= 0) ? eb.res + res_row + n_first : nullptr;
    dst_ptr[i] = dst_row >= 0 ? eb.out_f + dst_row + n_first : nullptr;
  }
  // The residual pieces come into shared memory by asynchronous copies, RES_SLOTS chunks ahead of their use: the copies
  // of a whole tile are in flight while the accumulator is still being computed, and they cost no registers.
  // Slot ch % RES_SLOTS holds chunk ch; a lane reads what it has copied itself, so nothing but its own copies is waited for.  One
  // commit group per chunk, also when there is nothing left to fetch, so that "all but the newest RES_SLOTS - 1 groups are
  // complete" always covers the chunk about to be used.
  auto fetch = [&](int ch) {
    if (MODE != EPI_MERGE && ch < n_chunks) {
      float* slot = res_ring + (ch % RES_SLOTS) * EPI_CHUNK_FLOATS + 4 * lane;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (res_ptr[i]) cp_async16(slot + 128 * i, res_ptr[i] + ch * col_step);
        else *reinterpret_cast<float4*>(slot + 128 * i) = make_float4(0.f, 0.f, 0.f, 0.f);   // a pad token's residual input is zero
      }
    }
    cp_async_commit();
  };
  if (MODE != EPI_MERGE) {
#pragma unroll
    for (int ch = 0; ch < RES_SLOTS; ++ch) fetch(ch);
  }
  if (!acc_ready()) { cp_async_wait<0>(); return false; }
  auto walk = [&](auto narrow_tag) {
    constexpr bool NARROW = decltype(narrow_tag)::value;
    auto finish = [&](int ch, const int32_t (&a)[16]) {
      const int lc = lc_first + ch * col_step;
      Consts4 k;
      k.load<MODE != EPI_MERGE>(cc, lc);
      if (MODE != EPI_MERGE) cp_async_wait<RES_SLOTS - 1>();     // this lane's copies of chunk ch have landed
      const float* slot = res_ring + (ch % RES_SLOTS) * EPI_CHUNK_FLOATS + 4 * lane;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int o = 8 * (i >> 1) + 2 * (i & 1);
        float2 lo, hi;
        dequant4<MODE, TAPS, NARROW>(k, a[o], a[o + 1], a[o + 4], a[o + 5], tap_at(i, lc), lo, hi);
        if (!dst_ptr[i]) continue;
        if (MODE != EPI_MERGE) {
          const float4 rr = *reinterpret_cast<const float4*>(slot + 128 * i);
          lo = __fadd2_rn(make_float2(rr.x, rr.y), lo); hi = __fadd2_rn(make_float2(rr.z, rr.w), hi);
        }
        *reinterpret_cast<float4*>(dst_ptr[i] + ch * col_step) = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
      if (MODE != EPI_MERGE) fetch(ch + RES_SLOTS);              // the slot just read is free again
      __syncwarp();                                              // (lanes without a place to store to went another way)
    };
    // two chunks in turn, each requested one ahead
    int32_t even[16], odd[16];
    if (n_chunks > 0) tmem_ld_quads32(taddr, even);
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ch += 2) {
      tmem_ld_wait(even);
      if (ch + 1 < n_chunks) tmem_ld_quads32(taddr + (uint32_t)((ch + 1) * col_step), odd);
      finish(ch, even);
      if (ch + 1 >= n_chunks) break;
      tmem_ld_wait(odd);
      if (ch + 2 < n_chunks) tmem_ld_quads32(taddr + (uint32_t)((ch + 2) * col_step), even);
      finish(ch + 1, odd);
    }
  };
  if (narrow) walk(std::true_type{}); else walk(std::false_type{});
  if (MODE != EPI_MERGE) cp_async_wait<0>();                   // nothing of this tile is left in flight
  return true;
}

}  // namespace mixaq
