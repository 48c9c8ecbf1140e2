// Fused epilogues of the integer GEMMs (MixA-Q Section 3.2: shared integer weights, per-branch step sizes,
// zero points and biases).  One epilogue warp owns 32 rows (one TMEM lane quarter, one row per thread) and every
// c_step-th chunk of the tile, 32 columns wide for the code outputs and 16 for the binary32 outputs (the warps of a group
// that share a lane quarter deal the chunks round-robin):
//   raw[n] = sum_k a[m][k] * w[n][k]                   with UNSIGNED activation codes a;
//   acc[n] = raw[n] - z_a * sum_k w[n][k]              (zero-point correction, exact in int32)
//   v[n]       = fma((float)acc[n], s_a*s_w[n], bias[n])
// The per-column constants (pre, mult, bias) sit in shared memory; every lane reads the same
// column, so the reads are broadcasts.
#pragma once
#include "kernels.h"
#include "tc_ptx.cuh"
#include <type_traits>

namespace mixaq {

constexpr int CODE_NC = 32, F32_NC = 16;               // columns per chunk of the code and of the binary32 epilogues
constexpr int EPI_STAGE_FLOATS = 32 * F32_NC;          // per-warp transposition tile of the binary32 epilogues

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
// dequantization of NC columns; lc0 = first column in the warp's constants, n0 = its global index
template <int MODE, bool TAPS, bool NARROW, int NC>
__device__ __forceinline__ void dequant(const GemmBranch& br, int N, long m, bool row_ok, int n0, int lc0, const ColConsts& cc,
                                        const int32_t* acc, float (&v)[NC]) {
  if (TAPS && br.tap_acc && row_ok) {
#pragma unroll
    for (int i = 0; i < NC; ++i) br.tap_acc[m * N + n0 + i] = acc[i] + cc.pre[lc0 + i] - (int32_t)kMagicBits;
  }
#pragma unroll
  for (int i4 = 0; i4 < NC / 4; ++i4) {
    const int4 p4 = *reinterpret_cast<const int4*>(cc.pre + lc0 + 4 * i4);
    const int pp[4] = {p4.x, p4.y, p4.z, p4.w};
    const float4 m4 = *reinterpret_cast<const float4*>(cc.mult + lc0 + 4 * i4);
    const float mm[4] = {m4.x, m4.y, m4.z, m4.w};
    float bb[4] = {0.f, 0.f, 0.f, 0.f};
    if (MODE != EPI_MERGE) {
      const float4 b4 = *reinterpret_cast<const float4*>(cc.bias + lc0 + 4 * i4);
      bb[0] = b4.x; bb[1] = b4.y; bb[2] = b4.z; bb[3] = b4.w;
    }
    // two columns per packed instruction (each lane rounds like the scalar fma / mul)
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
      const int i = 4 * i4 + j;
      const float2 f = acc_to_float2<NARROW>(acc[i] + pp[j], acc[i + 1] + pp[j + 1]);
      const float2 r = MODE == EPI_MERGE ? __fmul2_rn(f, make_float2(mm[j], mm[j + 1]))
                                         : __ffma2_rn(f, make_float2(mm[j], mm[j + 1]), make_float2(bb[j], bb[j + 1]));
      v[i] = r.x; v[i + 1] = r.y;
    }
  }
}

// ---- quantizers of the code outputs ------------------------------------------------------------------------------------
// Both leave rne(x * inv_scale) (FC1: + zp) in the low 16 bits of every pattern, unclamped; sat_pack4 adds, clamps and
// packs.  They need |x * inv_scale| < 2^15, which `in_range` of the caller guarantees (the channel's bound + |bias|, times
// inv_scale); launches for which that cannot be shown take the exact functions with their binary32 clamps.
constexpr float kPatternRange = 30000.0f;

// QKV: t = x * inv_scale rounded, then the rounding add.  A packed multiply feeding a packed add would be contracted into
// one rounding; the multiply is therefore written as fma(x, inv_scale, -0) (same value) with a -0 the compiler cannot see.
__device__ __forceinline__ void quant_pattern2(float2 x, float inv_scale, float neg_zero, uint32_t& m0, uint32_t& m1) {
  const float2 t = __fadd2_rn(__ffma2_rn(x, f2(inv_scale), f2(neg_zero)), f2(12582912.0f));
  m0 = __float_as_uint(t.x); m1 = __float_as_uint(t.y);
}
// FC1: code of GELU(v) from the special-function exponential instead of the contract's polynomial (a third of the
// packed operations).  The value can differ from the contract's in the last bits, so `dist` collects the largest distance
// to the nearest integer; where it comes within the error bound of one half (see gelu_threshold) the caller recomputes.
// The zero point is part of the rounding constant; at exact ties that changes the parity rule, and ties are recomputed.
__device__ __forceinline__ void gelu_pattern2(float2 v, float inv_scale, float magic_zp, float& dist, uint32_t& m0, uint32_t& m1) {
  const float2 a = make_float2(fminf(fabsf(v.x), 5.0f), fminf(fabsf(v.y), 5.0f));
  const float2 q = gelu_log2_tail2(a);
  const float2 h = __fmul2_rn(a, make_float2(ex2_approx(q.x), ex2_approx(q.y)));
  const float2 g = sub2(make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f)), h);
  const float2 r = __ffma2_rn(g, f2(inv_scale), f2(magic_zp));
  const float2 n = __fadd2_rn(f2(magic_zp), make_float2(-r.x, -r.y));          // minus the rounded value, exactly
  const float2 d = __ffma2_rn(g, f2(inv_scale), n);
  dist = fmaxf(fmaxf(dist, fabsf(d.x)), fabsf(d.y));
  m0 = __float_as_uint(r.x); m1 = __float_as_uint(r.y);
}
// Distance of g * inv_scale from the contract's t: both exponentials are within 2^-22 of 2^q, h = a 2^q <= 0.17, so h differs
// by at most 0.17 * 2^-21 + one rounding < 1.0e-7; g is rounded in both evaluations and t in the contract's, which adds
// |t| * 3 * 2^-24, and |t| <= qmax + 1 for every t that is not clamped anyway; the distance itself is rounded by 2^-26.
__device__ __forceinline__ float gelu_threshold(float inv_scale, float qmaxf) {
  return 0.5f - __fmaf_rn(inv_scale, 1.1e-7f, (qmaxf + 2.0f) * 1.8e-7f);
}

// What a warp's epilogue needs of its branch, read once per branch (the parameters sit in constant memory, and a tile used
// to read them again field by field).
struct EpiBranch {
  int M, bits, cbits;                                      // code outputs: width of the codes, bits a stored code takes
  uint8_t* out_codes; float* out_f; const float* res; const int32_t* rowsrc;
  long row_bytes;                                          // code outputs: bytes of an output row
  float qmaxf;                                             // largest code
  __device__ __forceinline__ EpiBranch(const GemmBranch& b, int N)
      : M(b.M), bits(b.q0.bits), cbits(b.out_bits), out_codes(b.out_codes), out_f(b.out_f), res(b.res), rowsrc(b.rowsrc),
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
                                                   uint32_t taddr_tile, float* stage, bool narrow, bool in_range, float neg_zero, WaitFn acc_ready,
                                                   float* res_ring = nullptr /* per warp: RES_SLOTS x 32 x 16 floats */) {
  const long m = row0 + lane;
  const bool row_ok = m < eb.M;
  constexpr int NC = MODE == EPI_QKV || MODE == EPI_FC1 ? CODE_NC : F32_NC;
  const int n_chunks = c_first < c_total ? (c_total - c_first + c_step - 1) / c_step : 0;
  const int n_first = n_tile0 + c_first * NC;              // global column of the warp's first chunk
  const int col_step = c_step * NC;                        // distance between consecutive chunks of the warp
  const uint32_t taddr = taddr_tile + (uint32_t)(c_first * NC);

  if (MODE == EPI_QKV || MODE == EPI_FC1) {
    // ---- code outputs: every thread quantizes and packs the 32 codes of its own row ----
    // a tile lies within one of the q, k, v sections (its width divides a section's), so its quantizer is the tile's
    const AQ& q = MODE == EPI_FC1 || n_tile0 < C ? br.q0 : (n_tile0 < 2 * C ? br.q1 : br.q2);
    const float inv_scale = q.inv_scale, zpf = q.zpf;
    const int cbits = eb.cbits, bits = eb.bits;
    const uint32_t zbias = (MODE == EPI_FC1 ? 0u : (uint32_t)q.zp) - kMagicBits;
    const float magic_zp = 12582912.0f + zpf;                              // FC1
    const float thr = gelu_threshold(inv_scale, eb.qmaxf);                 // FC1
    // this thread's output position of the warp's first chunk
    uint8_t* out_ptr = eb.out_codes + m * eb.row_bytes + n_first * cbits / 8;
    const int out_step = col_step * cbits / 8;
    if (!acc_ready()) return false;
    // the quantizer's width as a constant (a shift in the packing)
    auto walk = [&](auto bits_tag) {
      constexpr int SH = 8 - decltype(bits_tag)::value;
      // 32 columns at a time, without a branch between them: the dependent chain of a value is about twenty operations
      // long, and with four warps per scheduler only independent values hide its latency.  The accumulator comes in halves of 16
      // columns, each requested a half ahead, the first one of the next chunk behind the second one of this.
      int32_t first[CODE_NC / 2], second[CODE_NC / 2];
      if (n_chunks > 0) tmem_ld(taddr, first);
#pragma unroll 1
      for (int ch = 0; ch < n_chunks; ++ch) {
        const uint32_t ta = taddr + (uint32_t)(ch * col_step);
        const int col = c_first * CODE_NC + ch * col_step;
        uint32_t w[8];
        float dist[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (g == 0) { tmem_ld_wait(first); tmem_ld(ta + CODE_NC / 2, second); }
          if (g == 2) { tmem_ld_wait(second); if (ch + 1 < n_chunks) tmem_ld(ta + (uint32_t)col_step, first); }
          float v[8];
          uint32_t c[8];
          dequant<MODE, TAPS, false, 8>(br, N, m, row_ok, n_tile0 + col + 8 * g, col + 8 * g, cc, (g < 2 ? first : second) + 8 * (g & 1), v);
          dist[g] = 0.0f;
#pragma unroll
          for (int i = 0; i < 8; i += 2) {
            if (MODE == EPI_FC1) gelu_pattern2(make_float2(v[i], v[i + 1]), inv_scale, magic_zp, dist[g], c[i], c[i + 1]);
            else quant_pattern2(make_float2(v[i], v[i + 1]), inv_scale, neg_zero, c[i], c[i + 1]);
          }
          w[2 * g] = sat_pack4<SH>(c[0], c[1], c[2], c[3], zbias << SH);
          w[2 * g + 1] = sat_pack4<SH>(c[4], c[5], c[6], c[7], zbias << SH);
        }
        // Eight columns again by the contract's own operations: where some value of the warp is too close to a rounding boundary
        // (FC1, a sixth of the chunks at A8), and all of them where the patterns above do not hold
        const bool near = MODE == EPI_FC1 && fmaxf(fmaxf(dist[0], dist[1]), fmaxf(dist[2], dist[3])) >= thr;
        if (!in_range || (MODE == EPI_FC1 && __any_sync(0xffffffffu, near))) {
#pragma unroll 1
          for (int g = 0; g < 4; ++g) {
            const float d = g == 0 ? dist[0] : g == 1 ? dist[1] : g == 2 ? dist[2] : dist[3];
            if (in_range && !__any_sync(0xffffffffu, d >= thr)) continue;
            int32_t again[8];
            tmem_ld(ta + (uint32_t)(8 * g), again);
            tmem_ld_wait(again);
            float v[8];
            uint32_t c[8];
            dequant<MODE, TAPS, false, 8>(br, N, m, row_ok, n_tile0 + col + 8 * g, col + 8 * g, cc, again, v);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              const float2 x = make_float2(v[i], v[i + 1]);
              quant_magic2(MODE == EPI_FC1 ? gelu_f2(x) : x, inv_scale, -zpf, eb.qmaxf - zpf, c[i], c[i + 1]);
            }
            const uint32_t zb = (uint32_t)q.zp - kMagicBits;
            const uint32_t w0 = sat_pack4<SH>(c[0], c[1], c[2], c[3], zb << SH), w1 = sat_pack4<SH>(c[4], c[5], c[6], c[7], zb << SH);
            w[0] = g == 0 ? w0 : w[0]; w[1] = g == 0 ? w1 : w[1];
            w[2] = g == 1 ? w0 : w[2]; w[3] = g == 1 ? w1 : w[3];
            w[4] = g == 2 ? w0 : w[4]; w[5] = g == 2 ? w1 : w[5];
            w[6] = g == 3 ? w0 : w[6]; w[7] = g == 3 ? w1 : w[7];
          }
        }
        if (row_ok) store_sat32(out_ptr + ch * out_step, w, bits, cbits);
      }
    };
    if (bits == 8) walk(std::integral_constant<int, 8>{});
    else if (bits == 4) walk(std::integral_constant<int, 4>{});
    else walk(std::integral_constant<int, 2>{});
    return true;
  }

  // ---- binary32 outputs (proj: x1 = x_window + out; fc2: y = x1 + out scattered to the token's own position;
  //      merge: out).  The raw sums of a 16-column chunk are transposed through shared memory so that global accesses are
  //      64-byte runs (4 lanes per row, 8 rows per instruction), and a lane then needs the constants of 4 columns only:
  //      these launches are bound by the load/store pipe, and constants read per row and column were a third of its work.
  //      (32-column chunks with 128-byte runs: 86 against 68 us for a proj of 296 450 rows of 128 channels -- half the
  //      chunks in flight per warp, and the addresses of eight rows spill.) ----
  const int cj = lane & 3, rsub = lane >> 2;
  long src_mine = -1;
  if (MODE != EPI_MERGE && row_ok) src_mine = eb.rowsrc[m];
  // this lane's four (row, 16-byte piece) positions of the warp's first chunk: residual source and output, NULL: none
  const float* res_ptr[4];
  float* dst_ptr[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 8 * i + rsub;
    const long mr = row0 + r;
    const long s = __shfl_sync(0xffffffffu, src_mine, r);
    const bool ok = mr < eb.M;
    long res_row, dst_row;               // row offsets (in elements), -1: none
    if (MODE == EPI_PROJ)     { res_row = (ok && s >= 0) ? s * N : -1;  dst_row = ok ? mr * N : -1; }
    else if (MODE == EPI_FC2) { res_row = (ok && s >= 0) ? mr * N : -1; dst_row = (ok && s >= 0) ? s * N : -1; }
    else                      { res_row = -1;                            dst_row = ok ? mr * N : -1; }
    res_ptr[i] = (MODE != EPI_MERGE && res_row >= 0) ? eb.res + res_row + n_first + 4 * cj : nullptr;
    dst_ptr[i] = dst_row >= 0 ? eb.out_f + dst_row + n_first + 4 * cj : nullptr;
  }
  // The residual rows come into shared memory by asynchronous copies, RES_SLOTS chunks ahead of their use: the copies
  // of a whole tile are in flight while the accumulator is still being computed, and they cost no registers.
  // Slot ch % RES_SLOTS holds chunk ch in the layout of the transposition tile (row r, 16-byte piece j at piece
  // j ^ ((r >> 1) & 3)).  One commit group per chunk, also when there is nothing left to fetch, so that "all but the
  // newest RES_SLOTS - 1 groups are complete" always covers the chunk about to be used.
  auto fetch = [&](int ch) {
    if (MODE != EPI_MERGE && ch < n_chunks) {
      float* slot = res_ring + (ch % RES_SLOTS) * EPI_STAGE_FLOATS;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + rsub;
        float* dst = slot + r * F32_NC + 4 * (cj ^ ((r >> 1) & 3));
        if (res_ptr[i]) cp_async16(dst, res_ptr[i] + ch * col_step);
        else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);   // a pad token's residual input is zero
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
    int32_t acc[F32_NC];
    if (n_chunks > 0) tmem_ld(taddr, acc);
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ++ch) {
      const int lc = c_first * F32_NC + ch * col_step + 4 * cj;       // this lane's first column within the tile
      tmem_ld_wait(acc);
      // row `lane`, logical 16-byte piece j is stored at piece j ^ ((lane >> 1) & 3): conflict-free both ways
#pragma unroll
      for (int j = 0; j < 4; ++j)
        *reinterpret_cast<int4*>(stage + lane * F32_NC + 4 * (j ^ ((lane >> 1) & 3))) =
            make_int4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
      // the TMEM load of the next chunk is in flight while this chunk is finished
      if (ch + 1 < n_chunks) tmem_ld(taddr + (uint32_t)((ch + 1) * col_step), acc);
      const int4 p4 = *reinterpret_cast<const int4*>(cc.pre + lc);
      const float4 m4 = *reinterpret_cast<const float4*>(cc.mult + lc);
      float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (MODE != EPI_MERGE) b4 = *reinterpret_cast<const float4*>(cc.bias + lc);
      if (MODE != EPI_MERGE) cp_async_wait<RES_SLOTS - 1>();     // this lane's copies of chunk ch have landed
      __syncwarp();
      const float* slot = res_ring + (ch % RES_SLOTS) * EPI_STAGE_FLOATS;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + rsub;
        const int off = r * F32_NC + 4 * (cj ^ ((r >> 1) & 3));
        const int4 a = *reinterpret_cast<const int4*>(stage + off);
        if (TAPS && br.tap_acc && row0 + r < eb.M) {
          int32_t* tp = br.tap_acc + (row0 + r) * N + n_tile0 + lc;
          tp[0] = a.x + p4.x - (int32_t)kMagicBits; tp[1] = a.y + p4.y - (int32_t)kMagicBits;
          tp[2] = a.z + p4.z - (int32_t)kMagicBits; tp[3] = a.w + p4.w - (int32_t)kMagicBits;
        }
        if (!dst_ptr[i]) continue;
        const float2 f0 = acc_to_float2<NARROW>(a.x + p4.x, a.y + p4.y), f1 = acc_to_float2<NARROW>(a.z + p4.z, a.w + p4.w);
        float2 lo, hi;
        if (MODE == EPI_MERGE) {
          lo = __fmul2_rn(f0, make_float2(m4.x, m4.y)); hi = __fmul2_rn(f1, make_float2(m4.z, m4.w));
        } else {
          const float4 rr = *reinterpret_cast<const float4*>(slot + off);
          lo = __fadd2_rn(make_float2(rr.x, rr.y), __ffma2_rn(f0, make_float2(m4.x, m4.y), make_float2(b4.x, b4.y)));
          hi = __fadd2_rn(make_float2(rr.z, rr.w), __ffma2_rn(f1, make_float2(m4.z, m4.w), make_float2(b4.z, b4.w)));
        }
        *reinterpret_cast<float4*>(dst_ptr[i] + ch * col_step) = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
      __syncwarp();
      if (MODE != EPI_MERGE) fetch(ch + RES_SLOTS);              // the slot just read is free again
    }
  };
  if (narrow) walk(std::true_type{}); else walk(std::false_type{});
  if (MODE != EPI_MERGE) cp_async_wait<0>();                   // nothing of this tile is left in flight
  return true;
}

}  // namespace mixaq
