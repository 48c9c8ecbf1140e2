// Integer GEMM on the 5th-generation tensor cores (tcgen05.mma kind::i8, u8 activations x s8 weights,
// int32 accumulators in tensor memory) with the fused epilogues of gemm_epilogue.cuh.
//
//   D[128 x BN] (TMEM) = A[128 x K] (u8, K-major, shared memory) * W[BN x K]^T (s8, K-major, shared memory)
//
// Persistent, warp-specialised: one CTA per SM walks over the output tiles t = blockIdx.x, + gridDim.x, ...
//   warp 0      TMA producer: weight tile and (8-bit branches) activation tile of every k-block into a ring of
//               128-byte-swizzled K-major stages (cp.async.bulk.tensor, no multicast), completion on mbarriers;
//   warp 1      MMA issuer: one elected lane feeds the tensor core; the tiles take turns on up to six TMEM accumulators, so
//               that the epilogue of a tile overlaps the loads and MMAs of the following ones;
//   warps 4-7   unpack producers for 4-bit / 2-bit branches: the bit-packed rows of the k-block arrive by TMA in a
//               staging slot of the stage; these warps expand them to one code per byte, shared to shared, into
//               the swizzled layout (rows whose byte pitch is no multiple of 16 cannot be described to the TMA
//               unit and are read with plain loads instead);
//   then        epilogue (12 warps for the code outputs, 8 for the binary32 outputs): tcgen05.ld (a quad of lanes
//               per row, 16 columns per load) + the fused epilogue of the mode.
// Every wait on an mbarrier is bounded; on expiry the CTA raises the status word, then waits (bounded again) for the
// copies it has issued to land and for the MMAs it has issued to retire, frees its tensor memory and returns.
#include "tc_ptx.cuh"
#include "gemm_epilogue.cuh"

namespace mixaq {

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = 148;
  }
  return n;
}

namespace {

constexpr int BM = 128;            // rows per tile = TMEM lanes
constexpr int BK = 128;            // codes (bytes) per row and stage = one 128-byte swizzle row
constexpr int UMMA_K = 32;         // codes per tcgen05.mma kind::i8
constexpr int A_STAGE_BYTES = BM * BK;
// warps 4..7 expand sub-byte codes (two warps left the long-K main loops of 4-bit tiles waiting for the expansion;
// eight cost more registers than they return)
constexpr int UNPACK_WARPS = 4;
// Epilogue warps.  Code outputs: 12 (16 with fewer registers are no faster at any size).  Binary32 outputs: 8, which are as fast as 12
// for few row tiles and up to 16 % faster for many (best tiling of either, fc2 of 768 channels at 7 x 7: 6.7 against 6.8 us, at 25 x 42
// 8.1 against 8.5, at 4 x 32 x 32 15.3 against 18.2).
constexpr int F32_WARPS = 8, CODE_WARPS = 12;
// Warpgroups: TMA, MMA and TMEM set-up; unpack, only in launches with bit-packed rows; epilogue
constexpr int FIRST_UNPACK_WARP = 4;
__host__ __device__ constexpr int first_epi_warp(bool packed) { return FIRST_UNPACK_WARP + (packed ? UNPACK_WARPS : 0); }
__host__ __device__ constexpr int num_threads(int warps, bool packed) { return 32 * (first_epi_warp(packed) + warps); }
// Registers.  With 12 epilogue warps a block is launched with what its threads divide the file into (a scheduler's 16 384 among its
// warps: 128 a thread, 96 with the unpack warps too); the side warpgroups give back all but SIDE_REGS and the epilogue warps take
// them: 4 x 72 + 12 x 136 of 16 x 128, 8 x 72 + 12 x 112 of 20 x 96.  gemm_init checks that the shares fit
// into what the compiled kernels are launched with.  (No instance spills; with 56 for the side warps six did.)
constexpr int SIDE_REGS = 72;
__host__ __device__ constexpr int epi_regs(int warps, bool packed) { return warps != 12 ? 0 : packed ? 112 : 136; }    // 0: no exchange
constexpr int MAX_BN = 256;
__host__ __device__ constexpr bool code_mode(int mode) { return mode == EPI_QKV || mode == EPI_FC1; }
__host__ __device__ constexpr int lane_cols(int mode) { return (code_mode(mode) ? CODE_NC : F32_NC) / 4; }   // columns of a lane in a chunk
constexpr int MAX_RING = 6;
constexpr int TMEM_COLS = 512;                 // one CTA per SM: it takes all of the tensor memory
constexpr int MAX_ACC = 6;                     // accumulators in it, as far as the tile width allows

struct TcParams {
  GemmArgs g;
  int tiles_m0, tiles_m;   // 128-row tiles of the first (high) branch, of both
  int n_tiles, BN, k_blocks, ring;
  int step_m, step_n;      // a CTA walks over the tiles (row tile major) gridDim.x at a time: the step as (row, column) tiles
  // The epilogue warps of a lane quarter form `groups` groups; group g takes the CTA's tiles g, g + groups, ... (gstep: that
  // stride as (row, column) tiles), and the `split` warps of a group deal a tile's chunks among themselves.
  int groups, split, gstep_m, gstep_n;
  int const_cols;          // columns whose constants a CTA keeps in shared memory: BN where it stays on one column tile, else N
  int last_step;           // number of the CTA's last tile is the largest blockIdx.x + i * gridDim.x <= last_step
  int n_acc, acc_stride;   // accumulators in tensor memory and the columns between them
  int packed_bytes;        // bytes of the packed staging slot of a stage (0: no branch stages packed rows by TMA)
  int res_bytes;           // bytes of the residual rings (proj, fc2: RES_SLOTS chunks per epilogue warp; else 0)
  int tma_packed[2];       // branch i stages its bit-packed rows by TMA (tmA_i then describes the packed matrix)
  int* status;
};

// shared-memory carve-up (offsets from the 1024-byte aligned base)
struct SmemLayout {
  int stage_bytes, ring_bytes, consts_off, res_off, bars_off, total;
};
constexpr int NUM_BARS = 4 * MAX_RING + 2 * MAX_ACC + 2;        // full, empty, raw, unpacked; accumulator full, empty; constants, drain
__host__ __device__ inline SmemLayout smem_layout(int BN, int ring, int packed_bytes, int res_bytes, int const_cols) {
  SmemLayout L;
  L.stage_bytes = A_STAGE_BYTES + BN * BK + packed_bytes;
  L.ring_bytes = ring * L.stage_bytes;
  L.consts_off = L.ring_bytes;                                  // (pre, mult, bias) of const_cols columns
  L.res_off = L.consts_off + 3 * const_cols * 4;                // residual rings of proj and fc2
  L.bars_off = L.res_off + res_bytes;
  L.total = L.bars_off + NUM_BARS * 8 + 16;                     // then TMEM base, abort flag, constants-out-of-range flags
  return L;
}

// The tiles of a CTA, without a division per tile: tile number blockIdx.x, + gridDim.x, ..., row tile major.  The high
// branch's row tiles come first, so every role runs one loop per branch and keeps the branch's constants in registers.
struct TileWalk {
  int mt, nt;
  __device__ __forceinline__ explicit TileWalk(const TcParams& p) : mt((int)blockIdx.x / p.n_tiles), nt((int)blockIdx.x - mt * p.n_tiles) {}
  __device__ __forceinline__ void advance(int dm, int dn, int n_tiles) {
    mt += dm; nt += dn;
    if (nt >= n_tiles) { nt -= n_tiles; ++mt; }
  }
  __device__ __forceinline__ void next(const TcParams& p) { advance(p.step_m, p.step_n, p.n_tiles); }
};
// Position in the ring of stages (or of accumulators): slot and parity of the current pass.
struct RingPos {
  int slot = 0; uint32_t pass = 0;
  __device__ __forceinline__ void next(int n) { if (++slot == n) { slot = 0; pass ^= 1u; } }
};

// TAPS: the accumulator tap is compiled in only for calls that ask for it (and where always_taps says so)
//
// The loops of the TMA and the MMA warp bound a tile as much as the epilogue does, so they hold no division, and the whole warp
// walks through them with one elected lane issuing: in code that a single lane runs, an MMA of up to 64 columns takes 63 cycles to
// issue, elected in a converged warp 45 to 51.
template <int MODE, bool TAPS, int EW, bool PACKED>
__global__ void __launch_bounds__(num_threads(EW, PACKED), 1)
k_gemm_tc(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmA1,
          const __grid_constant__ CUtensorMap tmB, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;                 // swizzled tiles need 1024-byte alignment
  uint8_t* smem = smem_raw + (base - raw);
  const SmemLayout L = smem_layout(p.BN, p.ring, p.packed_bytes, p.res_bytes, p.const_cols);
  const int stage_bytes = L.stage_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars_off);
  const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8u * MAX_RING, bar_raw = bar_empty + 8u * MAX_RING;
  const uint32_t bar_unp = bar_raw + 8u * MAX_RING, bar_tfull = bar_unp + 8u * MAX_RING;
  const uint32_t bar_tempty = bar_tfull + 8u * MAX_ACC, bar_consts = bar_tempty + 8u * MAX_ACC, bar_drain = bar_consts + 8u;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  int* beyond_flags = reinterpret_cast<int*>(tmem_holder + 2);       // bit 0: some sum may reach 2^22; bit 1: some pattern its range
  // TMA warp: fills of ring stages so far; stages that held packed rows and the phase of the last ones (bit s of each).  Read by
  // the give-up path only.
  uint32_t fills = 0, raw_used = 0, raw_phase = 0;

  constexpr int LANE_COLS = lane_cols(MODE);
  constexpr int NUM_EPI_WARPS = EW, FIRST_EPI_WARP = first_epi_warp(PACKED);
  constexpr int NUM_UNPACK_WARPS = UNPACK_WARPS, NUM_UNPACK_THREADS = NUM_UNPACK_WARPS * 32;
  constexpr int UNPACK_ITEMS = BM * (BK / UMMA_K) / NUM_UNPACK_THREADS;   // (row, 32-code group) items per thread and stage
  // The warp number through a shuffle: the compiler then knows that it is the same in all lanes and that the roles' loops run
  // converged, and keeps addresses and descriptors in uniform registers (Swin-T 224 image / 800 x 1333: 393 / 788 us with
  // threadIdx.x >> 5, 371 / 758 so).
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

  // Every launch starts with a cold constant cache, and the roles below would miss on one parameter after the other
  // (1 800 cycles until the first copy was issued): the warps touch the lines of the parameter block side by side.
  {
    const int word = (warp * 16) % (int)(sizeof(TcParams) / 4);
    const int touched = reinterpret_cast<const int*>(&p)[word];
    asm volatile("" ::"r"(touched));
  }
  if (tid == 32) {
    // the descriptors are fetched while the barriers are set up
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA0) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA1) : "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < p.ring; ++s) {
      mbar_init(bar_full + 8u * s, 1u);                         // TMA thread; the operand bytes of the stage
      mbar_init(bar_empty + 8u * s, 1u);                        // tcgen05.commit
      mbar_init(bar_raw + 8u * s, 1u);                          // TMA thread (+ bytes): packed rows are there
      mbar_init(bar_unp + 8u * s, NUM_UNPACK_WARPS);            // unpack warps: the activation tile is expanded
    }
    for (int a = 0; a < p.n_acc; ++a) {
      mbar_init(bar_tfull + 8u * a, 1u);                        // tcgen05.commit of the tile's last MMA
      mbar_init(bar_tempty + 8u * a, 4u * (uint32_t)p.split);   // one arrival per epilogue warp of a group
    }
    mbar_init(bar_consts, NUM_EPI_WARPS);                       // constants of a branch: loaded / no longer in use
    *beyond_flags = 0;
    mbar_init(bar_drain, 1u);                                   // tcgen05.commit of the give-up path
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_holder)), "r"((uint32_t)TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_holder;
  griddep_launch();
  // Registers change hands by whole warpgroups, whose warps all execute the same instruction: it stands in front of the roles.
  if (epi_regs(EW, PACKED) > 0 && warp < FIRST_EPI_WARP) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SIDE_REGS));

  if (warp == 0) {
    // ---- TMA producer ----
    {
      const bool leader = elect_one();
      TileWalk w(p);
      RingPos rp;
      bool ok = true;
      const uint32_t b_bytes = (uint32_t)(p.BN * BK);
      bool waited = false;                                      // for the kernel that writes the activations (weights do not wait)
      const int k_blocks = p.k_blocks, ring = p.ring, BN = p.BN;
      for (int b = 0; b < 2 && ok; ++b) {
        const int m_first = b == 0 ? 0 : p.tiles_m0, m_end = b == 0 ? p.tiles_m0 : p.tiles_m;
        if (w.mt >= m_end) continue;
        const int abits = p.g.br[b].a_bits;
        const bool packed = PACKED && abits != 8, stage_packed = packed && p.tma_packed[b];
        const CUtensorMap* tmA = b == 0 ? &tmA0 : &tmA1;
        const uint32_t tx = b_bytes + (packed ? 0u : (uint32_t)A_STAGE_BYTES);
        const int pk_row = BK * abits / 8;                      // packed bytes per row and k-block
        for (; w.mt < m_end && ok; w.next(p)) {
          const int m_row = (w.mt - m_first) * BM, n_row = w.nt * BN;
          for (int kb = 0; kb < k_blocks; ++kb, rp.next(ring)) {
            const uint32_t o = 8u * (uint32_t)rp.slot;
            if (!mbar_wait_warp(bar_empty + o, rp.pass ^ 1u, abort_flag)) { ok = false; break; }    // (at once in the first pass)
            const uint32_t sa = base + (uint32_t)(rp.slot * stage_bytes), sb = sa + A_STAGE_BYTES;
            ++fills;
            if (leader) {
              mbar_arrive_expect_tx(bar_full + o, tx);
              tma_load_5d(sb, &tmB, kb * BK, n_row / (4 * LANE_COLS), bar_full + o);
            }
            if (!waited) { griddep_wait(); waited = true; }
            if (leader && !packed) tma_load_2d(sa, tmA, kb * BK, m_row, bar_full + o);
            if (packed) {
              const uint32_t bit = 1u << rp.slot;
              raw_phase = (raw_used & bit) ? raw_phase ^ bit : raw_phase & ~bit;
              raw_used |= bit;
              if (leader && stage_packed) {
                mbar_arrive_expect_tx(bar_raw + o, (uint32_t)(pk_row * BM));
                tma_load_2d(sb + b_bytes, tmA, kb * pk_row, m_row, bar_raw + o);
              } else if (leader) {
                mbar_arrive(bar_raw + o);
              }
            }
            __syncwarp();
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----
    {
      const bool leader = elect_one();
      const uint32_t idesc = (2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      const uint64_t adesc0 = smem_desc_sw128(base), bdesc0 = smem_desc_sw128(base + A_STAGE_BYTES);
      const uint32_t stage16 = (uint32_t)stage_bytes >> 4;      // stage pitch in descriptor units
      const int k_blocks = p.k_blocks, ring = p.ring, n_acc = p.n_acc;
      const int last_steps = (p.g.K - (k_blocks - 1) * BK) / UMMA_K;      // MMAs of the last k-block (4 in the others)
      TileWalk w(p);
      RingPos rp, ap;
      uint32_t unp_next = 0;                                    // bit s: parity of stage s' next expansion
      bool ok = true;
      for (int b = 0; b < 2 && ok; ++b) {
        const int m_end = b == 0 ? p.tiles_m0 : p.tiles_m;
        if (w.mt >= m_end) continue;
        const bool packed = PACKED && p.g.br[b].a_bits != 8;
        for (; w.mt < m_end && ok; w.next(p), ap.next(n_acc)) {
          // wait until the epilogue has drained this accumulator's previous use (at once in the first pass)
          if (!mbar_wait_warp(bar_tempty + 8u * ap.slot, ap.pass ^ 1u, abort_flag)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d_tmem = tmem_base + (uint32_t)(ap.slot * p.acc_stride);
          for (int kb = 0; kb < k_blocks; ++kb, rp.next(ring)) {
            const uint32_t o = 8u * (uint32_t)rp.slot;
            if (!mbar_wait_warp(bar_full + o, rp.pass, abort_flag)) { ok = false; break; }
            if (packed) {
              if (!mbar_wait_warp(bar_unp + o, (unp_next >> rp.slot) & 1u, abort_flag)) { ok = false; break; }
              unp_next ^= 1u << rp.slot;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t so = (uint64_t)((uint32_t)rp.slot * stage16);
            const uint64_t adesc = adesc0 + so, bdesc = bdesc0 + so;
            const int steps = kb == k_blocks - 1 ? last_steps : BK / UMMA_K;
            if (leader) {
#pragma unroll
              for (int kk = 0; kk < BK / UMMA_K; ++kk)
                if (kk < steps)
                  mma_i8(d_tmem, adesc + (uint64_t)(kk * (UMMA_K >> 4)), bdesc + (uint64_t)(kk * (UMMA_K >> 4)), idesc,
                         kk > 0 ? 1u : (uint32_t)(kb > 0));
              mma_commit(bar_empty + o);             // frees the ring slot when these MMAs have read it
              if (kb == k_blocks - 1) mma_commit(bar_tfull + 8u * ap.slot);    // accumulator complete
            }
            __syncwarp();
          }
        }
      }
    }
  } else if (warp < FIRST_UNPACK_WARP) {
    // (warps 2 and 3 fill up the warpgroup)
  } else if (PACKED && warp < FIRST_EPI_WARP) {
    // ---- unpack producers: bit-packed rows -> one code per byte, written in the swizzled layout ----
    const int ptid = tid - 32 * FIRST_UNPACK_WARP;   // 0 .. NUM_UNPACK_THREADS-1
    TileWalk w(p);
    int slot = 0;
    uint32_t raw_next = 0;                       // bit s: parity of stage s' next packed fill
    bool ok = true;
    for (int b = 0; b < 2 && ok; ++b) {
      const int m_first = b == 0 ? 0 : p.tiles_m0, m_end = b == 0 ? p.tiles_m0 : p.tiles_m;
      if (w.mt >= m_end) continue;
      const int abits = p.g.br[b].a_bits;
      if (abits == 8) {                          // nothing to expand: skip the stages of these tiles
        int tiles = 0;
        for (; w.mt < m_end; w.next(p)) ++tiles;
        slot = (slot + tiles * p.k_blocks) % p.ring;
        continue;
      }
      const bool staged = p.tma_packed[b];
      if (!staged) griddep_wait();               // these warps read the rows themselves
      const uint8_t* a = p.g.br[b].a;
      const int M = p.g.br[b].M, K = p.g.K;
      const long row_bytes = (long)K * abits / 8;
      const int grp_bytes = UMMA_K * abits / 8;                 // packed bytes of one 32-code group
      for (; w.mt < m_end && ok; w.next(p)) {
        const long m0 = (long)(w.mt - m_first) * BM;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          // the TMA thread arrives on raw[s] once it owns the stage (and, when staged, the packed bytes have landed)
          if (!mbar_wait_warp(bar_raw + 8u * slot, (raw_next >> slot) & 1u, abort_flag)) { ok = false; break; }
          raw_next ^= 1u << slot;
          uint8_t* sa = smem + (size_t)slot * stage_bytes;
          const uint8_t* sp = sa + A_STAGE_BYTES + p.BN * BK;
          const int kgroups = min(BK, K - kb * BK) / UMMA_K;
          // item i of this thread: row r = item / 4, 32-code group kg = item % 4, item = ptid + NUM_UNPACK_THREADS * i
#pragma unroll
          for (int i = 0; i < UNPACK_ITEMS; ++i) {
            const int item = ptid + NUM_UNPACK_THREADS * i;
            const int r = item >> 2, kg = item & 3;
            uint32_t c[8];
            bool have = true;
            if (staged) {
              // rows and columns outside the matrix were zero-filled by the TMA unit
              load_codes_32(sp + item * grp_bytes, abits, c);
            } else {
              have = kg < kgroups && m0 + r < M;
              if (have) load_codes_32(a + (m0 + r) * row_bytes + (long)(kb * BK + kg * UMMA_K) * abits / 8, abits, c);
            }
            if (have) {
              uint8_t* rowp = sa + (r >> 3) * 1024 + (r & 7) * 128;
              const int c0 = (2 * kg) ^ (r & 7), c1 = (2 * kg + 1) ^ (r & 7);
              *reinterpret_cast<uint4*>(rowp + c0 * 16) = make_uint4(c[0], c[1], c[2], c[3]);
              *reinterpret_cast<uint4*>(rowp + c1 * 16) = make_uint4(c[4], c[5], c[6], c[7]);
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // make the writes visible to the MMA proxy
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_unp + 8u * slot);
          if (++slot == p.ring) slot = 0;
        }
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue warps: warp e reads TMEM lanes 32*(e%4).. of its group's tiles, every split-th chunk ----
    if (epi_regs(EW, PACKED) > 0) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(epi_regs(EW, PACKED) > 0 ? epi_regs(EW, PACKED) : 24));
    const int e = warp - FIRST_EPI_WARP, q = warp & 3;         // any 4 consecutive warps cover the 4 lane quarters
    const int split = p.split, groups = p.groups, group = (e >> 2) / split, sub = (e >> 2) - group * split;
    float* res_ring = reinterpret_cast<float*>(smem + L.res_off) + e * RES_SLOTS * EPI_CHUNK_FLOATS;
    int32_t* c_pre = reinterpret_cast<int32_t*>(smem + L.consts_off);
    float* c_mult = reinterpret_cast<float*>(c_pre + p.const_cols);
    float* c_bias = c_mult + p.const_cols;
    const int c_total = p.BN / (code_mode(MODE) ? CODE_NC : F32_NC);   // BN is a multiple of 32
    const uint32_t tmem_q = tmem_base + ((uint32_t)(q * 32) << 16);
    TileWalk w(p);
    for (int g = 0; g < group; ++g) w.next(p);
    auto step = [&](TileWalk& t) { t.advance(p.gstep_m, p.gstep_n, p.n_tiles); };
    const int first_mt = (int)blockIdx.x / p.n_tiles;
    int acc = group;
    uint32_t acc_pass = 0;
    bool ok = true;
    // The per-column constants of a branch, for all columns the CTA can meet, are loaded once by all epilogue warps (a tile
    // that fetched its own waited 600 cycles per chunk for the dependent loads).  The waits are the bounded mbarrier waits.
    const int const_first = p.const_cols == p.BN ? (int)(blockIdx.x % (unsigned)p.n_tiles) * p.BN : 0;
    const int last_mt = (int)(blockIdx.x + (unsigned)(p.last_step - (int)blockIdx.x) / gridDim.x * gridDim.x) / p.n_tiles;
    uint32_t consts_pass = 0;
    bool waited = false;
    bool narrow = false, in_range = false;                     // sums and patterns of these columns stay in range
    auto all_warps = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_consts);
      const bool done = mbar_wait_warp(bar_consts, consts_pass, abort_flag);
      consts_pass ^= 1u;
      return done;
    };
    for (int b = 0; b < 2 && ok; ++b) {
      const int m_first = b == 0 ? 0 : p.tiles_m0, m_end = b == 0 ? p.tiles_m0 : p.tiles_m;
      if (first_mt >= m_end || last_mt < m_first) continue;     // the CTA has no tile of this branch
      const GemmBranch& br = p.g.br[b];
      const EpiBranch eb(br, p.g.N);
      if (b == 1 && first_mt < p.tiles_m0 && !all_warps()) { ok = false; break; }      // everybody is done with the first branch's
      int beyond = 0;
      for (int i = e * 32 + lane; i < p.const_cols; i += NUM_EPI_WARPS * 32) {
        const int n = const_first + i;
        const float bias = MODE != EPI_MERGE ? __ldg(br.bias + n) : 0.0f, bound = __ldg(br.bound + n);
        c_pre[i] = __ldg(br.pre + n);
        c_mult[i] = __ldg(br.mult + n);
        c_bias[i] = bias;
        const float inv = !code_mode(MODE) ? 0.0f : MODE == EPI_FC1 || n < p.g.C ? br.q0.inv_scale : (n < 2 * p.g.C ? br.q1.inv_scale : br.q2.inv_scale);
        beyond |= bound < 0.0f ? 1 : 0;
        beyond |= code_mode(MODE) && !((fabsf(bound) + fabsf(bias)) * inv < kPatternRange) ? 2 : 0;
      }
      if (beyond) atomicOr(beyond_flags, beyond);               // (a branch out of range takes the next one along: it is only slower)
      if (!all_warps()) { ok = false; break; }
      if (!waited) { griddep_wait(); waited = true; }           // residuals, row indices and outputs belong to earlier kernels
      const int flags = *reinterpret_cast<volatile int*>(beyond_flags);
      narrow = (flags & 1) == 0; in_range = (flags & 2) == 0;
      for (; w.mt < m_end; step(w)) {
        const int n_tile0 = w.nt * p.BN;
        const int c0 = n_tile0 - const_first;
        const ColConsts cc = {c_pre + c0, c_mult + c0, c_bias + c0};
        const long row0 = (long)(w.mt - m_first) * BM + q * 32;
        auto acc_ready = [&]() -> bool {
          if (!mbar_wait_warp<true>(bar_tfull + 8u * acc, acc_pass, abort_flag)) return false;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          return true;
        };
        if (!epilogue_warp_tile<MODE, TAPS>(br, eb, p.g.N, p.g.C, row0, lane, n_tile0, sub, split, c_total, cc,
                                            tmem_q + (uint32_t)(acc * p.acc_stride), narrow, in_range, p.g.neg_zero,
                                            acc_ready, res_ring)) { ok = false; break; }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty + 8u * acc);
        acc += groups;
        if (acc >= p.n_acc) { acc = group; acc_pass ^= 1u; }
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag) {
    // A wait ran out.  Before the CTA may exit, the copies already issued must have landed in its shared memory and
    // the MMAs already issued must have retired.  (1) The lane that issued the MMAs commits them to a barrier of their
    // own (a commit covers what its own thread has issued; elect.sync names the same lane of a full warp every time).
    // (2) A thread of the TMA warp waits, bounded, for the phase of the last fill of every stage, on the full barrier and on
    // the packed-rows barrier (both complete by the copies alone), and for that commit.
    if (warp == 1 && elect_one()) mma_commit(bar_drain);
    __syncthreads();
    if (tid == 0) {
      atomicExch(p.status, 1);
      auto drain = [](uint32_t bar, uint32_t parity) {
        for (uint32_t it = 0; it < (1u << 20); ++it) if (mbar_try_wait(bar, parity)) return;
      };
      for (uint32_t s = 0; s < (uint32_t)p.ring; ++s) {
        if (fills > s) drain(bar_full + 8u * s, (fills - 1u - s) / (uint32_t)p.ring & 1u);      // pass of the stage's last fill
        if (raw_used >> s & 1u) drain(bar_raw + 8u * s, raw_phase >> s & 1u);
      }
      drain(bar_drain, 0u);
    }
    __syncthreads();
  }
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
  }
}

// ---- host side -------------------------------------------------------------------------------------
// Tile width and the epilogue's division of labour.  The width is a multiple of 32 that divides `unit` (N; for QKV the
// width C of a section, so that a tile has one quantizer), at most 256.  A tile takes `mma` to multiply and each of its warps `epi`
// to convert, `groups` tiles are converted at once while the next ones are multiplied, and the first tiles have nothing to hide
// behind.  A wide tile reads its rows fewer times and pays the fixed part of the epilogue once for more columns; narrow ones spread a
// small problem over the SMs.  The constants (microseconds, roughly) were fitted to the times of all widths and groups of the four GEMMs
// at 25 maps from 768 x 7 x 7 to 128 x 384 x 384, each taken together with the kernel behind it.  With the present kernels the choice
// is 2.2 % above the fastest on average, within 10 % at 96 of 100.
struct Tiling { int bn, n_acc, groups, split; };
Tiling pick_tiling(int mode, int unit, int N, int m_tiles, int k_blocks, int sms, int warps) {
  Tiling best = {0, 0, 0, 0};
  double best_cost = 0.0;
  const int per_quarter = warps / 4;
  const int chunk = code_mode(mode) ? CODE_NC : F32_NC;
  const double fixed = code_mode(mode) ? 1.14 : 4.77, per_32 = mode == EPI_QKV ? 0.183 : mode == EPI_FC1 ? 0.0775 : 0.147;
  for (int bn = 32; bn <= MAX_BN; bn += 32) {
    if (unit % bn) continue;
    const int fit = TMEM_COLS / bn < MAX_ACC ? TMEM_COLS / bn : MAX_ACC;
    const long tiles = (long)m_tiles * (N / bn), per_cta = (tiles + sms - 1) / sms;
    // a launch that leaves SMs idle has more of the L2 for each tile: width then costs less
    const double mma = k_blocks * (0.256 + 0.246 * (bn / 32) * (tiles < sms ? (double)tiles / sms : 1.0));
    for (int groups = 1; groups <= per_quarter && groups <= fit; ++groups) {
      if (per_quarter % groups) continue;
      const int n_acc = fit / groups * groups;                // a group keeps to its own accumulators
      const int split = per_quarter / groups;
      const double epi = (bn / chunk + split - 1) / split * (chunk / 32.0) * per_32 + fixed;
      const long rounds = (per_cta + groups - 1) / groups;
      const double first = per_cta < groups ? per_cta * mma : groups * mma;
      const double cost = fmax(first + rounds * epi, per_cta * mma + epi);
      if (!best.bn || cost <= best_cost) { best = {bn, n_acc, groups, split}; best_cost = cost; }
    }
  }
  return best;
}

// Bit-packed launches of a block are those of calls with taps, and of blocks whose hidden layer is too wide for byte codes in their
// workspace (see carve_bytes): they share the instance with the tap.  Patch merging packs its codes and has no tap.
__host__ __device__ constexpr bool always_taps(int mode, bool packed) { return packed && mode != EPI_MERGE; }

template <int MODE, int EW, bool PACKED>
bool launch_mode_as(const GemmArgs& g, int* status, cudaStream_t st) {
  TcParams p;
  p.g = g; p.status = status;
  p.g.neg_zero = -0.0f;
  const int t0 = (g.br[0].M + BM - 1) / BM, t1 = (g.br[1].M + BM - 1) / BM;
  if (t0 + t1 == 0) return true;
  if (g.N % 32 || g.K % UMMA_K) return false;
  const int sms = sm_count();
  p.tiles_m0 = t0; p.tiles_m = t0 + t1;
  p.k_blocks = (g.K + BK - 1) / BK;
  const Tiling tl = pick_tiling(MODE, MODE == EPI_QKV ? g.C : g.N, g.N, t0 + t1, p.k_blocks, sms, EW);
  if (tl.bn == 0) return false;
  p.BN = tl.bn; p.n_acc = tl.n_acc; p.groups = tl.groups; p.split = tl.split;
  p.n_tiles = g.N / p.BN;
  const int total_tiles = (t0 + t1) * p.n_tiles;
  // packed branches whose row pitch the TMA unit accepts (a multiple of 16 bytes) are staged by TMA
  p.packed_bytes = 0;
  for (int i = 0; i < 2; ++i) {
    const int bits = g.br[i].a_bits;
    p.tma_packed[i] = g.br[i].M > 0 && bits != 8 && ((long)g.K * bits / 8) % 16 == 0;
    if (p.tma_packed[i]) p.packed_bytes = BM * (BK / 2);        // room for the widest packed format (4 bit)
  }
  p.res_bytes = (g.mode == EPI_PROJ || g.mode == EPI_FC2) ? EW * RES_SLOTS * EPI_CHUNK_FLOATS * 4 : 0;
  p.acc_stride = p.BN;
  CUtensorMap mA[2], mB;
  memset(mA, 0, sizeof(mA));
  for (int i = 0; i < 2; ++i) {
    const GemmBranch& b = g.br[i];
    bool ok;
    if (b.M > 0 && b.a_bits == 8)
      ok = make_map(&mA[i], b.a, (uint64_t)b.M, (uint64_t)g.K, BM);
    else if (p.tma_packed[i])
      ok = make_map(&mA[i], b.a, (uint64_t)b.M, (uint64_t)g.K * b.a_bits / 8, BM, (uint32_t)(BK * b.a_bits / 8), false);
    else   // no rows, or rows read with plain loads: a valid map of the weights that is never used
      ok = make_map(&mA[i], g.w, (uint64_t)g.N, (uint64_t)g.K, (uint32_t)p.BN);
    if (!ok) return false;
  }
  if (!make_quad_map(&mB, g.w, (uint64_t)g.N, (uint64_t)g.K, (uint32_t)p.BN, 4 * lane_cols(MODE))) return false;
  // a grid that is a multiple of the number of column tiles keeps every CTA on one column tile (t mod n_tiles);
  // taken only where it does not cost a wave of tiles
  int grid = total_tiles < sms ? total_tiles : sms;
  if (grid > p.n_tiles && grid < total_tiles) {
    const int g2 = grid - grid % p.n_tiles;
    if ((total_tiles + g2 - 1) / g2 == (total_tiles + grid - 1) / grid) grid = g2;
  }
  p.step_m = grid / p.n_tiles; p.step_n = grid % p.n_tiles;
  p.gstep_m = grid * p.groups / p.n_tiles; p.gstep_n = grid * p.groups % p.n_tiles;
  p.const_cols = p.step_n == 0 || total_tiles == grid ? p.BN : g.N;
  p.last_step = total_tiles - 1;
  p.ring = MAX_RING;
  while (p.ring > 2 && smem_layout(p.BN, p.ring, p.packed_bytes, p.res_bytes, p.const_cols).total + 1024 > 220 * 1024) --p.ring;
  const size_t smem = (size_t)smem_layout(p.BN, p.ring, p.packed_bytes, p.res_bytes, p.const_cols).total + 1024 /*alignment slack*/;
  if (smem > 227 * 1024) return false;
  constexpr bool TAPS = MODE != EPI_MERGE;
  if (TAPS && (g.br[0].tap_acc || g.br[1].tap_acc))
    launch_pdl(k_gemm_tc<MODE, TAPS, EW, PACKED>, dim3(grid), num_threads(EW, PACKED), smem, st, mA[0], mA[1], mB, p);
  else
    launch_pdl(k_gemm_tc<MODE, always_taps(MODE, PACKED), EW, PACKED>, dim3(grid), num_threads(EW, PACKED), smem, st, mA[0], mA[1], mB, p);
  ++g_launches;
  return true;
}
template <int MODE, int EW>
bool launch_mode(const GemmArgs& g, int* status, cudaStream_t st) {
  const bool packed = (g.br[0].M > 0 && g.br[0].a_bits != 8) || (g.br[1].M > 0 && g.br[1].a_bits != 8);
  return packed ? launch_mode_as<MODE, EW, true>(g, status, st) : launch_mode_as<MODE, EW, false>(g, status, st);
}

}  // namespace

// The bounded wait of this file on a barrier that nothing ever signals: it has to run out, raise the status word and
// let the CTA return normally.  (One CTA, one thread; no copy and no tensor memory is involved.)
__global__ void k_wait_probe(int* status, uint32_t tries) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bool done = false;
    for (uint32_t it = 0; it < tries && !done; ++it) done = mbar_try_wait(smem_u32(&bar), 0);
    if (!done) atomicExch(status, 1);
  }
}

void launch_wait_probe(int* status, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(status, 4096u);    // a few thousand tries: well under a millisecond
  ++g_launches;
}

// Issue-rate microbenchmark of the tensor core: every CTA (one per SM) keeps a 128 x 128-byte A tile and a
// 256 x 128-byte B tile in shared memory and issues `groups` x 4 MMAs of 128 x 256 x 32 into one TMEM accumulator,
// then waits (bounded) for the commit.  KIND 0: kind::i8 (u8 x s8 -> s32), the path the GEMMs use.
// KIND 1: kind::f8f6f4 with E4M3 operands (-> f32); this is also the path that carries 4-bit and 6-bit operand
// formats on sm_100a (in 8-bit shared-memory containers), so its rate bounds what a narrower operand type could give.
// KIND 2: kind::mxf4 (E2M1 operands packed two per byte, one UE8M0 scale per 32 values, -> f32): 128 x 256 x 64 per
// instruction from the same 32 bytes per row, the only narrower path with a higher nominal rate.
template <int KIND>
__global__ void __launch_bounds__(128, 1) k_mma_peak(int groups, unsigned long long* ns_out, int* status) {
  constexpr uint32_t PEAK_TMEM_COLS = KIND == 2 ? 512u : 256u;   // KIND 2 keeps its scale factors behind the accumulator
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + A_STAGE_BYTES + MAX_BN * BK);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < (A_STAGE_BYTES + MAX_BN * BK) / 4; i += blockDim.x)
    reinterpret_cast<uint32_t*>(smem)[i] = ((uint32_t)(i * 37 + 11) * 0x01010101u) & 0x3E3E3E3Eu;   // finite in E4M3 too
  if (tid == 0) { mbar_init(smem_u32(bar), 1u); asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(PEAK_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_holder;
  if (tid == 0) {
    // instruction descriptor: D format (s32 = 2 / f32 = 1) at bit 4, A format at 7, B format at 10, N/8 at 17, M/16 at 24
    // (block-scaled kinds: no D format field; A and B format 1 = E2M1 at bits 7 and 10, scale format 1 = UE8M0 at bit 23)
    const uint32_t idesc = KIND == 0 ? ((2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(MAX_BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24))
                         : KIND == 1 ? ((1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(MAX_BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24))
                                     : ((1u << 7) | (1u << 10) | ((uint32_t)(MAX_BN >> 3) << 17) | (1u << 23) | ((uint32_t)(BM >> 4) << 24));
    // KIND 2: the scale factors of A and B sit in tensor memory behind the accumulator (columns 256.., 264..); their
    // contents are whatever the allocation holds -- the products are meaningless, only the issue rate is measured
    const uint32_t sfa = tmem_base + 256u, sfb = tmem_base + 264u;
    const uint64_t adesc = smem_desc_sw128(base), bdesc = smem_desc_sw128(base + A_STAGE_BYTES);
    unsigned long long t0, t1;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int g = 0; g < groups; ++g)
      for (int kk = 0; kk < BK / UMMA_K; ++kk) {
        const uint32_t accumulate = (g > 0 || kk > 0) ? 1u : 0u;
        if (KIND == 0) {
          mma_i8(tmem_base, adesc + (uint64_t)(kk * (UMMA_K >> 4)), bdesc + (uint64_t)(kk * (UMMA_K >> 4)), idesc, accumulate);
        } else if (KIND == 2) {
          // 32 bytes of a row are 64 E2M1 values: one MMA of 128 x 256 x 64 with one UE8M0 scale per 32 values
          asm volatile(
              "{\n\t.reg .pred p;\n\t"
              "setp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
              ::"r"(tmem_base), "l"(adesc + (uint64_t)(kk * (UMMA_K >> 4))), "l"(bdesc + (uint64_t)(kk * (UMMA_K >> 4))),
                "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
        } else {
          asm volatile(
              "{\n\t.reg .pred p;\n\t"
              "setp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
              ::"r"(tmem_base), "l"(adesc + (uint64_t)(kk * (UMMA_K >> 4))), "l"(bdesc + (uint64_t)(kk * (UMMA_K >> 4))),
                "r"(idesc), "r"(accumulate) : "memory");
        }
      }
    mma_commit(smem_u32(bar));
    bool done = false;
    for (uint32_t it = 0; it < MAX_POLLS && !done; ++it) done = mbar_try_wait(smem_u32(bar), 0);
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
    if (!done) atomicExch(status, 1);
    ns_out[blockIdx.x] = t1 - t0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(PEAK_TMEM_COLS) : "memory");
}

// ns_out: one entry per SM (device memory).  Returns the grid size, 0 on failure.
int launch_mma_peak(int kind, int groups, unsigned long long* ns_out, int* status, cudaStream_t st) {
  const int sms = sm_count();
  const size_t smem = A_STAGE_BYTES + MAX_BN * BK + 1024 + 64;
  if (kind == 0) {
    if (cudaFuncSetAttribute(k_mma_peak<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    k_mma_peak<0><<<sms, 128, smem, st>>>(groups, ns_out, status);
  } else if (kind == 1) {
    if (cudaFuncSetAttribute(k_mma_peak<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    k_mma_peak<1><<<sms, 128, smem, st>>>(groups, ns_out, status);
  } else {
    if (cudaFuncSetAttribute(k_mma_peak<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    k_mma_peak<2><<<sms, 128, smem, st>>>(groups, ns_out, status);
  }
  ++g_launches;
  return sms;
}

// One-time set-up per device context (kept out of the launch path so that launches can be stream-captured):
// opt-in to large dynamic shared memory for every epilogue mode, resolve the tensor-map encoder, read the SM count.
bool gemm_init() {
  bool ok = encode_fn() != nullptr && sm_count() > 0;
  // the register shares of the code epilogues have to add up to no more than the block is launched with
  auto set_up = [&](auto kernel, int warps, bool packed) {
    cudaFuncAttributes a;
    const int side = first_epi_warp(packed), regs = epi_regs(warps, packed);
    ok &= cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess &&
          cudaFuncGetAttributes(&a, kernel) == cudaSuccess && (regs == 0 || side * SIDE_REGS + warps * regs <= (side + warps) * a.numRegs);
  };
  auto set_up_all = [&](auto mode_tag, auto warps_tag) {
    constexpr int MODE = decltype(mode_tag)::value, EW = decltype(warps_tag)::value;
    constexpr bool TAPS = MODE != EPI_MERGE;                  // (a merge has none)
    set_up(k_gemm_tc<MODE, false, EW, false>, EW, false); set_up(k_gemm_tc<MODE, TAPS, EW, false>, EW, false);
    set_up(k_gemm_tc<MODE, always_taps(MODE, true), EW, true>, EW, true);
  };
  set_up_all(std::integral_constant<int, EPI_QKV>{}, std::integral_constant<int, CODE_WARPS>{});
  set_up_all(std::integral_constant<int, EPI_FC1>{}, std::integral_constant<int, CODE_WARPS>{});
  set_up_all(std::integral_constant<int, EPI_PROJ>{}, std::integral_constant<int, F32_WARPS>{});
  set_up_all(std::integral_constant<int, EPI_FC2>{}, std::integral_constant<int, F32_WARPS>{});
  set_up_all(std::integral_constant<int, EPI_MERGE>{}, std::integral_constant<int, F32_WARPS>{});
  return ok;
}

bool launch_gemm(const GemmArgs& g, cudaStream_t st) {
  switch (g.mode) {
    case EPI_QKV:   return launch_mode<EPI_QKV, CODE_WARPS>(g, g.status, st);
    case EPI_FC1:   return launch_mode<EPI_FC1, CODE_WARPS>(g, g.status, st);
    case EPI_PROJ:  return launch_mode<EPI_PROJ, F32_WARPS>(g, g.status, st);
    case EPI_FC2:   return launch_mode<EPI_FC2, F32_WARPS>(g, g.status, st);
    case EPI_MERGE: return launch_mode<EPI_MERGE, F32_WARPS>(g, g.status, st);
  }
  return false;
}

}  // namespace mixaq
