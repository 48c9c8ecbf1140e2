// Host side of the C ABI declared in include/mixaq.h: argument validation, workspace carving, the launch
// schedule of one Two-Branch Swin Block (MixA-Q Section 3.2, Figure 3) and of the backbone loop.
// Nothing here computes: every step of the path runs in the kernels.
#include <nvtx3/nvToolsExt.h>
#include "../../include/mixaq.h"
#include "graph_cache.h"
#include "kernels.h"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <mutex>
#include <new>
#include <string>
#include <vector>

namespace mixaq {
bool ln_dim_supported(int C);
bool merge_dim_supported(int C);
thread_local int g_launches = 0;
}  // namespace mixaq

using namespace mixaq;

struct ProfRec { int cat; cudaEvent_t e0, e1; };
// Writes the key of a call (the exact bytes of every argument that shapes its launches) field by field: the structs contain
// padding bytes whose content the caller does not control.
struct KeyWriter {
  std::string& key;
  void put(const void* ptr, size_t n) { key.append((const char*)ptr, n); }
  template <class T> void val(const T& v) { put(&v, sizeof(v)); }
  void aq(const mixaq_aq& q) { val(q.bits); val(q.scale); val(q.inv_scale); val(q.zero_point); }
  void linear(const mixaq_linear& l) { val(l.codes); val(l.scale); val(l.out_features); val(l.in_features); val(l.bits); }
  void branch(const mixaq_branch& b) {
    const float* ptrs[8] = {b.ln1_g, b.ln1_b, b.ln2_g, b.ln2_b, b.b_qkv, b.b_proj, b.b_fc1, b.b_fc2};
    put(ptrs, sizeof(ptrs));
    aq(b.qkv_in); aq(b.q); aq(b.k); aq(b.v); aq(b.proj_in); aq(b.fc1_in); aq(b.fc2_in);
    val(b.bits);
  }
  void block(const mixaq_block_params& q) {
    const int dims[5] = {q.dim, q.heads, q.window, q.shift, q.hidden};
    put(dims, sizeof(dims));
    linear(q.qkv); linear(q.proj); linear(q.fc1); linear(q.fc2);
    val(q.relpos_table);
    branch(q.hi); branch(q.lo);
    val(q.score_inv_scale); val(q.prepared); val(q.byte_codes);
  }
};
constexpr size_t MAX_BACKBONE_GRAPHS = 16, MAX_BLOCK_GRAPHS = 8;     // kept, and calls remembered (see graph_cache.h)
struct mixaq_ctx {
  int device;
  int* d_status;
  int launches;
  char err[256];
  bool profiling;
  bool graph_cache;                    // replay backbone forwards as CUDA graphs (see mixaq_set_graph_cache)
  bool reverse_selection;              // backbone: worst-case selection order (Table 4) in every block
  bool prof_capture;                   // the profiled call is being captured: event records become graph nodes
  std::vector<cudaGraphExec_t> prof_execs;   // graphs of profiled forwards, destroyed when the profiling ends
  bool guards;                         // fill the guard zones of the workspace before a forward, compare them after it
  bool nvtx;                           // name every kernel family, stage and block with an NVTX range (host side)
  bool allow_elevation;                // backbone: every pair uses its own ratios even if an earlier pair of the stage had larger ones
  cudaStream_t capture_stream;         // calls are recorded here, not on the caller's stream (see replay_record_or_run)
  cudaStream_t side_stream; cudaEvent_t fork, join;   // output norms run beside the next stage inside a captured forward
  std::mutex graph_lock;               // for what follows and the two streams above
  GraphCache<cudaGraphExec_t> graphs{MAX_BACKBONE_GRAPHS, MAX_BACKBONE_GRAPHS};      // of backbone forwards
  GraphCache<cudaGraphExec_t> block_graphs{MAX_BLOCK_GRAPHS, MAX_BLOCK_GRAPHS};
  std::vector<ProfRec> prof;          // event pairs recorded since mixaq_profile_begin
  std::vector<cudaEvent_t> pool;      // events ready for reuse
};

namespace mixaq {
// accessors for translation units that do not see the context's layout
int* ctx_status_word(mixaq_ctx* ctx) { return ctx->d_status; }
int ctx_device(const mixaq_ctx* ctx) { return ctx->device; }
void ctx_note(mixaq_ctx* ctx, const char* msg, int launches) {
  if (msg) snprintf(ctx->err, sizeof(ctx->err), "%s", msg);
  ctx->launches = launches;
}
}  // namespace mixaq

enum ProfCat { PC_ENERGY = 0, PC_SELECT, PC_LN1, PC_QKV, PC_ATTN, PC_PROJ, PC_LN2, PC_FC1, PC_FC2, PC_COPY,
               PC_MERGE_GATHER, PC_MERGE_GEMM, PC_STEM, PC_OUT_NORM, PC_BRACKET, PC_COUNT };
static const char* kProfNames[PC_COUNT] = {"energy", "select", "gather_ln1_quant", "gemm_qkv", "attention",
                                           "gemm_proj", "ln2_quant", "gemm_fc1_gelu", "gemm_fc2_scatter",
                                           "copy_pruned", "merge_gather_ln_quant", "gemm_merge", "patch_embed",
                                           "stage_output_norm", "empty_event_bracket"};

namespace {

inline size_t align_up(size_t v, size_t a = 256) { return (v + a - 1) / a * a; }
// The kernels read and write feature maps, parameters and codes with 16-byte accesses and describe operand matrices
// to the TMA unit (16-byte aligned base); workspaces and prepared buffers are carved in 256-byte steps.  A pointer
// that breaks this would fault on the device, so it is refused on the host.
inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }
inline bool all_aligned_to(size_t a, std::initializer_list<const void*> ptrs) {
  for (const void* p : ptrs) if (!aligned_to(p, a)) return false;
  return true;
}

// Every buffer carved out of a workspace is followed by a guard zone of GUARD_BYTES that no kernel has a reason to
// touch.  With mixaq_set_workspace_guards the zones are filled with a pattern before a forward and compared after it.
thread_local std::vector<void*>* t_guard_log = nullptr;     // where the carver notes its guard zones (NULL: nowhere)
struct Carver {
  char* base; size_t off; bool guarded;
  // guarded = false: the `prepared` parameter tables, written once by the prepare calls (their layout is also read by
  // code that does not carve)
  explicit Carver(void* p, bool with_guards = true) : base((char*)p), off(0), guarded(with_guards) {}
  template <class T> T* take(size_t n) {
    T* p = base ? (T*)(base + off) : nullptr;
    off += align_up(n * sizeof(T));
    if (guarded) {
      if (base && t_guard_log) t_guard_log->push_back(base + off);
      off += GUARD_BYTES;
    }
    return p;
  }
};
// bytes a guarded carver needs for one buffer of n bytes
inline size_t carved_bytes(size_t n) { return align_up(n) + GUARD_BYTES; }
// scope in which carvers log their guard zones into `list` (when the context asks for guards)
struct GuardScope {
  std::vector<void*>* prev;
  GuardScope(const mixaq_ctx* ctx, std::vector<void*>* list) : prev(t_guard_log) { t_guard_log = (ctx && ctx->guards) ? list : nullptr; }
  ~GuardScope() { t_guard_log = prev; }
};

AQ to_aq(const mixaq_aq& q) {
  AQ a; a.scale = q.scale; a.inv_scale = q.inv_scale; a.zp = q.zero_point; a.bits = q.bits;
  a.zpf = (float)q.zero_point; a.qmaxf = (float)((1 << q.bits) - 1);
  return a;
}

mixaq_status fail(mixaq_ctx* ctx, mixaq_status s, const char* msg) {
  if (ctx) snprintf(ctx->err, sizeof(ctx->err), "%s", msg);
  return s;
}

mixaq_status check_cuda(mixaq_ctx* ctx, const char* where) {
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return MIXAQ_OK;
  if (ctx) snprintf(ctx->err, sizeof(ctx->err), "%s: %s", where, cudaGetErrorString(e));
  return MIXAQ_CUDA_ERROR;
}

// Per-kernel CUDA-event timing (only while profiling is on; the events sit on the launching stream).
struct ProfScope {
  mixaq_ctx* ctx; cudaStream_t st; cudaEvent_t e1; bool on, range;
  ProfScope(mixaq_ctx* c, int cat, cudaStream_t s) : ctx(c), st(s), e1(nullptr), on(c && c->profiling), range(c && c->nvtx) {
    if (range) nvtxRangePushA(kProfNames[cat]);
    if (!on) return;
    cudaEvent_t ev[2];
    for (int i = 0; i < 2; ++i) {
      if (!ctx->pool.empty()) { ev[i] = ctx->pool.back(); ctx->pool.pop_back(); }
      else if (cudaEventCreate(&ev[i]) != cudaSuccess) { on = false; return; }
    }
    record(ev[0]);
    e1 = ev[1];
    ctx->prof.push_back({cat, ev[0], ev[1]});
  }
  // inside a stream capture the record becomes a graph node of its own (an "external" event keeps its timestamp)
  void record(cudaEvent_t e) {
    if (ctx->prof_capture) cudaEventRecordWithFlags(e, st, cudaEventRecordExternal);
    else cudaEventRecord(e, st);
  }
  ~ProfScope() { if (on) record(e1); if (range) nvtxRangePop(); }
};
// NVTX range over a stage or a block of the backbone walk (only with mixaq_set_nvtx)
struct NvtxScope {
  bool on;
  NvtxScope(const mixaq_ctx* c, const char* what, int index) : on(c && c->nvtx) {
    if (!on) return;
    char name[48];
    snprintf(name, sizeof(name), "%s %d", what, index);
    nvtxRangePushA(name);
  }
  ~NvtxScope() { if (on) nvtxRangePop(); }
};
#define PROF(cat) ProfScope prof_scope_##cat(ctx, cat, st)

bool bits_ok(int b) { return b == 8 || b == 4 || b == 2; }
bool aq_ok(const mixaq_aq& q, int bits) {
  return q.bits == bits && q.scale > 0.f && q.inv_scale > 0.f && q.zero_point >= 0 && q.zero_point < (1 << bits);
}
bool linear_ok(const mixaq_linear& l, int out_f, int in_f) {
  return l.codes && l.scale && l.out_features == out_f && l.in_features == in_f;
}
bool branch_ok(const mixaq_branch& b) {
  if (!bits_ok(b.bits)) return false;
  if (!b.ln1_g || !b.ln1_b || !b.ln2_g || !b.ln2_b || !b.b_qkv || !b.b_proj || !b.b_fc1 || !b.b_fc2) return false;
  return aq_ok(b.qkv_in, b.bits) && aq_ok(b.q, b.bits) && aq_ok(b.k, b.bits) && aq_ok(b.v, b.bits) &&
         aq_ok(b.proj_in, b.bits) && aq_ok(b.fc1_in, b.bits) && aq_ok(b.fc2_in, b.bits);
}

bool branch_ptrs_ok(const mixaq_branch& b) {
  return b.ln1_g && b.ln1_b && b.ln2_g && b.ln2_b && b.b_qkv && b.b_proj && b.b_fc1 && b.b_fc2;
}

// need_quantizers = false: the calibration pass, which runs before any quantizer exists
mixaq_status validate_block(mixaq_ctx* ctx, const mixaq_block_params* p, bool need_quantizers = true) {
  if (!p) return fail(ctx, MIXAQ_INVALID_ARG, "block params are NULL");
  if (p->window != WS) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "window must be 7");
  if (p->dim <= 0 || p->dim % 32 || !ln_dim_supported(p->dim)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "unsupported dim");
  if (p->heads <= 0 || p->dim != p->heads * HEAD_DIM) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "dim/heads must be 32");
  if (p->hidden <= 0 || p->hidden % 32) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "hidden must be a multiple of 32");
  if (p->shift < 0 || p->shift >= WS) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "shift must be in [0, window)");
  if (!linear_ok(p->qkv, 3 * p->dim, p->dim) || !linear_ok(p->proj, p->dim, p->dim) ||
      !linear_ok(p->fc1, p->hidden, p->dim) || !linear_ok(p->fc2, p->dim, p->hidden))
    return fail(ctx, MIXAQ_INVALID_ARG, "weight matrix missing or of the wrong shape");
  if (!p->relpos_table) return fail(ctx, MIXAQ_INVALID_ARG, "relpos_table is NULL");
  {
    const void* q16[] = {p->qkv.codes, p->proj.codes, p->fc1.codes, p->fc2.codes,
                         p->hi.ln1_g, p->hi.ln1_b, p->hi.ln2_g, p->hi.ln2_b, p->lo.ln1_g, p->lo.ln1_b, p->lo.ln2_g, p->lo.ln2_b};
    for (const void* q : q16)
      if (!aligned_to(q, 16)) return fail(ctx, MIXAQ_INVALID_ARG, "weight codes and LayerNorm parameters must be 16-byte aligned");
    const bool words = all_aligned_to(4, {p->qkv.scale, p->proj.scale, p->fc1.scale, p->fc2.scale, p->relpos_table,
                                          p->hi.b_qkv, p->hi.b_proj, p->hi.b_fc1, p->hi.b_fc2,
                                          p->lo.b_qkv, p->lo.b_proj, p->lo.b_fc1, p->lo.b_fc2});
    if (!words) return fail(ctx, MIXAQ_INVALID_ARG, "step sizes, biases and the relative-position table must be 4-byte aligned");
    if (p->prepared && !aligned_to(p->prepared, 256)) return fail(ctx, MIXAQ_INVALID_ARG, "prepared buffer must be 256-byte aligned");
  }
  if (p->byte_codes != 0 && p->byte_codes != 1) return fail(ctx, MIXAQ_INVALID_ARG, "byte_codes must be 0 or 1");
  if (!need_quantizers) {
    if (!branch_ptrs_ok(p->hi) || !branch_ptrs_ok(p->lo)) return fail(ctx, MIXAQ_INVALID_ARG, "branch parameters invalid");
    return MIXAQ_OK;
  }
  if (!branch_ok(p->hi) || !branch_ok(p->lo)) return fail(ctx, MIXAQ_INVALID_ARG, "branch parameters invalid");
  if (!(p->score_inv_scale > 0.f)) return fail(ctx, MIXAQ_INVALID_ARG, "score_inv_scale must be positive");
  return MIXAQ_OK;
}

// layout of a block's prepared buffer
struct Prepared {
  float* mult[4][2]; int32_t* pre[4][2]; float* bound[4][2]; float* relbias; size_t bytes;
};
Prepared carve_prepared(const mixaq_block_params* p, void* base) {
  Prepared r; Carver c(base, false);
  const int N[4] = {3 * p->dim, p->dim, p->hidden, p->dim};
  for (int l = 0; l < 4; ++l)
    for (int b = 0; b < 2; ++b) {
      r.mult[l][b] = c.take<float>(N[l]); r.pre[l][b] = c.take<int32_t>(N[l]); r.bound[l][b] = c.take<float>(N[l]);
    }
  r.relbias = c.take<float>((size_t)p->heads * 4 * 7 * 32 * 4);   // fragment order, see k_prepare_relbias
  r.bytes = c.off;
  return r;
}

struct Geometry { int Hp, Wp, nwx, nW, n_hi, n_lo, n_pr; };
Geometry geometry(int H, int W, float low, float prune) {
  Geometry g;
  g.Hp = (H + WS - 1) / WS * WS; g.Wp = (W + WS - 1) / WS * WS;
  g.nwx = g.Wp / WS; g.nW = (g.Hp / WS) * g.nwx;
  g.n_pr = mixaq_low_count(prune, g.nW);
  g.n_lo = mixaq_low_count(low, g.nW - g.n_pr);
  g.n_hi = g.nW - g.n_pr - g.n_lo;
  return g;
}

// buffers the selection kernels fill for one block (all sized for the worst split)
struct SelWs {
  int64_t* score; int32_t* order; uint8_t* cls; int32_t *rowsrc[3], *win[2]; size_t bytes;
};
SelWs carve_sel(int B, int H, int W, void* base) {
  SelWs w; Carver c(base);
  Geometry g = geometry(H, W, 0.f, 0.f);
  const size_t slots = (size_t)B * g.nW, rows = slots * WT;
  w.score = c.take<int64_t>(slots); w.order = c.take<int32_t>(slots); w.cls = c.take<uint8_t>(slots);
  for (int i = 0; i < 3; ++i) w.rowsrc[i] = c.take<int32_t>(rows);
  for (int i = 0; i < 2; ++i) w.win[i] = c.take<int32_t>(slots);
  w.bytes = c.off;
  return w;
}

// workspace of one block call; sized for the worst split (all windows in the wider branch)
struct BlockWs {
  int32_t* energy; SelWs sel;
  uint8_t *a[2], *qkv[2], *o[2], *f1[2], *f2[2]; float* x1[2];
  size_t bytes;
};
BlockWs carve_block(const mixaq_block_params* p, int B, int H, int W, void* base) {
  BlockWs w; Carver c(base);
  Geometry g = geometry(H, W, 0.f, 0.f);
  const size_t slots = (size_t)B * g.nW, rows = slots * WT;
  const int C = p->dim, Hd = p->hidden;
  w.energy = c.take<int32_t>((size_t)B * H * W);
  w.sel = carve_sel(B, H, W, base ? (char*)base + c.off : nullptr);
  c.off += w.sel.bytes;
  for (int i = 0; i < 2; ++i) {
    const int bits = p->byte_codes ? 8 : (i == 0 ? p->hi.bits : p->lo.bits);     // container of a code
    w.a[i]   = c.take<uint8_t>(rows * C * bits / 8);
    w.qkv[i] = c.take<uint8_t>(rows * 3 * C * bits / 8);
    w.o[i]   = c.take<uint8_t>(rows * C * bits / 8);
    w.x1[i]  = c.take<float>(rows * C);
    w.f1[i]  = c.take<uint8_t>(rows * C * bits / 8);
    w.f2[i]  = c.take<uint8_t>(rows * Hd * bits / 8);
  }
  w.bytes = c.off;
  return w;
}

// The code buffers of a bit-packed block laid out anew with one byte per code, for the M[i] rows that the branches have in this call.
// Expanding packed codes in front of every MMA costs more than their bytes save (Swin-T 800 x 1333, bit-packed against bytes: 916
// and 841 us; Swin-S 4 x 1024 x 1024 at A4 / A2: 3 918 and 3 487), and nobody sees the storage but the taps.  The packed carving
// sizes each branch for all rows and keeps apart what is never alive at once, so bytes fit into the same memory: x1; the q, k, v
// codes and after them fc1's; the codes of LN1 and after them LN2's; those of the attention.  Guard zones follow these buffers as they
// do the packed ones (four in the room of twelve).  false: not enough room (hidden layers beyond 10 C at two bits); ws is left as it is.
bool carve_bytes(const mixaq_block_params* p, const int (&M)[2], void* workspace, BlockWs& ws) {
  const size_t rows = (size_t)M[0] + M[1], C = p->dim, Hd = p->hidden, wide = std::max(3 * C, Hd);
  const size_t need = carved_bytes(rows * C * sizeof(float)) + carved_bytes(rows * wide) + 2 * carved_bytes(rows * C);
  if (need > (size_t)((char*)workspace + ws.bytes - (char*)ws.a[0])) return false;
  // the zones of the packed buffers lie inside the new ones
  if (t_guard_log) {
    auto inside = [&](void* zone) { return (char*)zone >= (char*)ws.a[0]; };
    t_guard_log->erase(std::remove_if(t_guard_log->begin(), t_guard_log->end(), inside), t_guard_log->end());
  }
  Carver c(ws.a[0]);
  float* x1 = c.take<float>(rows * C);
  uint8_t *big = c.take<uint8_t>(rows * wide), *ln = c.take<uint8_t>(rows * C), *o = c.take<uint8_t>(rows * C);
  const size_t m0 = M[0];
  for (int i = 0; i < 2; ++i) {
    const size_t r = i == 0 ? 0 : m0;                        // the high branch's rows come first
    ws.x1[i] = x1 + r * C;
    ws.qkv[i] = big + r * 3 * C; ws.f2[i] = big + r * Hd;
    ws.a[i] = ws.f1[i] = ln + r * C; ws.o[i] = o + r * C;
  }
  return true;
}

SelectArgs make_select_args(const SelWs& sel, const int32_t* energy, int B, int H, int W, int shift, const Geometry& g,
                            int reverse, bool own_energy) {
  SelectArgs sa;
  sa.energy = energy; sa.score = sel.score; sa.order = sel.order; sa.cls = sel.cls;
  sa.rowsrc_hi = sel.rowsrc[0]; sa.rowsrc_lo = sel.rowsrc[1]; sa.rowsrc_pr = sel.rowsrc[2];
  sa.win_hi = sel.win[0]; sa.win_lo = sel.win[1];
  sa.B = B; sa.H = H; sa.W = W; sa.shift = shift; sa.nwx = g.nwx; sa.nW = g.nW;
  sa.n_hi = g.n_hi; sa.n_lo = g.n_lo; sa.n_pr = g.n_pr; sa.reverse = reverse; sa.narrow = own_energy;
  return sa;
}

void fill_gemm_branch(GemmBranch& g, const uint8_t* a, int M, int a_bits, const float* mult, const int32_t* pre,
                      const float* bound, const float* bias) {
  memset(&g, 0, sizeof(g));
  g.a = a; g.M = M; g.a_bits = a_bits; g.mult = mult; g.pre = pre; g.bound = bound; g.bias = bias;
}

}  // namespace

// =================================================================================================
extern "C" {

int mixaq_low_count(float ratio, int n) { return (int)std::floor((double)ratio * (double)n + 1e-6); }

mixaq_status mixaq_branch_counts(int H, int W, int window, float low_ratio, float prune_ratio, int* counts) {
  if (!counts || window != WS || H <= 0 || W <= 0) return MIXAQ_INVALID_ARG;
  if (!(low_ratio >= 0.f && low_ratio <= 1.f) || !(prune_ratio >= 0.f && prune_ratio <= 1.f)) return MIXAQ_INVALID_ARG;
  Geometry g = geometry(H, W, low_ratio, prune_ratio);
  counts[0] = g.n_hi; counts[1] = g.n_lo; counts[2] = g.n_pr;
  return MIXAQ_OK;
}

mixaq_status mixaq_create(mixaq_ctx** out, int device) {
  if (!out) return MIXAQ_INVALID_ARG;
  *out = nullptr;
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) { cudaGetLastError(); return MIXAQ_CUDA_ERROR; }
  if (cudaSetDevice(device) != cudaSuccess) { cudaGetLastError(); return MIXAQ_CUDA_ERROR; }
  mixaq_ctx* c = new (std::nothrow) mixaq_ctx();
  if (!c) return MIXAQ_INTERNAL;
  c->device = device; c->launches = 0; c->err[0] = 0; c->d_status = nullptr; c->profiling = false; c->graph_cache = true; c->allow_elevation = false; c->reverse_selection = false; c->nvtx = false; c->prof_capture = false; c->guards = false; c->capture_stream = nullptr; c->side_stream = nullptr; c->fork = c->join = nullptr;
  if (cudaMalloc(&c->d_status, sizeof(int)) != cudaSuccess || cudaMemset(c->d_status, 0, sizeof(int)) != cudaSuccess ||
      !gemm_init() || !ln_init()) {
    cudaGetLastError(); if (c->d_status) cudaFree(c->d_status); delete c; return MIXAQ_CUDA_ERROR;
  }
  *out = c;
  return MIXAQ_OK;
}

mixaq_status mixaq_destroy(mixaq_ctx* ctx) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (ctx->d_status) cudaFree(ctx->d_status);
  if (ctx->capture_stream) cudaStreamDestroy(ctx->capture_stream);
  if (ctx->side_stream) { cudaStreamDestroy(ctx->side_stream); cudaEventDestroy(ctx->fork); cudaEventDestroy(ctx->join); }
  ctx->graphs.clear(cudaGraphExecDestroy);
  ctx->block_graphs.clear(cudaGraphExecDestroy);
  for (cudaGraphExec_t g : ctx->prof_execs) cudaGraphExecDestroy(g);
  for (auto& r : ctx->prof) { cudaEventDestroy(r.e0); cudaEventDestroy(r.e1); }
  for (auto e : ctx->pool) cudaEventDestroy(e);
  delete ctx;
  return MIXAQ_OK;
}

const char* mixaq_last_error(const mixaq_ctx* ctx) { return ctx ? ctx->err : "no context"; }
int mixaq_last_launch_count(const mixaq_ctx* ctx) { return ctx ? ctx->launches : 0; }

mixaq_status mixaq_last_device_status(mixaq_ctx* ctx, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  int h = 0;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (cudaMemcpyAsync(&h, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
  { check_cuda(ctx, "status read"); return MIXAQ_CUDA_ERROR; }
  return h == 0 ? MIXAQ_OK : ((h & 2) ? MIXAQ_WORKSPACE_OVERRUN : MIXAQ_DEVICE_TIMEOUT);
}

mixaq_status mixaq_clear_device_status(mixaq_ctx* ctx, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (cudaMemsetAsync(ctx->d_status, 0, sizeof(int), (cudaStream_t)cuda_stream) != cudaSuccess) return check_cuda(ctx, "clear status");
  return MIXAQ_OK;
}

mixaq_status mixaq_selftest_wait_timeout(mixaq_ctx* ctx, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  launch_wait_probe(ctx->d_status, (cudaStream_t)cuda_stream);
  return check_cuda(ctx, "selftest_wait_timeout");
}

mixaq_status mixaq_measure_mma_peak(mixaq_ctx* ctx, int kind, int groups, void* scratch, size_t scratch_bytes,
                                    double* tera_ops_per_s, void* cuda_stream) {
  if (!ctx || !scratch || !tera_ops_per_s || groups <= 0 || kind < 0 || kind > 2) return MIXAQ_INVALID_ARG;
  if (scratch_bytes < 1024 * sizeof(unsigned long long)) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "mma peak: scratch of 8 KiB needed");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  unsigned long long* d_ns = (unsigned long long*)scratch;
  const int sms = launch_mma_peak(kind, groups, d_ns, ctx->d_status, st);
  if (sms <= 0 || sms > 1024) return check_cuda(ctx, "mma peak") == MIXAQ_OK ? MIXAQ_INTERNAL : MIXAQ_CUDA_ERROR;
  std::vector<unsigned long long> ns(sms);
  if (cudaMemcpyAsync(ns.data(), d_ns, sizeof(unsigned long long) * sms, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) return check_cuda(ctx, "mma peak");
  unsigned long long worst = 1;
  for (auto v : ns) worst = v > worst ? v : worst;
  // every SM issued groups x 4 MMAs of 128 x 256 x 32 (kind 2: x 64) multiply-accumulates; all SMs ran at once: the
  // slowest one counts
  const double k_per_mma = kind == 2 ? 64.0 : 32.0;
  const double ops = 2.0 * 128.0 * 256.0 * k_per_mma * 4.0 * (double)groups * (double)sms;
  *tera_ops_per_s = ops / ((double)worst * 1e-9) / 1e12;
  return check_cuda(ctx, "mma peak");
}

int mixaq_profile_categories(void) { return PC_COUNT; }
const char* mixaq_profile_category_name(int cat) { return (cat >= 0 && cat < PC_COUNT) ? kProfNames[cat] : ""; }

mixaq_status mixaq_profile_begin(mixaq_ctx* ctx) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  for (auto& r : ctx->prof) { ctx->pool.push_back(r.e0); ctx->pool.push_back(r.e1); }
  ctx->prof.clear();
  ctx->profiling = true;
  return MIXAQ_OK;
}

mixaq_status mixaq_profile_end(mixaq_ctx* ctx, void* cuda_stream, float* ms_per_category, int* launches_per_category) {
  if (!ctx || !ms_per_category || !launches_per_category) return MIXAQ_INVALID_ARG;
  ctx->profiling = false;
  if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) return check_cuda(ctx, "profile_end");
  for (cudaGraphExec_t g : ctx->prof_execs) cudaGraphExecDestroy(g);
  ctx->prof_execs.clear();
  for (int i = 0; i < PC_COUNT; ++i) { ms_per_category[i] = 0.f; launches_per_category[i] = 0; }
  for (auto& r : ctx->prof) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.e0, r.e1) == cudaSuccess) { ms_per_category[r.cat] += ms; launches_per_category[r.cat] += 1; }
    ctx->pool.push_back(r.e0); ctx->pool.push_back(r.e1);
  }
  ctx->prof.clear();
  return check_cuda(ctx, "profile_end");
}

mixaq_status mixaq_profile_end_records(mixaq_ctx* ctx, void* cuda_stream, int* category, float* ms, int capacity, int* count) {
  if (!ctx || !category || !ms || !count || capacity < 0) return MIXAQ_INVALID_ARG;
  ctx->profiling = false;
  if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) return check_cuda(ctx, "profile_end_records");
  for (cudaGraphExec_t g : ctx->prof_execs) cudaGraphExecDestroy(g);
  ctx->prof_execs.clear();
  int n = 0;
  for (auto& r : ctx->prof) {
    float t = 0.f;
    if (n < capacity) {
      if (cudaEventElapsedTime(&t, r.e0, r.e1) != cudaSuccess) { cudaGetLastError(); t = 0.f; }
      category[n] = r.cat; ms[n] = t;
    }
    ++n;
    ctx->pool.push_back(r.e0); ctx->pool.push_back(r.e1);
  }
  ctx->prof.clear();
  *count = n;
  return check_cuda(ctx, "profile_end_records");
}

// -------------------------------------------------------------------------------------------------
size_t mixaq_block_prepared_bytes(const mixaq_block_params* p) {
  if (!p || p->dim <= 0 || p->hidden <= 0 || p->heads <= 0) return 0;
  return carve_prepared(p, nullptr).bytes;
}

mixaq_status mixaq_block_prepare(mixaq_ctx* ctx, const mixaq_block_params* p, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  mixaq_status s = validate_block(ctx, p);
  if (s != MIXAQ_OK) return s;
  if (!p->prepared) return fail(ctx, MIXAQ_INVALID_ARG, "prepared buffer is NULL");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Prepared pr = carve_prepared(p, p->prepared);
  const mixaq_linear* L[4] = {&p->qkv, &p->proj, &p->fc1, &p->fc2};
  for (int b = 0; b < 2; ++b) {
    const mixaq_branch& br = b == 0 ? p->hi : p->lo;
    const mixaq_aq* in[4] = {&br.qkv_in, &br.proj_in, &br.fc1_in, &br.fc2_in};
    for (int l = 0; l < 4; ++l)
      launch_prepare_linear(L[l]->codes, L[l]->scale, L[l]->out_features, L[l]->in_features, in[l]->scale,
                            in[l]->zero_point, in[l]->bits, pr.mult[l][b], pr.pre[l][b], pr.bound[l][b], st);
  }
  launch_prepare_relbias(p->relpos_table, p->heads, pr.relbias, st);
  return check_cuda(ctx, "block_prepare");
}

size_t mixaq_merge_prepared_bytes(const mixaq_merge_params* p) {
  if (!p || p->reduction.out_features <= 0) return 0;
  return align_up((size_t)p->reduction.out_features * 4) * 3;
}

mixaq_status mixaq_merge_prepare(mixaq_ctx* ctx, const mixaq_merge_params* p, void* cuda_stream) {
  if (!ctx || !p) return MIXAQ_INVALID_ARG;
  if (!p->prepared || !p->reduction.codes || !p->reduction.scale) return fail(ctx, MIXAQ_INVALID_ARG, "merge params incomplete");
  if (!all_aligned_to(4, {p->prepared, p->reduction.scale}))
    return fail(ctx, MIXAQ_INVALID_ARG, "merge: step sizes and prepared must be 4-byte aligned");
  Carver c(p->prepared, false);
  float* mult = c.take<float>(p->reduction.out_features);
  int32_t* pre = c.take<int32_t>(p->reduction.out_features);
  float* bound = c.take<float>(p->reduction.out_features);
  launch_prepare_linear(p->reduction.codes, p->reduction.scale, p->reduction.out_features, p->reduction.in_features,
                        p->in.scale, p->in.zero_point, p->in.bits, mult, pre, bound, (cudaStream_t)cuda_stream);
  return check_cuda(ctx, "merge_prepare");
}

mixaq_status mixaq_stage_energy(mixaq_ctx* ctx, const float* x, int32_t* energy, int B, int H, int W, int C,
                                float score_inv_scale, void* cuda_stream) {
  if (!ctx || !x || !energy || B <= 0 || H <= 0 || W <= 0 || C <= 0 || !(score_inv_scale > 0.f)) return MIXAQ_INVALID_ARG;
  if (!aligned_to(x, 16) || !aligned_to(energy, 4)) return fail(ctx, MIXAQ_INVALID_ARG, "stage_energy: x must be 16-byte aligned");
  launch_energy(x, energy, (long)B * H * W, C, score_inv_scale, (cudaStream_t)cuda_stream);
  return check_cuda(ctx, "stage_energy");
}

// -------------------------------------------------------------------------------------------------
size_t mixaq_block_workspace_bytes(const mixaq_block_params* p, int B, int H, int W) {
  if (!p || B <= 0 || H <= 0 || W <= 0 || p->dim <= 0 || p->hidden <= 0) return 0;
  return carve_block(p, B, H, W, nullptr).bytes;
}

}  // extern "C"

// What the kernels read or write through the optional arguments, by whole 32-bit elements.  (cls, order, score and the taps
// that are filled by copies may sit at any address.)
static bool optional_buffers_aligned(const mixaq_select_opts* opts, const mixaq_selection* sel, const mixaq_taps* taps) {
  bool ok = !opts || aligned_to(opts->energy, 4);
  if (sel) ok &= all_aligned_to(4, {sel->idx_hi, sel->idx_lo, sel->idx_pr});
  if (taps)
    for (const mixaq_branch_taps* t : {&taps->hi, &taps->lo})
      ok &= all_aligned_to(4, {t->qkv_acc, t->probs, t->pv_acc, t->proj_acc, t->fc1_acc, t->fc2_acc});
  return ok;
}

// `presel`: selection buffers already filled for this block (the backbone selects once per stage); NULL: select here.
static mixaq_status block_forward_impl(mixaq_ctx* ctx, const mixaq_block_params* p, const float* x, float* y,
                                       int B, int H, int W, float low_ratio, float prune_ratio,
                                       const mixaq_select_opts* opts, const mixaq_selection* sel_out,
                                       void* workspace, size_t workspace_bytes, const mixaq_taps* taps,
                                       const SelWs* presel, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  mixaq_status s = validate_block(ctx, p);
  if (s != MIXAQ_OK) return s;
  if (!x || !y || x == y) return fail(ctx, MIXAQ_INVALID_ARG, "x / y NULL or aliased");
  if (!aligned_to(x, 16) || !aligned_to(y, 16)) return fail(ctx, MIXAQ_INVALID_ARG, "x and y must be 16-byte aligned");
  if (!optional_buffers_aligned(opts, sel_out, taps))
    return fail(ctx, MIXAQ_INVALID_ARG, "energy, window lists, accumulator taps and softmax taps must be 4-byte aligned");
  if (B <= 0 || H <= 0 || W <= 0) return fail(ctx, MIXAQ_INVALID_ARG, "B, H, W must be positive");
  if (!(low_ratio >= 0.f && low_ratio <= 1.f) || !(prune_ratio >= 0.f && prune_ratio <= 1.f))
    return fail(ctx, MIXAQ_INVALID_ARG, "ratios must lie in [0, 1]");
  if (!p->prepared) return fail(ctx, MIXAQ_INVALID_ARG, "block was not prepared (prepared == NULL)");
  if ((long)B * H * W >= (1L << 31) / WT) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "too many tokens");
  Geometry g = geometry(H, W, low_ratio, prune_ratio);
  if ((size_t)g.nW * 8 > 48 * 1024) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "too many windows per image (max 6144)");
  if (!workspace) return fail(ctx, MIXAQ_INVALID_ARG, "workspace is NULL");
  if (!aligned_to(workspace, 256)) return fail(ctx, MIXAQ_INVALID_ARG, "workspace must be 256-byte aligned");
  std::vector<void*> guard_zones;
  GuardScope guard_scope(ctx, &guard_zones);
  BlockWs ws = carve_block(p, B, H, W, workspace);
  if (ws.bytes > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "workspace too small");
  const int M[2] = {B * g.n_hi * WT, B * g.n_lo * WT};
  // bits a stored code occupies: a whole byte, or the branch's bit width (bit-packed: what the taps hand out)
  const bool bytes = p->byte_codes || (!taps && carve_bytes(p, M, workspace, ws));
  const int cb[2] = {bytes ? 8 : p->hi.bits, bytes ? 8 : p->lo.bits};
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int C = p->dim, Hd = p->hidden;
  Prepared pr = carve_prepared(p, p->prepared);
  if (!guard_zones.empty()) launch_guards(guard_zones.data(), (int)guard_zones.size(), true, ctx->d_status, st);
  g_launches = 0;

  // 1. scores and selection
  SelWs sel = presel ? *presel : ws.sel;
  if (sel_out && !presel) {
    // the selection kernels write the caller's buffers themselves, whole elements at a time; a buffer whose address does
    // not allow that is filled by a copy
    if (sel_out->cls) sel.cls = sel_out->cls;
    if (sel_out->order && aligned_to(sel_out->order, alignof(int32_t))) sel.order = sel_out->order;
    if (sel_out->score && aligned_to(sel_out->score, alignof(int64_t))) sel.score = sel_out->score;
  }
  if (!presel) {
    const int32_t* energy = opts ? opts->energy : nullptr;
    const bool own_energy = !energy;
    if (own_energy) { PROF(PC_ENERGY); launch_energy(x, ws.energy, (long)B * H * W, C, p->score_inv_scale, st); energy = ws.energy; }
    SelectArgs sa = make_select_args(sel, energy, B, H, W, p->shift, g, opts ? opts->reverse : 0, own_energy);
    { PROF(PC_SELECT); launch_select(&sa, 1, st); }
  }
  if (sel_out) {
    const size_t n = (size_t)B * g.nW;
    if (sel_out->order && sel.order != sel_out->order) cudaMemcpyAsync(sel_out->order, sel.order, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    if (sel_out->score && sel.score != sel_out->score) cudaMemcpyAsync(sel_out->score, sel.score, n * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    if (sel_out->idx_hi || sel_out->idx_lo || sel_out->idx_pr) {
      int32_t* const lists[3] = {sel_out->idx_hi, sel_out->idx_lo, sel_out->idx_pr};
      const int cnt[3] = {g.n_hi, g.n_lo, g.n_pr};
      launch_class_lists(sel.cls, B, g.nW, lists, cnt, st);
    }
  }

  const mixaq_branch* brp[2] = {&p->hi, &p->lo};
  const int slots[2] = {B * g.n_hi, B * g.n_lo};
  const mixaq_branch_taps* tp[2] = {taps ? &taps->hi : nullptr, taps ? &taps->lo : nullptr};

  // 2. gather + LN1 + quantize + pack
  LnBranch lb[2];
  for (int i = 0; i < 2; ++i) {
    lb[i].src = x; lb[i].rowsrc = sel.rowsrc[i]; lb[i].gamma = brp[i]->ln1_g; lb[i].beta = brp[i]->ln1_b;
    lb[i].out = ws.a[i]; lb[i].q = to_aq(brp[i]->qkv_in); lb[i].q.bits = cb[i]; lb[i].M = M[i];
  }
  { PROF(PC_LN1); launch_ln_quant(lb[0], lb[1], C, st); }

  // 3. QKV GEMM -> q, k, v codes
  GemmArgs ga;
  ga.status = ctx->d_status;
  ga.w = p->qkv.codes; ga.N = 3 * C; ga.K = C; ga.C = C; ga.mode = EPI_QKV;
  for (int i = 0; i < 2; ++i) {
    fill_gemm_branch(ga.br[i], ws.a[i], M[i], cb[i], pr.mult[0][i], pr.pre[0][i], pr.bound[0][i], brp[i]->b_qkv);
    ga.br[i].q0 = to_aq(brp[i]->q); ga.br[i].q1 = to_aq(brp[i]->k); ga.br[i].q2 = to_aq(brp[i]->v);
    ga.br[i].out_bits = cb[i]; ga.br[i].out_codes = ws.qkv[i];
    ga.br[i].tap_acc = tp[i] ? tp[i]->qkv_acc : nullptr;
  }
  { PROF(PC_QKV); if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)"); }

  // 4. window attention
  AttnArgs aa;
  aa.relbias = pr.relbias; aa.C = C; aa.heads = p->heads; aa.shift = p->shift; aa.Hp = g.Hp; aa.Wp = g.Wp;
  aa.nwx = g.nwx; aa.nW = g.nW;
  const float rs = (float)(1.0 / std::sqrt((double)HEAD_DIM));
  for (int i = 0; i < 2; ++i) {
    AttnBranch& ab = aa.br[i];
    ab.qkv = ws.qkv[i]; ab.out = ws.o[i]; ab.win = sel.win[i];
    ab.q = to_aq(brp[i]->q); ab.k = to_aq(brp[i]->k); ab.v = to_aq(brp[i]->v); ab.o = to_aq(brp[i]->proj_in);
    ab.bits = brp[i]->bits; ab.cbits = cb[i]; ab.slots = slots[i];
    ab.alpha = (brp[i]->q.scale * brp[i]->k.scale) * rs;
    ab.so = (1.0f / (float)((1 << brp[i]->bits) - 1)) * brp[i]->v.scale;
    ab.tap_p = tp[i] ? tp[i]->p_codes : nullptr; ab.tap_probs = tp[i] ? tp[i]->probs : nullptr; ab.tap_pv = tp[i] ? tp[i]->pv_acc : nullptr;
  }
  { PROF(PC_ATTN); launch_attention(aa, st); }

  // 5. proj GEMM + attention residual -> x1
  ga.w = p->proj.codes; ga.N = C; ga.K = C; ga.mode = EPI_PROJ;
  for (int i = 0; i < 2; ++i) {
    fill_gemm_branch(ga.br[i], ws.o[i], M[i], cb[i], pr.mult[1][i], pr.pre[1][i], pr.bound[1][i], brp[i]->b_proj);
    ga.br[i].out_f = ws.x1[i]; ga.br[i].res = x; ga.br[i].rowsrc = sel.rowsrc[i];
    ga.br[i].tap_acc = tp[i] ? tp[i]->proj_acc : nullptr;
  }
  { PROF(PC_PROJ); if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)"); }

  // 6. LN2 + quantize + pack
  for (int i = 0; i < 2; ++i) {
    lb[i].src = ws.x1[i]; lb[i].rowsrc = nullptr; lb[i].gamma = brp[i]->ln2_g; lb[i].beta = brp[i]->ln2_b;
    lb[i].out = ws.f1[i]; lb[i].q = to_aq(brp[i]->fc1_in); lb[i].q.bits = cb[i]; lb[i].M = M[i];
  }
  { PROF(PC_LN2); launch_ln_quant(lb[0], lb[1], C, st); }

  // 7. fc1 GEMM + GELU + requantize
  ga.w = p->fc1.codes; ga.N = Hd; ga.K = C; ga.mode = EPI_FC1;
  for (int i = 0; i < 2; ++i) {
    fill_gemm_branch(ga.br[i], ws.f1[i], M[i], cb[i], pr.mult[2][i], pr.pre[2][i], pr.bound[2][i], brp[i]->b_fc1);
    ga.br[i].q0 = to_aq(brp[i]->fc2_in); ga.br[i].out_bits = cb[i]; ga.br[i].out_codes = ws.f2[i];
    ga.br[i].tap_acc = tp[i] ? tp[i]->fc1_acc : nullptr;
  }
  { PROF(PC_FC1); if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)"); }

  // 8. fc2 GEMM + residual + scatter (reverse shift, crop)
  ga.w = p->fc2.codes; ga.N = C; ga.K = Hd; ga.mode = EPI_FC2;
  for (int i = 0; i < 2; ++i) {
    fill_gemm_branch(ga.br[i], ws.f2[i], M[i], cb[i], pr.mult[3][i], pr.pre[3][i], pr.bound[3][i], brp[i]->b_fc2);
    ga.br[i].out_f = y; ga.br[i].res = ws.x1[i]; ga.br[i].rowsrc = sel.rowsrc[i];
    ga.br[i].tap_acc = tp[i] ? tp[i]->fc2_acc : nullptr;
  }
  { PROF(PC_FC2); if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)"); }

  // 9. pruned windows are forwarded unchanged
  if (g.n_pr > 0) { PROF(PC_COPY); launch_copy_rows(x, y, sel.rowsrc[2], B * g.n_pr * WT, C, st); }

  if (taps) {
    for (int i = 0; i < 2; ++i) {
      const size_t rows = (size_t)M[i]; const int bits = cb[i];
      if (rows == 0) continue;
      if (tp[i]->a_codes)   cudaMemcpyAsync(tp[i]->a_codes, ws.a[i], rows * C * bits / 8, cudaMemcpyDeviceToDevice, st);
      if (tp[i]->qkv_codes) cudaMemcpyAsync(tp[i]->qkv_codes, ws.qkv[i], rows * 3 * C * bits / 8, cudaMemcpyDeviceToDevice, st);
      if (tp[i]->o_codes)   cudaMemcpyAsync(tp[i]->o_codes, ws.o[i], rows * C * bits / 8, cudaMemcpyDeviceToDevice, st);
      if (tp[i]->x1)        cudaMemcpyAsync(tp[i]->x1, ws.x1[i], rows * C * 4, cudaMemcpyDeviceToDevice, st);
      if (tp[i]->f1_codes)  cudaMemcpyAsync(tp[i]->f1_codes, ws.f1[i], rows * C * bits / 8, cudaMemcpyDeviceToDevice, st);
      if (tp[i]->f2_codes)  cudaMemcpyAsync(tp[i]->f2_codes, ws.f2[i], rows * Hd * bits / 8, cudaMemcpyDeviceToDevice, st);
    }
  }
  ctx->launches = g_launches;
  if (!guard_zones.empty()) launch_guards(guard_zones.data(), (int)guard_zones.size(), false, ctx->d_status, st);
  return check_cuda(ctx, "block_forward");
}

// ---- graphs of whole calls ---------------------------------------------------------------------------------------------
// the legacy default stream cannot be captured itself
static bool is_legacy(cudaStream_t st) { return st == nullptr || st == cudaStreamLegacy; }
static bool caller_is_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (is_legacy(st) || (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone)) return false;
  cudaGetLastError();
  return true;
}
// The call `forward(stream, recording)` with this key: replayed when it was recorded before, recorded (and launched) when
// that is worth it and works, else issued on the caller's stream: recording takes device memory, which a call does not
// otherwise need, so that it fails is no reason for the call to fail.  What a call costs (us, Swin-T forwards on the default stream,
// waited for one by one; 224 x 224 image / 800 x 1333 map): 393 / 802 replayed, 433 / 801 issued, 798 / 1 119 recorded.
// Calls are recorded on a stream of the context's own: the legacy default stream cannot be captured, and while another one
// is, it refuses what other threads put on it (a blocking one makes work on the default stream fail too).
// The caller holds graph_lock.
template <class Forward>
static mixaq_status replay_record_or_run(mixaq_ctx* ctx, GraphCache<cudaGraphExec_t>& cache, std::string&& key,
                                         cudaStream_t user_stream, const char* what, Forward forward) {
  if (const auto* g = cache.replay(key)) {
    if (cudaGraphLaunch(g->exec, user_stream) != cudaSuccess) return check_cuda(ctx, what);
    ctx->launches = g->launches;
    return MIXAQ_OK;
  }
  bool record = cache.worth_recording(key);
  if (record && !ctx->capture_stream && cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking) != cudaSuccess) {
    ctx->capture_stream = nullptr; record = false;
  }
  if (record && cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) record = false;
  if (!record) {
    cudaGetLastError();
    const mixaq_status result = forward(user_stream, false);
    if (result == MIXAQ_OK) cache.saw(std::move(key));
    return result;
  }
  const mixaq_status result = forward(ctx->capture_stream, true);
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  const bool recorded = cudaStreamEndCapture(ctx->capture_stream, &graph) == cudaSuccess && graph && result == MIXAQ_OK &&
                        cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
  if (graph) cudaGraphDestroy(graph);
  if (recorded) {
    if (cudaGraphLaunch(exec, user_stream) == cudaSuccess) {
      cache.recorded(std::move(key), exec, ctx->launches, cudaGraphExecDestroy);
      return MIXAQ_OK;
    }
    cudaGraphExecDestroy(exec);
  }
  cudaGetLastError();
  cache.not_recorded(key);
  return forward(user_stream, false);
}

extern "C" {

mixaq_status mixaq_block_forward(mixaq_ctx* ctx, const mixaq_block_params* p, const float* x, float* y,
                                 int B, int H, int W, float low_ratio, float prune_ratio,
                                 const mixaq_select_opts* opts, const mixaq_selection* sel_out,
                                 void* workspace, size_t workspace_bytes, const mixaq_taps* taps,
                                 void* cuda_stream) {
  const cudaStream_t user_stream = (cudaStream_t)cuda_stream;
  auto forward = [&](cudaStream_t st) {
    return block_forward_impl(ctx, p, x, y, B, H, W, low_ratio, prune_ratio, opts, sel_out, workspace, workspace_bytes,
                              taps, nullptr, st);
  };
  // A call repeated with the same arguments replays a graph: issuing its eleven launches and their tensor maps takes the
  // host longer than a small block takes the GPU (C = 96 at 56 x 56: 41 to 51 us a call without a replay, 31 with; C = 384 at
  // 50 x 84 with pruning, bound by the GPU but for the gaps between stream launches: 54.5 and 51.5).
  if (!ctx || !p || taps || !ctx->graph_cache || ctx->profiling || ctx->guards || ctx->nvtx) return forward(user_stream);
  if (caller_is_capturing(user_stream)) return forward(user_stream);
  std::string key;
  key.reserve(1024);
  KeyWriter k{key};
  k.val(x); k.val(y); k.val(workspace); k.val(workspace_bytes); k.val(user_stream);
  const int32_t* energy = opts ? opts->energy : nullptr;
  const int dims[5] = {B, H, W, opts ? opts->reverse : 0, sel_out ? 1 : 0};
  k.put(dims, sizeof(dims));
  k.val(energy); k.val(low_ratio); k.val(prune_ratio);
  if (sel_out) {
    const void* ptrs[6] = {sel_out->cls, sel_out->order, sel_out->score, sel_out->idx_hi, sel_out->idx_lo, sel_out->idx_pr};
    k.put(ptrs, sizeof(ptrs));
  }
  k.block(*p);
  std::lock_guard<std::mutex> lock(ctx->graph_lock);
  return replay_record_or_run(ctx, ctx->block_graphs, std::move(key), user_stream, "block_forward (graph launch)",
                              [&](cudaStream_t st, bool) { return forward(st); });
}

// -------------------------------------------------------------------------------------------------
size_t mixaq_merge_workspace_bytes(const mixaq_merge_params* p, int B, int H, int W) {
  if (!p || B <= 0 || H <= 0 || W <= 0) return 0;
  const size_t toks = (size_t)B * ((H + 1) / 2) * ((W + 1) / 2);
  return align_up(toks * p->reduction.in_features * p->in.bits / 8);
}

mixaq_status mixaq_merge_forward(mixaq_ctx* ctx, const mixaq_merge_params* p, const float* x, float* y,
                                 int B, int H, int W, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!ctx || !p) return MIXAQ_INVALID_ARG;
  if (!x || !y || !workspace || B <= 0 || H <= 0 || W <= 0) return fail(ctx, MIXAQ_INVALID_ARG, "merge: bad argument");
  if (!aligned_to(x, 16) || !aligned_to(y, 16) || !aligned_to(workspace, 256) || !aligned_to(p->prepared, 256) ||
      !aligned_to(p->reduction.codes, 16) || !aligned_to(p->ln_g, 16) || !aligned_to(p->ln_b, 16))
    return fail(ctx, MIXAQ_INVALID_ARG, "merge: x, y, weights and LayerNorm parameters must be 16-byte aligned, workspace and prepared 256-byte");
  const int K = p->reduction.in_features, N = p->reduction.out_features, C = K / 4;
  if (K % 4 || N % 32 || !merge_dim_supported(C)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "merge: unsupported dims");
  if (!p->ln_g || !p->ln_b || !p->reduction.codes || !p->reduction.scale || !p->prepared || !bits_ok(p->in.bits) ||
      !aq_ok(p->in, p->in.bits))
    return fail(ctx, MIXAQ_INVALID_ARG, "merge params incomplete");
  if (mixaq_merge_workspace_bytes(p, B, H, W) > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "merge workspace");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  g_launches = 0;
  const int M = B * ((H + 1) / 2) * ((W + 1) / 2);
  MergeGatherArgs mg;
  mg.x = x; mg.gamma = p->ln_g; mg.beta = p->ln_b; mg.out = (uint8_t*)workspace; mg.q = to_aq(p->in);
  mg.B = B; mg.H = H; mg.W = W; mg.C = C;
  { PROF(PC_MERGE_GATHER); launch_merge_gather(mg, st); }
  Carver c(p->prepared, false);
  float* mult = c.take<float>(N);
  int32_t* pre = c.take<int32_t>(N);
  float* bound = c.take<float>(N);
  GemmArgs ga;
  ga.status = ctx->d_status;
  ga.w = p->reduction.codes; ga.N = N; ga.K = K; ga.C = N; ga.mode = EPI_MERGE;
  fill_gemm_branch(ga.br[0], (const uint8_t*)workspace, M, p->in.bits, mult, pre, bound, nullptr);
  ga.br[0].out_f = y;
  fill_gemm_branch(ga.br[1], nullptr, 0, p->in.bits, mult, pre, bound, nullptr);
  { PROF(PC_MERGE_GEMM); if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)"); }
  ctx->launches = g_launches;
  return check_cuda(ctx, "merge_forward");
}

// -------------------------------------------------------------------------------------------------
namespace {
struct BackboneWs {
  float* scratch; int32_t* energy; void* merge; void* block; char* sel;
  float* tokens;            // patch-embedding output (only with p->embed)
  void* embed;              // patch-embedding workspace
  float* raw[16];           // un-normalised stage maps (only with output norms)
  size_t merge_bytes, block_bytes, sel_bytes, embed_bytes, bytes;
};
// H0, W0: size of the token map entering stage 1
BackboneWs carve_backbone(const mixaq_backbone_params* p, int B, int H0, int W0, int Hi, int Wi, void* base) {
  BackboneWs w; Carver c(base);
  size_t max_map = 0, max_tok = 0, max_merge = 0, max_block = 0, max_sel = 0;
  int H = H0, W = W0, blk = 0;
  const bool norms = p->out_norm_g && p->out_norm_b;
  for (int s = 0; s < p->num_stages; ++s) {
    if (s > 0) {
      max_merge = std::max(max_merge, mixaq_merge_workspace_bytes(&p->merges[s - 1], B, H, W));
      H = (H + 1) / 2; W = (W + 1) / 2;
    }
    const mixaq_block_params* b0 = &p->blocks[blk];
    max_map = std::max(max_map, (size_t)B * H * W * b0->dim);
    max_tok = std::max(max_tok, (size_t)B * H * W);
    for (int i = 0; i < p->depths[s]; ++i, ++blk)
      max_block = std::max(max_block, mixaq_block_workspace_bytes(&p->blocks[blk], B, H, W));
    max_sel = std::max(max_sel, (size_t)p->depths[s] * carve_sel(B, H, W, nullptr).bytes);   // one set per block of the stage
    w.raw[s] = (norms && s < 16) ? c.take<float>((size_t)B * H * W * b0->dim) : nullptr;
  }
  w.scratch = c.take<float>(max_map);
  w.energy = c.take<int32_t>(max_tok);
  w.merge = c.take<uint8_t>(max_merge); w.merge_bytes = align_up(max_merge);
  w.block = c.take<uint8_t>(max_block); w.block_bytes = align_up(max_block);
  w.sel = (char*)c.take<uint8_t>(max_sel); w.sel_bytes = align_up(max_sel);
  w.tokens = nullptr; w.embed = nullptr; w.embed_bytes = 0;
  if (p->embed) {
    w.tokens = c.take<float>((size_t)B * H0 * W0 * p->blocks[0].dim);
    const size_t eb = mixaq_embed_workspace_bytes(p->embed, B, Hi, Wi);
    w.embed = c.take<uint8_t>(eb); w.embed_bytes = align_up(eb);
  }
  w.bytes = c.off;
  return w;
}
}  // namespace

// ---- the walk over a backbone -------------------------------------------------------------------------------------------
namespace {
// a validated backbone call; H0 x W0 is the token map of stage 1, Hi x Wi the size that the caller gave
struct BackboneCall {
  const mixaq_backbone_params* p;
  const float* x0; float* const* stage_out;
  int B, H0, W0, Hi, Wi;
  const float *low, *prune;              // per pair; prune nullable
  BackboneWs ws;
};

// Issues every launch of the call on `st`.  recording: the stream is being captured into a graph that will be kept.
mixaq_status issue_backbone(mixaq_ctx* ctx, const BackboneCall& c, bool recording, cudaStream_t st) {
  const mixaq_backbone_params* p = c.p;
  const BackboneWs& ws = c.ws;
  const int B = c.B;
  const bool norms = p->out_norm_g && p->out_norm_b;
  // Inside a recorded forward the output norms leave the chain: nothing waits for them but the end of the forward.
  bool side = recording && norms;
  if (side && !ctx->side_stream) {
    if (cudaStreamCreateWithFlags(&ctx->side_stream, cudaStreamNonBlocking) != cudaSuccess) { ctx->side_stream = nullptr; side = false; }
    else if (cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming) != cudaSuccess ||
             cudaEventCreateWithFlags(&ctx->join, cudaEventDisableTiming) != cudaSuccess) {
      cudaStreamDestroy(ctx->side_stream); ctx->side_stream = nullptr; side = false;
    }
    if (!side) cudaGetLastError();
  }
  mixaq_status result = MIXAQ_OK;
  int total = 0, H = c.H0, W = c.W0, blk = 0;
  const float* cur = c.x0;
  // while profiling: a few event pairs with nothing between them, so that what a bracket itself adds to every kernel's
  // time can be read off the same record
  if (ctx->profiling) for (int i = 0; i < 4; ++i) { PROF(PC_BRACKET); }
  if (p->embed) {
    // image -> token map of stage 1 (patch embedding), inside the same captured graph
    result = mixaq_embed_forward(ctx, p->embed, c.x0, ws.tokens, B, c.Hi, c.Wi, ws.embed, ws.embed_bytes, st);
    total += ctx->launches;
    cur = ws.tokens;
  }
  for (int s = 0; s < p->num_stages && result == MIXAQ_OK; ++s) {
    NvtxScope stage_range(ctx, "stage", s + 1);
    const int d = p->depths[s];
    // with output norms the un-normalised map stays in the workspace (the next stage reads it) and the caller's
    // buffer receives its LayerNorm
    float* out_s = norms ? ws.raw[s] : c.stage_out[s];
    if (s > 0) {
      // the merge writes where the first block of the stage does NOT write
      float* mdst = (d % 2 == 0) ? out_s : ws.scratch;
      result = mixaq_merge_forward(ctx, &p->merges[s - 1], cur, mdst, B, H, W, ws.merge, ws.merge_bytes, st);
      if (result != MIXAQ_OK) break;
      total += ctx->launches;
      cur = mdst; H = (H + 1) / 2; W = (W + 1) / 2;
    }
    // importance is scored once per stage, before its first block (Section 3.2): one energy map, and from it the
    // window classes and batch bookkeeping of EVERY block of the stage (own shift, own pair's ratios) in one go
    const mixaq_block_params* b0 = &p->blocks[blk];
    { PROF(PC_ENERGY); launch_energy(cur, ws.energy, (long)B * H * W, b0->dim, b0->score_inv_scale, st); }
    total += 1;
    const size_t sel_stride = carve_sel(B, H, W, nullptr).bytes;
    std::vector<SelWs> sels(d);
    std::vector<SelectArgs> sargs(d);
    // Windows keep their precision class within a stage (Section 4.4, "Windows Elevation"): unless elevation is
    // allowed, a pair's effective ratios are the largest ratios of the stage's pairs so far.
    std::vector<float> lr_eff(d), pr_eff(d);
    float lmax = 0.f, pmax = 0.f;
    for (int i = 0; i < d; ++i) {
      float lr = c.low[(blk + i) / 2], pr = c.prune ? c.prune[(blk + i) / 2] : 0.f;
      if (!ctx->allow_elevation) { lmax = std::max(lmax, lr); pmax = std::max(pmax, pr); lr = lmax; pr = pmax; }
      lr_eff[i] = lr; pr_eff[i] = pr;
    }
    for (int i = 0; i < d; ++i) {
      const float lr = lr_eff[i], pr = pr_eff[i];
      Geometry g = geometry(H, W, lr, pr);
      if ((size_t)g.nW * 8 > 48 * 1024) { result = fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "too many windows per image (max 6144)"); break; }
      sels[i] = carve_sel(B, H, W, ws.sel + (size_t)i * sel_stride);
      sargs[i] = make_select_args(sels[i], ws.energy, B, H, W, p->blocks[blk + i].shift, g, ctx->reverse_selection ? 1 : 0, true);
    }
    if (result != MIXAQ_OK) break;
    g_launches = 0;
    { PROF(PC_SELECT); launch_select(sargs.data(), d, st); }
    total += g_launches;
    for (int i = 0; i < d; ++i, ++blk) {
      float* dst = ((d - 1 - i) % 2 == 0) ? out_s : ws.scratch;
      NvtxScope block_range(ctx, "block", blk);
      result = block_forward_impl(ctx, &p->blocks[blk], cur, dst, B, H, W, lr_eff[i], pr_eff[i], nullptr, nullptr,
                                  ws.block, ws.block_bytes, nullptr, &sels[i], st);
      if (result != MIXAQ_OK) break;
      total += ctx->launches;
      cur = dst;
    }
    if (result == MIXAQ_OK && norms) {
      PROF(PC_OUT_NORM);
      g_launches = 0;
      if (side) { cudaEventRecord(ctx->fork, st); cudaStreamWaitEvent(ctx->side_stream, ctx->fork, 0); }
      if (!launch_bias_ln(out_s, nullptr, p->out_norm_g[s], p->out_norm_b[s], c.stage_out[s], (long)B * H * W, b0->dim,
                          side ? ctx->side_stream : st))
        result = fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "output norm: unsupported width");
      total += g_launches;
    }
  }
  if (side) { cudaEventRecord(ctx->join, ctx->side_stream); cudaStreamWaitEvent(st, ctx->join, 0); }
  if (result != MIXAQ_OK) return result;
  ctx->launches = total;
  return check_cuda(ctx, "backbone_forward");
}

// A profiled forward on a capturable stream is captured too, with the event records around its kernels as graph nodes,
// launched once and not kept: the kernels are then timed as they run inside a graph, not with a stream launch between the
// events.  On the legacy stream the launches are profiled as they are.
mixaq_status profile_backbone(mixaq_ctx* ctx, const BackboneCall& c, cudaStream_t st) {
  if (is_legacy(st) || cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return issue_backbone(ctx, c, false, st);
  }
  ctx->prof_capture = true;
  const mixaq_status result = issue_backbone(ctx, c, false, st);
  ctx->prof_capture = false;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  const cudaError_t e = cudaStreamEndCapture(st, &graph);
  if (result != MIXAQ_OK) { if (graph) cudaGraphDestroy(graph); cudaGetLastError(); return result; }
  if (e != cudaSuccess || !graph || cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return check_cuda(ctx, "backbone_forward (graph capture)") == MIXAQ_OK
               ? fail(ctx, MIXAQ_CUDA_ERROR, "backbone_forward: graph capture failed") : MIXAQ_CUDA_ERROR;
  }
  cudaGraphDestroy(graph);
  ctx->prof_execs.push_back(exec);
  if (cudaGraphLaunch(exec, st) != cudaSuccess) return check_cuda(ctx, "backbone_forward (graph launch)");
  return MIXAQ_OK;
}
}  // namespace

size_t mixaq_backbone_workspace_bytes(const mixaq_backbone_params* p, int B, int H0, int W0) {
  if (!p || !p->depths || !p->blocks || p->num_stages <= 0 || p->num_stages > 16 || B <= 0 || H0 <= 0 || W0 <= 0) return 0;
  if (p->num_stages > 1 && !p->merges) return 0;
  const int Ht = p->embed ? (H0 + 3) / 4 : H0, Wt = p->embed ? (W0 + 3) / 4 : W0;
  return carve_backbone(p, B, Ht, Wt, H0, W0, nullptr).bytes;
}

mixaq_status mixaq_backbone_forward(mixaq_ctx* ctx, const mixaq_backbone_params* p, const float* x0,
                                    float* const* stage_out, int B, int H0, int W0,
                                    const float* low_ratio_per_pair, const float* prune_ratio_per_pair,
                                    void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (!p || !p->depths || !p->blocks || p->num_stages <= 0 || (p->num_stages > 1 && !p->merges))
    return fail(ctx, MIXAQ_INVALID_ARG, "backbone params incomplete");
  if (!x0 || !stage_out || !low_ratio_per_pair || !workspace || B <= 0 || H0 <= 0 || W0 <= 0)
    return fail(ctx, MIXAQ_INVALID_ARG, "backbone: bad argument");
  if (!aligned_to(x0, 16) || !aligned_to(workspace, 256))
    return fail(ctx, MIXAQ_INVALID_ARG, "backbone: x0 must be 16-byte aligned, the workspace 256-byte");
  if (p->num_stages > 16) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "at most 16 stages");
  if ((p->out_norm_g != nullptr) != (p->out_norm_b != nullptr)) return fail(ctx, MIXAQ_INVALID_ARG, "output norms need gamma and beta");
  const bool norms = p->out_norm_g && p->out_norm_b;
  if (norms)
    for (int s = 0; s < p->num_stages; ++s)
      if (!p->out_norm_g[s] || !p->out_norm_b[s]) return fail(ctx, MIXAQ_INVALID_ARG, "output norm parameters of a stage are NULL");
  if (p->embed && (!p->embed->prepared || p->embed->proj.out_features != p->blocks[0].dim))
    return fail(ctx, MIXAQ_INVALID_ARG, "embed: not prepared, or its width differs from the first stage's");
  // with a patch embedding in front, H0 x W0 is the image; the token map of stage 1 is a quarter of it
  const int Hi = H0, Wi = W0;
  if (p->embed) { H0 = (Hi + 3) / 4; W0 = (Wi + 3) / 4; }
  int nblk = 0;
  for (int s = 0; s < p->num_stages; ++s) {
    if (p->depths[s] <= 0 || (p->depths[s] != 1 && p->depths[s] % 2)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "depths must be even or 1");
    if (!stage_out[s]) return fail(ctx, MIXAQ_INVALID_ARG, "stage_out entry is NULL");
    if (!aligned_to(stage_out[s], 16)) return fail(ctx, MIXAQ_INVALID_ARG, "stage_out entries must be 16-byte aligned");
    nblk += p->depths[s];
  }
  for (int b = 0; b < nblk; ++b) {
    mixaq_status s = validate_block(ctx, &p->blocks[b]);
    if (s != MIXAQ_OK) return s;
    float r = low_ratio_per_pair[b / 2], q = prune_ratio_per_pair ? prune_ratio_per_pair[b / 2] : 0.f;
    if (!(r >= 0.f && r <= 1.f) || !(q >= 0.f && q <= 1.f)) return fail(ctx, MIXAQ_INVALID_ARG, "ratios must lie in [0, 1]");
  }
  BackboneWs ws = carve_backbone(p, B, H0, W0, Hi, Wi, workspace);
  if (ws.bytes > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "backbone workspace too small");
  const BackboneCall call = {p, x0, stage_out, B, H0, W0, Hi, Wi, low_ratio_per_pair, prune_ratio_per_pair, ws};
  const cudaStream_t user_stream = (cudaStream_t)cuda_stream;
  if (!ctx->graph_cache) return issue_backbone(ctx, call, false, user_stream);
  std::lock_guard<std::mutex> lock(ctx->graph_lock);
  if (caller_is_capturing(user_stream)) return issue_backbone(ctx, call, false, user_stream);
  if (ctx->profiling) return profile_backbone(ctx, call, user_stream);
  // guard zones and NVTX ranges are asked for on the calls that follow: a graph recorded before does not have them
  if (ctx->guards || ctx->nvtx) return issue_backbone(ctx, call, false, user_stream);

  std::string key;
  KeyWriter k{key};
  const int npairs = (nblk + 1) / 2;
  // what changes from call to call comes first: two keys that differ are then told apart by their first bytes
  k.val(x0); k.put(stage_out, sizeof(float*) * p->num_stages);
  k.val(workspace); k.val(workspace_bytes); k.val(user_stream);
  const int dims[5] = {B, H0, W0, Hi, Wi};
  k.put(dims, sizeof(dims));
  k.put(low_ratio_per_pair, sizeof(float) * npairs);
  const char flags = (p->embed ? 1 : 0) | (norms ? 2 : 0) | (prune_ratio_per_pair ? 4 : 0) | (ctx->allow_elevation ? 8 : 0) |
                     (ctx->reverse_selection ? 16 : 0);
  k.val(flags);
  if (prune_ratio_per_pair) k.put(prune_ratio_per_pair, sizeof(float) * npairs);
  k.val(p->num_stages); k.put(p->depths, sizeof(int) * p->num_stages);
  for (int b = 0; b < nblk; ++b) k.block(p->blocks[b]);
  for (int m = 0; m + 1 < p->num_stages; ++m) {
    const mixaq_merge_params& q = p->merges[m];
    k.val(q.ln_g); k.val(q.ln_b); k.aq(q.in); k.linear(q.reduction); k.val(q.prepared);
  }
  if (p->embed) {
    const mixaq_embed_params& q = *p->embed;
    k.val(q.ln_g); k.val(q.ln_b); k.val(q.bias); k.aq(q.in); k.linear(q.proj); k.val(q.prepared);
  }
  if (norms) { k.put(p->out_norm_g, sizeof(float*) * p->num_stages); k.put(p->out_norm_b, sizeof(float*) * p->num_stages); }
  return replay_record_or_run(ctx, ctx->graphs, std::move(key), user_stream, "backbone_forward (graph launch)",
                              [&](cudaStream_t st, bool recording) { return issue_backbone(ctx, call, recording, st); });
}

// -------------------------------------------------------------------------------------------------
// stem and output norms
namespace {
constexpr int EMBED_K = 48, EMBED_KP = 64;     // patch vector, padded to a multiple of 32 codes
struct EmbedPrepared { int8_t* w; float* mult; int32_t* pre; float* bound; size_t bytes; };
EmbedPrepared carve_embed(const mixaq_embed_params* p, void* base) {
  EmbedPrepared r; Carver c(base, false);
  const int N = p->proj.out_features;
  r.w = c.take<int8_t>((size_t)N * EMBED_KP); r.mult = c.take<float>(N); r.pre = c.take<int32_t>(N); r.bound = c.take<float>(N);
  r.bytes = c.off;
  return r;
}
bool embed_ok(const mixaq_embed_params* p) {
  return p && p->ln_g && p->ln_b && p->bias && p->proj.codes && p->proj.scale && p->proj.in_features == EMBED_K &&
         p->proj.out_features > 0 && p->proj.out_features % 32 == 0 && ln_dim_supported(p->proj.out_features) &&
         bits_ok(p->in.bits) && aq_ok(p->in, p->in.bits) && p->in.bits == 8;
}
}  // namespace

size_t mixaq_embed_prepared_bytes(const mixaq_embed_params* p) {
  if (!p || p->proj.out_features <= 0) return 0;
  return carve_embed(p, nullptr).bytes;
}

mixaq_status mixaq_embed_prepare(mixaq_ctx* ctx, const mixaq_embed_params* p, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (!embed_ok(p) || !p->prepared) return fail(ctx, MIXAQ_INVALID_ARG, "embed params incomplete (8-bit input, [C0][48] projection, C0 % 32 == 0)");
  if (!all_aligned_to(4, {p->prepared, p->proj.scale}))
    return fail(ctx, MIXAQ_INVALID_ARG, "embed: step sizes and prepared must be 4-byte aligned");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  EmbedPrepared pr = carve_embed(p, p->prepared);
  const int N = p->proj.out_features;
  launch_pad_weights(p->proj.codes, N, EMBED_K, EMBED_KP, pr.w, st);
  launch_prepare_linear(pr.w, p->proj.scale, N, EMBED_KP, p->in.scale, p->in.zero_point, p->in.bits, pr.mult, pr.pre, pr.bound, st);
  return check_cuda(ctx, "embed_prepare");
}

size_t mixaq_embed_workspace_bytes(const mixaq_embed_params* p, int B, int Hi, int Wi) {
  if (!p || B <= 0 || Hi <= 0 || Wi <= 0 || p->proj.out_features <= 0) return 0;
  const size_t toks = (size_t)B * ((Hi + 3) / 4) * ((Wi + 3) / 4);
  return carved_bytes(toks * EMBED_KP) + carved_bytes(toks * p->proj.out_features * sizeof(float));
}

mixaq_status mixaq_embed_forward(mixaq_ctx* ctx, const mixaq_embed_params* p, const float* image, float* x0,
                                 int B, int Hi, int Wi, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (!embed_ok(p) || !p->prepared) return fail(ctx, MIXAQ_INVALID_ARG, "embed params incomplete");
  if (!image || !x0 || !workspace || B <= 0 || Hi <= 0 || Wi <= 0) return fail(ctx, MIXAQ_INVALID_ARG, "embed: bad argument");
  if (!aligned_to(image, 4) || !aligned_to(x0, 16) || !aligned_to(workspace, 256) || !aligned_to(p->prepared, 256) ||
      !aligned_to(p->ln_g, 16) || !aligned_to(p->ln_b, 16) || !aligned_to(p->bias, 16))
    return fail(ctx, MIXAQ_INVALID_ARG, "embed: x0 and parameters must be 16-byte aligned, workspace and prepared 256-byte");
  if (mixaq_embed_workspace_bytes(p, B, Hi, Wi) > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "embed workspace");
  const size_t toks = (size_t)B * ((Hi + 3) / 4) * ((Wi + 3) / 4);
  if (toks >= (size_t)1 << 31) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "too many tokens");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int N = p->proj.out_features;
  Carver c(workspace);
  uint8_t* codes = c.take<uint8_t>(toks * EMBED_KP);
  float* t = c.take<float>(toks * N);
  EmbedPrepared pr = carve_embed(p, p->prepared);
  g_launches = 0;
  PatchGatherArgs pg; pg.img = image; pg.out = codes; pg.q = to_aq(p->in); pg.B = B; pg.Hi = Hi; pg.Wi = Wi;
  PROF(PC_STEM);
  launch_patch_gather(pg, st);
  GemmArgs ga;
  ga.status = ctx->d_status;
  ga.w = pr.w; ga.N = N; ga.K = EMBED_KP; ga.C = N; ga.mode = EPI_MERGE;      // dequantize only: acc * mult
  fill_gemm_branch(ga.br[0], codes, (int)toks, 8, pr.mult, pr.pre, pr.bound, nullptr);
  ga.br[0].out_f = t;
  fill_gemm_branch(ga.br[1], nullptr, 0, 8, pr.mult, pr.pre, pr.bound, nullptr);
  if (!launch_gemm(ga, st)) return fail(ctx, MIXAQ_INTERNAL, "GEMM launch set-up failed (tensor map / tile shape)");
  if (!launch_bias_ln(t, p->bias, p->ln_g, p->ln_b, x0, (long)toks, N, st)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "embed: unsupported C0");
  ctx->launches = g_launches;
  return check_cuda(ctx, "embed_forward");
}

mixaq_status mixaq_norm_forward(mixaq_ctx* ctx, const float* gamma, const float* beta, const float* x, float* y,
                                long rows, int C, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  if (!gamma || !beta || !x || !y || rows <= 0 || C <= 0) return fail(ctx, MIXAQ_INVALID_ARG, "norm: bad argument");
  if (!aligned_to(gamma, 16) || !aligned_to(beta, 16) || !aligned_to(x, 16) || !aligned_to(y, 16))
    return fail(ctx, MIXAQ_INVALID_ARG, "norm: pointers must be 16-byte aligned");
  g_launches = 0;
  if (!launch_bias_ln(x, nullptr, gamma, beta, y, rows, C, (cudaStream_t)cuda_stream))
    return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "norm: unsupported C");
  ctx->launches = g_launches;
  return check_cuda(ctx, "norm_forward");
}

mixaq_status mixaq_set_reverse_selection(mixaq_ctx* ctx, int reverse) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  ctx->reverse_selection = reverse != 0;
  return MIXAQ_OK;
}

mixaq_status mixaq_set_workspace_guards(mixaq_ctx* ctx, int enabled) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  ctx->guards = enabled != 0;
  return MIXAQ_OK;
}

mixaq_status mixaq_selftest_workspace_guards(mixaq_ctx* ctx, void* buffer, size_t bytes, int overrun, void* cuda_stream) {
  if (!ctx || !buffer || bytes < 4 * (size_t)(256 + GUARD_BYTES)) return MIXAQ_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  std::vector<void*> zones;
  uint8_t* second = nullptr;
  {
    const bool was = ctx->guards;
    ctx->guards = true;
    GuardScope gs(ctx, &zones);
    Carver c(buffer);
    c.take<uint8_t>(256);
    second = c.take<uint8_t>(256);
    ctx->guards = was;
  }
  launch_guards(zones.data(), (int)zones.size(), true, ctx->d_status, st);
  // a writer that runs one byte past the end of the second buffer (an ordinary write inside the caller's memory)
  if (overrun) cudaMemsetAsync(second + 256, 0, 1, st);
  launch_guards(zones.data(), (int)zones.size(), false, ctx->d_status, st);
  return check_cuda(ctx, "selftest_workspace_guards");
}

mixaq_status mixaq_set_nvtx(mixaq_ctx* ctx, int enabled) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  ctx->nvtx = enabled != 0;
  return MIXAQ_OK;
}

mixaq_status mixaq_set_window_elevation(mixaq_ctx* ctx, int allow) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  ctx->allow_elevation = allow != 0;
  return MIXAQ_OK;
}

mixaq_status mixaq_set_graph_cache(mixaq_ctx* ctx, int enabled) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  std::lock_guard<std::mutex> lock(ctx->graph_lock);
  ctx->graph_cache = enabled != 0;
  if (!enabled) {
    ctx->graphs.clear(cudaGraphExecDestroy);
    ctx->block_graphs.clear(cudaGraphExecDestroy);
  }
  return MIXAQ_OK;
}

// -------------------------------------------------------------------------------------------------
// calibration (Section 4.3)
namespace {
struct CalWs { int32_t *rowsrc, *expo; float *ln, *qkv, *o, *x1, *h; uint8_t *slices, *slices_fc2; uint32_t* obs; size_t bytes; };
CalWs carve_cal(const mixaq_block_params* p, int B, int H, int W, void* base) {
  CalWs w; Carver c(base);
  Geometry g = geometry(H, W, 0.f, 0.f);
  const size_t M = (size_t)B * g.nW * WT;
  w.obs = c.take<uint32_t>(CAL_OBS);
  w.rowsrc = c.take<int32_t>(M);
  w.expo = c.take<int32_t>(M);
  w.x1 = c.take<float>(M * p->dim); w.h = c.take<float>(M * p->hidden);
  // fc2's byte planes, which are the largest, start where the inputs of the products before it lay: 48 C bytes a row at hidden = 4 C
  // (68 C with a place of their own, 40 C for the arrays that are not planes)
  const size_t shared = c.off;
  w.ln = c.take<float>(M * p->dim); w.qkv = c.take<float>(M * 3 * p->dim); w.o = c.take<float>(M * p->dim);
  const size_t planes = CAL_SLICES * M * p->dim, planes_fc2 = CAL_SLICES * M * p->hidden, dead = c.off - shared;
  w.slices_fc2 = reinterpret_cast<uint8_t*>(w.ln);
  w.slices = c.take<uint8_t>(std::max(planes, planes_fc2 > dead ? planes_fc2 - dead : 0));
  w.bytes = c.off;
  return w;
}
// reads the observers' keys and the call's status back (synchronises) and decodes them
mixaq_status read_ranges(mixaq_ctx* ctx, const uint32_t* d_obs, int sites, mixaq_range* out, cudaStream_t st) {
  uint32_t keys[CAL_OBS];
  if (cudaMemcpyAsync(keys, d_obs, sizeof(keys), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) return check_cuda(ctx, "calibrate (read ranges)") == MIXAQ_OK ? MIXAQ_CUDA_ERROR : MIXAQ_CUDA_ERROR;
  if (keys[CAL_STATUS]) return fail(ctx, MIXAQ_DEVICE_TIMEOUT, "calibrate: a bounded wait inside a product ran out");
  for (int i = 0; i < sites; ++i) { out[i].lo = cal_key_to_float(keys[2 * i]); out[i].hi = cal_key_to_float(keys[2 * i + 1]); }
  return MIXAQ_OK;
}
}  // namespace

size_t mixaq_calibrate_block_workspace_bytes(const mixaq_block_params* p, int B, int H, int W) {
  if (!p || B <= 0 || H <= 0 || W <= 0 || p->dim <= 0 || p->hidden <= 0) return 0;
  return carve_cal(p, B, H, W, nullptr).bytes;
}

mixaq_status mixaq_calibrate_block(mixaq_ctx* ctx, const mixaq_block_params* p, int branch, const float* x, float* y,
                                   int B, int H, int W, mixaq_block_ranges* ranges,
                                   void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!ctx) return MIXAQ_INVALID_ARG;
  mixaq_status s = validate_block(ctx, p, false);
  if (s != MIXAQ_OK) return s;
  if (!x || !y || x == y || !ranges || !workspace || B <= 0 || H <= 0 || W <= 0 || (branch != 0 && branch != 1))
    return fail(ctx, MIXAQ_INVALID_ARG, "calibrate_block: bad argument");
  if (!aligned_to(x, 16) || !aligned_to(y, 16) || !aligned_to(workspace, 256))
    return fail(ctx, MIXAQ_INVALID_ARG, "calibrate_block: x and y must be 16-byte aligned, the workspace 256-byte");
  if ((long)B * H * W >= (1L << 31) / WT) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "too many tokens");
  CalWs ws = carve_cal(p, B, H, W, workspace);
  if (ws.bytes > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "calibrate_block workspace too small");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const mixaq_branch& br = branch == 0 ? p->hi : p->lo;
  CalBlockArgs c;
  c.x = x; c.y = y; c.B = B; c.H = H; c.W = W; c.C = p->dim; c.heads = p->heads; c.hidden = p->hidden; c.shift = p->shift;
  c.ln1_g = br.ln1_g; c.ln1_b = br.ln1_b; c.ln2_g = br.ln2_g; c.ln2_b = br.ln2_b;
  c.b_qkv = br.b_qkv; c.b_proj = br.b_proj; c.b_fc1 = br.b_fc1; c.b_fc2 = br.b_fc2;
  c.w_qkv = p->qkv.codes; c.w_proj = p->proj.codes; c.w_fc1 = p->fc1.codes; c.w_fc2 = p->fc2.codes;
  c.s_qkv = p->qkv.scale; c.s_proj = p->proj.scale; c.s_fc1 = p->fc1.scale; c.s_fc2 = p->fc2.scale; c.relpos = p->relpos_table;
  c.rowsrc = ws.rowsrc; c.ln = ws.ln; c.qkv = ws.qkv; c.o = ws.o; c.x1 = ws.x1; c.h = ws.h; c.obs = ws.obs;
  c.slices = ws.slices; c.slices_fc2 = ws.slices_fc2; c.expo = ws.expo; c.status = ctx->d_status;
  g_launches = 0;
  if (!launch_calibrate_block(c, st)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "calibrate_block: unsupported dim");
  ctx->launches = g_launches;
  s = check_cuda(ctx, "calibrate_block");
  if (s != MIXAQ_OK) return s;
  return read_ranges(ctx, ws.obs, 8, &ranges->qkv_in, st);
}

size_t mixaq_calibrate_merge_workspace_bytes(const mixaq_merge_params* p, int B, int H, int W) {
  if (!p || B <= 0 || H <= 0 || W <= 0 || p->reduction.in_features <= 0) return 0;
  const size_t toks = (size_t)B * ((H + 1) / 2) * ((W + 1) / 2);
  return carved_bytes(CAL_OBS * sizeof(uint32_t)) + carved_bytes(toks * p->reduction.in_features * sizeof(float)) +
         carved_bytes(toks * sizeof(int32_t)) + carved_bytes(CAL_SLICES * toks * p->reduction.in_features);
}

mixaq_status mixaq_calibrate_merge(mixaq_ctx* ctx, const mixaq_merge_params* p, const float* x, float* y,
                                   int B, int H, int W, mixaq_range* range,
                                   void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!ctx || !p) return MIXAQ_INVALID_ARG;
  if (!x || !y || !range || !workspace || B <= 0 || H <= 0 || W <= 0) return fail(ctx, MIXAQ_INVALID_ARG, "calibrate_merge: bad argument");
  if (!aligned_to(x, 16) || !aligned_to(y, 16) || !aligned_to(workspace, 256) || !aligned_to(p->reduction.codes, 16))
    return fail(ctx, MIXAQ_INVALID_ARG, "calibrate_merge: x, y and weights must be 16-byte aligned, the workspace 256-byte");
  const int K = p->reduction.in_features, N = p->reduction.out_features, C = K / 4;
  if (K % 4 || N <= 0 || !merge_dim_supported(C)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "calibrate_merge: unsupported dims");
  if (!p->ln_g || !p->ln_b || !p->reduction.codes || !p->reduction.scale) return fail(ctx, MIXAQ_INVALID_ARG, "merge params incomplete");
  if (!all_aligned_to(4, {p->ln_g, p->ln_b, p->reduction.scale}))
    return fail(ctx, MIXAQ_INVALID_ARG, "calibrate_merge: LayerNorm parameters and step sizes must be 4-byte aligned");
  if (mixaq_calibrate_merge_workspace_bytes(p, B, H, W) > workspace_bytes) return fail(ctx, MIXAQ_WORKSPACE_TOO_SMALL, "calibrate_merge workspace");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Carver cv(workspace);
  CalMergeArgs c;
  c.obs = cv.take<uint32_t>(CAL_OBS);
  const size_t toks = (size_t)B * ((H + 1) / 2) * ((W + 1) / 2);
  c.ln = cv.take<float>(toks * K);
  c.expo = cv.take<int32_t>(toks); c.slices = cv.take<uint8_t>(CAL_SLICES * toks * K);
  c.x = x; c.y = y; c.B = B; c.H = H; c.W = W; c.C = C; c.N = N;
  c.ln_g = p->ln_g; c.ln_b = p->ln_b; c.w = p->reduction.codes; c.sw = p->reduction.scale; c.status = ctx->d_status;
  g_launches = 0;
  if (!launch_calibrate_merge(c, st)) return fail(ctx, MIXAQ_UNSUPPORTED_SHAPE, "calibrate_merge: unsupported dim");
  ctx->launches = g_launches;
  mixaq_status s = check_cuda(ctx, "calibrate_merge");
  if (s != MIXAQ_OK) return s;
  return read_ranges(ctx, c.obs, 1, range, st);
}

mixaq_status mixaq_aq_from_range(float lo, float hi, int bits, mixaq_aq* out) {
  if (!out || !bits_ok(bits) || !(hi > lo)) return MIXAQ_INVALID_ARG;
  const int qmax = (1 << bits) - 1;
  out->bits = bits;
  out->scale = (float)(((double)hi - (double)lo) / (double)qmax);
  out->inv_scale = 1.0f / out->scale;
  double z = std::nearbyint(-(double)lo / (double)out->scale);
  out->zero_point = (int)std::fmin(std::fmax(z, 0.0), (double)qmax);
  return MIXAQ_OK;
}

}  // extern "C"
