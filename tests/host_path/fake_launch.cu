// The kernel launchers of the stand-in: they count their launch on its stream.
#include "../../paper_2507_19131_b200/csrc/kernels.h"
#include "fake.h"
#include <initializer_list>

extern "C" {
mixaq::SelectArgs last_select;
struct Range { const void* at; size_t bytes; int code_bits; };      // code_bits: 0 for binary32
Range written[256]; int written_count;                              // what the kernels since fake_reset write, guard zones apart
const void* last_calibration[10];
const void* guard_zones[64]; int guard_count;                       // the zones of the last check
}
static void note(const void* at, size_t elements, int bits) {
  if (elements && written_count < 256) written[written_count++] = {at, elements * (bits ? bits : 32) / 8, bits};
}

namespace mixaq {
#define LAUNCH(st) do { ++g_launches; enqueue(st); } while (0)
bool gemm_init() { return true; }
bool ln_init() { return true; }
bool ln_dim_supported(int C) { return C % 32 == 0; }
bool merge_dim_supported(int C) { return C % 32 == 0; }
void launch_energy(const float*, int32_t*, long, int, float, cudaStream_t st) { LAUNCH(st); }
void launch_select(const SelectArgs* a, int, cudaStream_t st) { last_select = a[0]; LAUNCH(st); }
void launch_class_lists(const uint8_t*, int, int, int32_t* const*, const int*, cudaStream_t st) { LAUNCH(st); }
void launch_ln_quant(const LnBranch& hi, const LnBranch& lo, int C, cudaStream_t st) {
  for (const LnBranch* b : {&hi, &lo}) note(b->out, (size_t)b->M * C, b->q.bits);
  LAUNCH(st);
}
void launch_merge_gather(const MergeGatherArgs&, cudaStream_t st) { LAUNCH(st); }
void launch_guards(void* const* zones, int count, bool, int*, cudaStream_t st) {
  guard_count = count < 64 ? count : 64;
  for (int i = 0; i < guard_count; ++i) guard_zones[i] = zones[i];
  ++counts.guard_launches; enqueue(st);
}
void launch_copy_rows(const float*, float*, const int32_t*, int, int, cudaStream_t st) { LAUNCH(st); }
void launch_patch_gather(const PatchGatherArgs&, cudaStream_t st) { LAUNCH(st); }
bool launch_bias_ln(const float*, const float*, const float*, const float*, float*, long, int, cudaStream_t st) { LAUNCH(st); return true; }
void launch_pad_weights(const int8_t*, int, int, int, int8_t*, cudaStream_t st) { LAUNCH(st); }
bool launch_gemm(const GemmArgs& g, cudaStream_t st) {
  for (const GemmBranch& b : g.br) {
    if (g.mode == EPI_QKV || g.mode == EPI_FC1) note(b.out_codes, (size_t)b.M * g.N, b.out_bits);
    else if (g.mode == EPI_PROJ) note(b.out_f, (size_t)b.M * g.N, 0);           // (fc2 writes the caller's map)
  }
  LAUNCH(st); return true;
}
void launch_attention(const AttnArgs& a, cudaStream_t st) {
  for (const AttnBranch& b : a.br) note(b.out, (size_t)b.slots * WT * a.C, b.cbits);
  LAUNCH(st);
}
void launch_prepare_linear(const int8_t*, const float*, int, int, float, int, int, float*, int32_t*, float*, cudaStream_t st) { LAUNCH(st); }
void launch_prepare_relbias(const float*, int, float*, cudaStream_t st) { LAUNCH(st); }
void launch_wait_probe(int*, cudaStream_t st) { LAUNCH(st); }
int launch_mma_peak(int, int, unsigned long long*, int*, cudaStream_t) { return 0; }
bool launch_calibrate_block(const CalBlockArgs& c, cudaStream_t st) {
  const void* at[10] = {c.obs, c.rowsrc, c.expo, c.x1, c.h, c.ln, c.qkv, c.o, c.slices, c.slices_fc2};
  for (int i = 0; i < 10; ++i) last_calibration[i] = at[i];
  LAUNCH(st); return true;
}
bool launch_calibrate_merge(const CalMergeArgs&, cudaStream_t st) { LAUNCH(st); return true; }
float cal_key_to_float(uint32_t) { return 0.f; }
}  // namespace mixaq
