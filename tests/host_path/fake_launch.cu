// The kernel launchers of the stand-in: they count their launch on its stream.
#include "../../paper_2507_19131_b200/csrc/kernels.h"
#include "fake.h"

extern "C" { mixaq::SelectArgs last_select; }

namespace mixaq {
#define LAUNCH(st) do { ++g_launches; enqueue(st); } while (0)
bool gemm_init() { return true; }
bool ln_init() { return true; }
bool ln_dim_supported(int C) { return C % 32 == 0; }
bool merge_dim_supported(int C) { return C % 32 == 0; }
void launch_energy(const float*, int32_t*, long, int, float, cudaStream_t st) { LAUNCH(st); }
void launch_select(const SelectArgs* a, int, cudaStream_t st) { last_select = a[0]; LAUNCH(st); }
void launch_class_lists(const uint8_t*, int, int, int32_t* const*, const int*, cudaStream_t st) { LAUNCH(st); }
void launch_ln_quant(const LnBranch&, const LnBranch&, int, cudaStream_t st) { LAUNCH(st); }
void launch_merge_gather(const MergeGatherArgs&, cudaStream_t st) { LAUNCH(st); }
void launch_guards(void* const*, int, bool, int*, cudaStream_t st) { ++counts.guard_launches; enqueue(st); }
void launch_copy_rows(const float*, float*, const int32_t*, int, int, cudaStream_t st) { LAUNCH(st); }
void launch_patch_gather(const PatchGatherArgs&, cudaStream_t st) { LAUNCH(st); }
bool launch_bias_ln(const float*, const float*, const float*, const float*, float*, long, int, cudaStream_t st) { LAUNCH(st); return true; }
void launch_pad_weights(const int8_t*, int, int, int, int8_t*, cudaStream_t st) { LAUNCH(st); }
bool launch_gemm(const GemmArgs&, cudaStream_t st) { LAUNCH(st); return true; }
void launch_attention(const AttnArgs&, cudaStream_t st) { LAUNCH(st); }
void launch_prepare_linear(const int8_t*, const float*, int, int, float, int, int, float*, int32_t*, float*, cudaStream_t st) { LAUNCH(st); }
void launch_prepare_relbias(const float*, int, float*, cudaStream_t st) { LAUNCH(st); }
void launch_wait_probe(int*, cudaStream_t st) { LAUNCH(st); }
int launch_mma_peak(int, int, unsigned long long*, int*, cudaStream_t) { return 0; }
bool launch_calibrate_block(const CalBlockArgs&, cudaStream_t st) { LAUNCH(st); return true; }
bool launch_calibrate_merge(const CalMergeArgs&, cudaStream_t st) { LAUNCH(st); return true; }
float cal_key_to_float(uint32_t) { return 0.f; }
}  // namespace mixaq
