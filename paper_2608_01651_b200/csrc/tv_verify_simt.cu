// The general fp32 verify kernels by operand type and rule.  Each of the four sets is a translation unit and
// so a module of its own: the first call that launches one of its kernels loads that set and not all four
// (1.8 ms against 17.5, once per process).
#include "tv_internal.h"

int tv_simt_f32_gated(const VerifyArgs& a, cudaStream_t stream);
int tv_simt_f32_delta(const VerifyArgs& a, cudaStream_t stream);
int tv_simt_bf16_gated(const VerifyArgs& a, cudaStream_t stream);
int tv_simt_bf16_delta(const VerifyArgs& a, cudaStream_t stream);
int tv_simt_f32_gated_prepare();
int tv_simt_f32_delta_prepare();
int tv_simt_bf16_gated_prepare();
int tv_simt_bf16_delta_prepare();

int tv_prepare_verify_simt() {
  int st = tv_simt_f32_gated_prepare();
  if (st == TV_OK) st = tv_simt_f32_delta_prepare();
  if (st == TV_OK) st = tv_simt_bf16_gated_prepare();
  if (st == TV_OK) st = tv_simt_bf16_delta_prepare();
  return st;
}

int tv_launch_verify_simt(const VerifyArgs& a, cudaStream_t stream) {
  const bool delta = a.rule == TV_GATED_DELTA;
  if (a.bf16) return delta ? tv_simt_bf16_delta(a, stream) : tv_simt_bf16_gated(a, stream);
  return delta ? tv_simt_f32_delta(a, stream) : tv_simt_f32_gated(a, stream);
}
