// General fp32 verify kernels: f32 operands, delta rule.
#include "tv_verify_simt.cuh"

int tv_simt_f32_delta(const VerifyArgs& a, cudaStream_t stream) { return launch_nodes<false, true>(a, stream); }
int tv_simt_f32_delta_prepare() { return prepare_all<false, true>(); }
