// General fp32 verify kernels: f32 operands, gated rule.
#include "tv_verify_simt.cuh"

int tv_simt_f32_gated(const VerifyArgs& a, cudaStream_t stream) { return launch_nodes<false, false>(a, stream); }
int tv_simt_f32_gated_prepare() { return prepare_all<false, false>(); }
