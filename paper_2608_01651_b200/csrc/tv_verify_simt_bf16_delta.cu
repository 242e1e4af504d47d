// General fp32 verify kernels: bf16 operands, delta rule.
#include "tv_verify_simt.cuh"

int tv_simt_bf16_delta(const VerifyArgs& a, cudaStream_t stream) { return launch_nodes<true, true>(a, stream); }
int tv_simt_bf16_delta_prepare() { return prepare_all<true, true>(); }
