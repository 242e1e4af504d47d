// General fp32 verify kernels: bf16 operands, gated rule.
#include "tv_verify_simt.cuh"

int tv_simt_bf16_gated(const VerifyArgs& a, cudaStream_t stream) { return launch_nodes<true, false>(a, stream); }
int tv_simt_bf16_gated_prepare() { return prepare_all<true, false>(); }
