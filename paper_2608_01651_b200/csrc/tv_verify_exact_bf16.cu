// Verify kernels at fp32 accuracy on the tensor cores: bf16 operands.
#include "tv_verify_exact.cuh"

int tv_exact_bf16(const VerifyArgs& a, int32_t* status, cudaStream_t stream) { return tvexact::launch_any<true>(a, status, stream); }
int tv_exact_bf16_prepare() { return tvexact::prepare_any<true>(); }
