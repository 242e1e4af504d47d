// Verify kernels at fp32 accuracy on the tensor cores: f32 operands.
#include "tv_verify_exact.cuh"

int tv_exact_f32(const VerifyArgs& a, int32_t* status, cudaStream_t stream) { return tvexact::launch_any<false>(a, status, stream); }
int tv_exact_f32_prepare() { return tvexact::prepare_any<false>(); }
