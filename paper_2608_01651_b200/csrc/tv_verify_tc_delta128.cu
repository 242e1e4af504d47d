// Delta-rule tensor-core verification, trees of 65..128 nodes (tv_verify_tc_delta.cuh; one module per row-block count).
#include "tv_verify_tc_delta.cuh"

bool tv_verify_tc_delta128_supports(const VerifyArgs& a) { return tvdelta::supports<2>(a); }
int tv_launch_verify_tc_delta128(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  return tvdelta::launch<2>(a, status, stream);
}
