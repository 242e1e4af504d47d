// Delta-rule tensor-core verification, trees of up to 64 nodes (tv_verify_tc_delta.cuh; one module per row-block count).
#include "tv_verify_tc_delta.cuh"

bool tv_verify_tc_delta_supports(const VerifyArgs& a) { return tvdelta::supports<1>(a); }
int tv_launch_verify_tc_delta(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  return tvdelta::launch<1>(a, status, stream);
}
