// The verify kernels at fp32 accuracy on the tensor cores: which calls take them, by operand type.
#include "tv_internal.h"

int tv_exact_f32(const VerifyArgs& a, int32_t* status, cudaStream_t stream);
int tv_exact_bf16(const VerifyArgs& a, int32_t* status, cudaStream_t stream);
int tv_exact_f32_prepare();
int tv_exact_bf16_prepare();

// Up to 64 nodes, widths of 64 and 128.  Device time per launch, us, general fp32 kernel / this one, the delta rule at
// 128 x 128 unless said otherwise:
//     items                       4            32            64           128           256           512
//     17 nodes, f32, depth 8   9.0 /  9.8   9.3 / 10.1   12.1 / 10.7   13.9 / 13.8   22.1 / 21.9   41.1 / 43
//     32 nodes, f32, depth 8  10.8 / 10.1  11.4 / 10.4   14.7 / 11.0   17.2 / 14.5   25.3 / 25.4   46.9 / 47.4
//     64 nodes, f32, depth 8  18.1 / 11.5  18.6 / 12.0   25.6 / 12.8   30.2 / 17.6   55.5 / 31.9    109 / 61.3
//     17 nodes, bf16, chain    9.2 /  7.3   9.5 /  7.6   12.7 /  8.3   16.1 /  9.4   27.4 / 16.4   51.8 / 31.2
//     64 nodes, bf16, chain   18.7 / 13.1  19.6 / 13.4   25.4 / 14.0   33.6 / 17.0   65.6 / 29.7    130 / 56.1
//     64 nodes, f32, gated    10.0 / 10.9  10.4 / 11.2   14.7 / 12.0   18.8 / 17.0   35.3 / 32.1   69.3 / 62.6
//     the same, 64 x 64        8.6 /  8.2   8.8 /  8.4    9.1 /  8.5   12.2 /  8.9                 30.9 / 31.4
// What an item costs here hardly depends on its nodes: up to 16 the general kernel is the faster one everywhere
// (6.7 / 10.1 on 4 items of 16), under the gated rule up to 48 (32 nodes, 512 items: 30 / 51).
bool tv_verify_exact_takes(const VerifyArgs& a) {
  if (a.T > 64 || (a.dk != 64 && a.dk != 128) || (a.dv != 64 && a.dv != 128)) return false;
  const int64_t items = (int64_t)a.L * a.B * a.H;
  const int sms = tv_sm_count();
  if (a.rule != TV_GATED_DELTA) return a.T > 48 && (a.bf16 || (items > 32 && (a.dv == 128 || items <= sms)));
  if (a.T > 32) return true;
  if (a.bf16 || a.tree.max_depth_all >= 16) return a.T > 16;   // (depths that only the device knows count as deep)
  return a.T > 16 && items <= sms && (a.T > 24 || items > 32);
}
int tv_prepare_verify_exact() {
  const int st = tv_exact_f32_prepare();
  return st == TV_OK ? tv_exact_bf16_prepare() : st;
}
int tv_launch_verify_exact(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  return a.bf16 ? tv_exact_bf16(a, status, stream) : tv_exact_f32(a, status, stream);
}
