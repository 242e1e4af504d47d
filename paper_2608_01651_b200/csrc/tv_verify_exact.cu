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
// (6.7 / 10.1 on 4 items of 16), under the gated rule up to 48 (32 nodes, 512 items: 30 / 51).  It hardly depends on
// the widths either, and one CTA per SM goes through its items one by one, where the general kernel has several
// narrow ones on an SM; so below 33 nodes (below 49 where f32 operands make three pieces of everything) narrow items lose
// outside a range of counts:
//     items                              32            64           148           160           256           352           512
//     24 nodes, bf16, chain, 64 x 64  7.7 /  7.6   7.8 /  7.7  10.0 /  8.4  12.8 / 12.6  16.4 / 13.0  17.1 / 18.1  25.4 / 23.4
//     32 nodes, bf16, chain, 64 x 128 8.0 /  8.2  10.2 /  8.7  12.9 / 10.0  19.7 / 15.0  21.2 / 15.8  31.4 / 22.2  40.4 / 28.9
//     24 nodes, f32, chain, 64 x 64   7.4 /  8.4   7.6 /  8.5   9.7 /  9.2  12.6 / 15.0  16.4 / 15.8  17.2 / 22.8  24.6 / 29.9
//     24 nodes, f32, chain, 64 x 128  7.5 /  8.7   9.6 /  9.0  12.0 / 11.8  18.4 / 20.1  19.5 / 20.9  29.1 / 30.4  37.4 / 39.5
//     24 nodes, f32, chain, 128 x 64  9.0 / 10.0   9.2 / 10.2  12.5 / 10.9  17.8 / 18.8  24.5 / 19.4  25.5 / 27.7  33.2 / 36.5
//     24 nodes, f32, chain, 128 wide  9.2 / 10.3  12.4 / 10.7  16.8 / 13.5  26.6 / 23.2  27.6 / 24.1  39.9 / 34.7  52.0 / 45.4
//     33 nodes, f32, chain, 64 x 64  10.6 / 10.9  10.9 / 11.0  13.9 / 11.6  18.1 / 19.9  18.9 / 20.8  31.0 / 30.1  36.9 / 39.9
//     64 nodes, f32, chain, 64 x 64  14.0 / 14.4  14.4 / 14.5  19.2 / 15.0  26.8 / 26.4                42.7 / 39.1  53.3 / 51.0
//     56 nodes, f32, gated, 128 x 64  9.9 / 10.9  10.1 / 10.9  15.3 / 12.5
//     (64 nodes, f32, gated, chain, 64 x 64: 72 items 8.9 / 9.5, 96 11.5 / 9.7; beyond half an item per SM the
//     general kernel no longer splits 64 value columns over two CTAs)
// (600, 800, 1024 items of 17 nodes, bf16, chain, 64 x 64: 28.5 / 27.3, 32.8 / 33.5, 40.0 / 39.0.)
bool tv_verify_exact_takes(const VerifyArgs& a) {
  if (a.T > 64 || a.T <= (a.rule == TV_GATED_DELTA ? 16 : 48)) return false;
  if ((a.dk != 64 && a.dk != 128) || (a.dv != 64 && a.dv != 128)) return false;
  const int64_t items = (int64_t)a.L * a.B * a.H;
  const int sms = tv_sm_count();
  const bool wide = a.dk == 128 && a.dv == 128, narrow = a.dk == 64 && a.dv == 64;
  if (a.rule != TV_GATED_DELTA)
    return a.bf16 || (a.dv == 128 ? items > 32 : 2 * items > sms && items <= sms);
  if (a.bf16) {
    if (a.T > 32) return true;
    if (narrow) return items <= 2 * sms || (items > 3 * sms && items <= 4 * sms);
    return a.dk == 128 || a.T <= 28 || items > 32;
  }
  if (a.tree.max_depth_all < 16) return a.T > 32 || (items <= sms && (a.T > 24 || (a.dk == a.dv && items > 32)));
  // f32 operands, deep trees (depths that only the device knows count as deep)
  if (a.T > 32 && a.dk == 128) return true;
  if (wide || a.T > 48 || (a.T > 32 && a.dv == 128)) return items > 32;
  return items <= sms && items > (a.T > 32 || a.dv == 128 ? 32 : 64);
}
int tv_prepare_verify_exact() {
  const int st = tv_exact_f32_prepare();
  return st == TV_OK ? tv_exact_bf16_prepare() : st;
}
int tv_launch_verify_exact(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  return a.bf16 ? tv_exact_bf16(a, status, stream) : tv_exact_f32(a, status, stream);
}
