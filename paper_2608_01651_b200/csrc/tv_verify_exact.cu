// The verify kernels at fp32 accuracy on the tensor cores: which calls take them, by operand type.
#include "tv_internal.h"

int tv_exact_f32(const VerifyArgs& a, int32_t* status, cudaStream_t stream);
int tv_exact_bf16(const VerifyArgs& a, int32_t* status, cudaStream_t stream);
int tv_exact_f32_prepare();
int tv_exact_bf16_prepare();

// Up to 64 nodes, widths of 64 and 128.  Device time per launch, us, general fp32 kernel / this one, at 128 x 128 unless
// said otherwise:
//     items                                4            32            64           128           256           512          2048
//     17 nodes, f32, depth 8         8.1 /  9.9  10.3 / 10.3  14.0 / 10.9  15.4 / 13.3  23.4 / 24.1  41.5 / 45.2   137 / 151
//     32 nodes, f32, depth 8        10.4 / 10.1  11.0 / 10.6  14.5 / 11.1  17.4 / 14.0  26.6 / 25.4  48.2 / 47.1   155 / 157
//     64 nodes, f32, depth 8        16.9 / 11.5  18.9 / 12.1  25.8 / 12.9  30.2 / 17.0  56.4 / 31.1   109 / 58.9   376 / 191
//     17 nodes, bf16, chain          9.4 /  7.3   9.6 /  7.6  12.8 /  8.3  16.1 /  9.6  27.7 / 16.4  52.1 / 30.9   171 / 103
//     64 nodes, bf16, chain         19.1 / 12.7  19.7 / 13.1  25.4 / 13.7  33.7 / 16.5  65.9 / 29.0   130 / 54.5   454 / 184
//     64 nodes, f32, gated           9.6 / 10.9  10.7 / 11.6  15.1 / 12.4  19.1 / 16.0  36.0 / 29.1  69.8 / 55.5   238 / 179
//     the same, 64 x 64              8.4 /  8.9   9.2 /  8.9   9.4 /  9.0  12.3 /  9.4  17.1 / 17.2  31.1 / 32.1   101 / 105
//     64 nodes, bf16, gated, 64x128  9.1 /  6.1  10.1 /  6.3  13.2 /  6.7  14.3 /  7.7  28.8 / 13.7  56.2 / 24.9   197 / 80.3
//     49 nodes, bf16, gated, 64x64   8.7 /  6.0   8.8 /  6.1   9.6 /  6.1  12.2 /  6.5  15.8 / 10.6  31.9 / 19.4   107 / 61.2
// What an item costs here hardly depends on its nodes: up to 16 the general kernel is the faster one everywhere
// (6.7 / 10.1 on 4 items of 16), under the gated rule up to 48 with f32 operands (32 nodes, 512 items: 30.5 / 45.3).  It
// hardly depends on the widths either, and one CTA per SM goes through its items one by one, where the general kernel has
// several narrow ones on an SM; so below 33 nodes (below 49 where f32 operands make three pieces of everything) narrow items
// lose outside a range of counts.  The general kernel cuts an item's columns into as many CTAs as find an SM, 128 columns
// in up to four, 64 in two: chains of f32 operands and the gated rule go over where a quarter or half of the SMs have an item.
//     items                              32            37            38            74            75           152           256           512
//     24 nodes, bf16, chain, 64 x 64  7.9 /  7.6   7.8 /  7.5   7.8 /  7.6   8.0 /  7.7   9.9 /  7.7  12.9 / 12.1  16.4 / 12.8  25.7 / 23.0
//     32 nodes, bf16, chain, 64 x 128 8.2 /  8.2   8.2 /  8.2  10.2 /  8.3  10.4 /  8.9  12.7 /  9.1  19.8 / 15.0  21.2 / 15.9  40.5 / 28.7
//     24 nodes, f32, chain, 64 x 64   7.5 /  8.5   7.5 /  8.5   7.6 /  8.5   7.7 /  8.6   9.7 /  8.7  12.7 / 15.1  16.2 / 15.9  24.6 / 29.8
//     24 nodes, f32, chain, 64 x 128  7.7 /  8.8   7.8 /  8.8   9.7 /  8.9   9.9 /  9.3  11.9 / 10.8  18.5 / 19.5  19.7 / 20.6  37.6 / 38.2
//     24 nodes, f32, chain, 128 x 64  9.2 / 10.2   9.2 / 10.3   9.2 / 10.2   9.5 / 10.6  12.5 / 10.5  17.9 / 18.7  24.8 / 19.6  33.4 / 36.7
//     24 nodes, f32, chain, 128 wide  9.4 / 10.4   9.4 / 10.6  12.5 / 10.7  12.8 / 11.3  15.7 / 12.4  26.8 / 22.7  28.0 / 23.9  52.2 / 44.6
//     33 nodes, f32, chain, 64 x 64  10.9 / 10.8  10.8 / 10.7  10.9 / 10.7  11.3 / 10.9  13.8 / 10.9  18.2 / 19.3  19.1 / 20.4  36.9 / 39.1
//     64 nodes, f32, chain, 64 x 64  14.6 / 14.2                                                      26.6 / 25.9  28.5 / 26.8  53.1 / 50.2
//     56 nodes, f32, gated, 128 x 64 11.1 / 11.1  11.1 / 11.1  11.2 / 11.1  11.6 / 11.3  15.4 / 11.2  23.2 / 21.3  24.4 / 22.2  44.6 / 41.2
//     56 nodes, f32, gated, 64 x 128  8.9 /  9.7   9.1 /  9.7  11.7 /  9.7  12.0 / 10.2  13.8 / 12.2  27.7 / 22.5  29.0 / 24.0  56.7 / 44.4
//     56 nodes, f32, gated, 64 x 64   8.9 /  9.4   8.8 /  9.4   8.8 /  9.5   8.9 /  9.6  11.6 /  9.5  15.7 / 16.4  16.9 / 17.2  31.9 / 32.1
// (17 nodes, bf16, chain, 64 x 64, 444, 448, 592, 640, 888, 1024 items: 17.2 / 17.9, 23.4 / 21.8, 25.6 / 23.0, 28.9 / 27.6,
// 33.2 / 33.3, 40.0 / 38.2.)  Past 1024 items the ratios stay: 6144 of 64 nodes, f32 delta 1111 / 564, f32 gated 696 / 517.
// Shallow f32 trees of 25 to 32 nodes, ratio of the times over five trees each: one item 0.99 to 1.16, two 0.89 to 1.08,
// three 0.87 to 1.03, four 0.83 to 1.01; it depends on the tree's levels more than on its nodes.
bool tv_verify_exact_takes(const VerifyArgs& a) {
  if (a.T > 64 || a.T <= (a.rule == TV_GATED_DELTA ? 16 : 48)) return false;
  if ((a.dk != 64 && a.dk != 128) || (a.dv != 64 && a.dv != 128)) return false;
  const int64_t items = (int64_t)a.L * a.B * a.H;
  const int sms = tv_sm_count();
  const bool wide = a.dk == 128 && a.dv == 128, narrow = a.dk == 64 && a.dv == 64;
  if (a.bf16 && wide && (a.rule != TV_GATED_DELTA || a.tree.max_depth_all < 16)) return false;   // the gated and the delta kernel's
  const bool crowded = a.dv == 128 ? 4 * items > sms : 2 * items > sms;   // more CTAs of the general kernel than SMs
  if (a.rule != TV_GATED_DELTA) return a.bf16 || (crowded && (a.dv == 128 || items <= sms));
  if (a.bf16) {
    if (a.T > 32) return true;
    if (narrow) return items <= 2 * sms || (items > 3 * sms && items <= 4 * sms);
    return a.dk == 128 || a.T <= 28 || items > 32;
  }
  if (a.tree.max_depth_all < 16) return a.T > 32 || (items <= sms && (a.T > 24 ? items > 2 : a.dk == a.dv && items > 32));
  // f32 operands, deep trees (depths that only the device knows count as deep)
  if (a.T <= 32) return crowded && (wide || items <= sms);
  if (a.dk == 128) return true;
  return items > 32 && (a.dv == 128 || a.T > 48 || items <= sms);
}
int tv_prepare_verify_exact() {
  const int st = tv_exact_f32_prepare();
  return st == TV_OK ? tv_exact_bf16_prepare() : st;
}
int tv_launch_verify_exact(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  return a.bf16 ? tv_exact_bf16(a, status, stream) : tv_exact_f32(a, status, stream);
}
