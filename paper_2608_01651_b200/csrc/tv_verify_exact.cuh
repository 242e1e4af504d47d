// Tree verification at fp32 accuracy on the tensor cores (tcgen05 + TMEM): up to 64 nodes of any depth, f32 or
// bf16 operands, both rules, dk and dv of 64 or 128.
//
// Algebra (Theorem 1, Eq. 2; Lemma 2).  With C_ij = (P_i / P_j) q_i.k_j and G_ij = beta_i (P_i / P_j) k_i.k_j on the
// tree's paths, R = D_beta (V - D_P K S_pre^T) and N = (I + G)^-1:
//     U = R + (N - I) R,     O = D_P Q S_pre^T + C N R        (gated rule: U = R = V, O = D_P Q S_pre^T + C V)
// Every product of the size of the item is dense and on the tensor cores, whatever the tree: [Q ; K] K^T, [Q ; K] S_pre^T and
// [C N ; N - I] R, with the 64 q rows and the 64 k rows of an item as the 128 rows of one tile.  The rows of C N and N come from
// the triangular systems x (I + G) = c_i or e_i, in one of two forms: over the entries of a path of at most 16 nodes
// (PATHS), or, for trees of any depth, in blocks of 16 columns.
//
// Accuracy.  An fp32 operand is three bf16 pieces of 8 mantissa bits each, so a product of two is six products of
// pieces (the other three lie below 2^-24 of it); bf16 operands are their own only piece.  The pieces are those of
// 2^16 times the value, and the sums are brought back where they are read: bf16 ends at 2^-133, fp32 at 2^-149, and
// without the factor a value of 2^-120 keeps 14 of its bits.  Values of 2^112 and sums of 2^96 and more leave fp32's range
// by it and take the way of values that are not finite (below), in fp32 throughout.  The tensor core adds into
// its fp32 accumulator without rounding to nearest, so the products of the lower pieces go in first, the
// leading ones on top of them, and the two halves of a contraction over 128 have an accumulator each, added here.
// Error of a 128 x 128 x 128 product of normal / positive numbers against 64 bits 0.75e-7 / 0.75e-7; one chain of
// leading products 1.2e-7 / 1.5e-7, fp32 FMA in pairs 1.46e-7 / 0.87e-7, pieces in falling order 6.5e-7 and more.
//
// Layout.  Persistent, 20 warps: 16 workers go through an item together (split the operands into pieces, C and G from the
// scores, systems and R, pieces of both, outputs), one warp issues the products, two make the tables of the next item
// (masks, gates, products of alpha from each node up its path, four steps at a time), one works out where the next item
// lies and brings it near.  f32 q, k and state pass through registers into their pieces; bf16 q and k are copied, an item
// ahead.  Beside the general fp32 kernel, whose state product alone is 13 of 27 us on 128 items (fp32 FMA rate: 8.6):
//     128 items of 63 nodes, f32, delta          29.6 -> 17.0 us        512 of 64   109 -> 58.6
//     256 items, chains of 40 nodes, bf16        48.0 -> 22.7           512 of 64   130 -> 54.3
//     256 items of 24 nodes, bf16, depth unknown 25.3 -> 16.8
// What bounds it: the phases of an item one after the other (128 items of 63 nodes, thousands of cycles: operands 8, of
// which 6 at the copy rate; scores 2; C and G 1; state product behind them 4; R 2; last product 3; outputs 3), and code
// of 70 KiB that runs once per item through an instruction cache smaller than that: loops stay rolled, and one kernel
// that held both forms of the systems was 10 % slower on chains.  The f32 variants of 128 value columns spill (124 to 184 bytes
// of stores and 176 to 236 of loads a thread): two batches of operands on their way take 64 registers of it.  The SM's four quarters matter too: the warps of the q
// rows sit on two of them (a warp reads the tensor memory lanes of its number mod 4).
//
// Values that are not finite reach the rows that the recurrence takes them to and no others: rows of R and G that hold any
// are zeroed before the dense products, and the rows below them are worked out again at the end, in fp32 (redo_rows).
// Every wait is bounded (status word on expiry).
#pragma once
#include <type_traits>

#include "tv_tc_common.cuh"

namespace tvexact {

using namespace tvtc;

constexpr int kNodes = 64;
constexpr int kMaxItems = 32;   // of a CTA
constexpr int kPath = 16;       // entries of a path list
constexpr float kUp = 65536.f;  // on every operand that is split into pieces

constexpr int kWorkers = 16;                    // warps; four more: products, tables (two), requests to L2
constexpr int kThreads = 32 * (kWorkers + 4);
constexpr int kWorkerRegs = 104, kServiceRegs = 64;   // a thread, by groups of four warps, of 96 at launch

// Where a unit of work lies: elements of its first node in q and k | v | gates | O and U (value column included).
struct Place {
  size_t qk0, v0, g0, o0, meta0;
  const float* S;
  int32_t n, pad;
};

template <bool BF16, bool DELTA, int DK, int DVC>
struct Cfg {
  static constexpr int NP = BF16 ? 1 : 3;               // pieces of q and k
  static constexpr int NR = BF16 && !DELTA ? 1 : 3;     // pieces of R
  static constexpr int KH = DK / 64;                    // halves of the contraction over dk
  static constexpr int NQ = BF16 ? 2 : 1;               // sets of q and k rows
  static constexpr float kXDown = NP == 3 ? 1.f / (kUp * kUp) : 1.f / kUp;      // the sums, back
  static constexpr float kLastDown = NR == 3 ? 1.f / (kUp * kUp) : 1.f / kUp;
  static constexpr int CW = DVC / 4;                    // columns of a tile row that a worker thread has
  static constexpr int SU = DVC / 32;                   // 16-byte chunks of the state per thread and half
  // bytes from the 1024-aligned base
  static constexpr uint32_t kHalf = 16384;              // [Q ; K]: [128 rows][64 bf16] per piece and 64 channels
  static constexpr uint32_t kStep = KH == 2 ? kHalf : 64;   // from one half of the channels to the other
  static constexpr uint32_t kSHalf = DVC * 128;         // state: [DVC rows][64 bf16] per piece and half
  static constexpr uint32_t kRPiece = kNodes * DVC * 2; // R: per piece, 64-column tiles of [64 nodes][64]
  static constexpr uint32_t kStage = 32 * CW * 4;       // outputs on their way: 32 rows of a warp's columns
  static constexpr uint32_t kQKSet = NP * KH * kHalf;
  static constexpr uint32_t kCols = 2 * DVC + 128 <= 256 ? 256 : 512;   // TMEM columns: X twice, scores and coefficients
  static constexpr uint32_t oQK = 0;
  static constexpr uint32_t oS = NQ * kQKSet;           // the state's pieces, then R's, then outputs
  static constexpr uint32_t kSBytes = 3 * KH * kSHalf > kWorkers * kStage ? 3 * KH * kSHalf : kWorkers * kStage;
  static constexpr uint32_t oTab = oS + kSBytes;
  static constexpr uint32_t kMat = 10 * 1024;           // a triangular matrix of 4 x 4 blocks of 16 x 16: C, G, decay ratios (then N)
  // redo_rows, where operands and matrices were: 128 rows of q and k, 64 state rows (then C and G), X
  static constexpr int kRedoLd = DK + 4;
  static constexpr uint32_t oRedoS = 2 * kNodes * kRedoLd * 4, kRedoCoef = 2 * kNodes * (kNodes + 1) * 4;
  static constexpr uint32_t oRedoX = oRedoS + (kNodes * kRedoLd * 4 > kRedoCoef ? kNodes * kRedoLd * 4 : kRedoCoef);
  static constexpr uint32_t kRedo = oRedoX + 2 * kNodes * DVC * 4;
  // A call, where the same code in line takes registers from the pipeline: 512 items of 64 nodes, in line / called, f32 gated
  // 61.8 / 55.2 us, bf16 gated 64 x 128 25.8 / 24.8; 128 x 64 21.4 / 22.0, bf16 delta 64 x 64 27.1 / 27.8.
  static constexpr bool kRedoCall = !BF16 || (!DELTA && DK < DVC);
  static constexpr uint32_t oJump4 = oTab + 3 * kMat > kRedo ? oTab + 3 * kMat : kRedo;   // float4 per node
  static constexpr uint32_t oUp4 = oJump4 + kNodes * 16;   // 4 x int8 per node
  static constexpr uint32_t oPath = oUp4 + kNodes * 4;     // uint8 [kPath] per node: its path by depth, itself last
  static constexpr uint32_t oDepth = oPath + kNodes * kPath;   // uint8 per node: four times its depth
  static constexpr uint32_t oLink = oDepth + kNodes;
  static constexpr uint32_t oMask = oLink + kNodes * 8;
  static constexpr uint32_t oP = oMask + kNodes * 8;
  static constexpr uint32_t oBe = oP + kNodes * 4;
  static constexpr uint32_t oBar = oBe + kNodes * 4;
  static constexpr uint32_t oBad = oBar + 8 * 16;       // per item of the CTA: node masks of values that are not finite
  static constexpr uint32_t oMisc = oBad + kMaxItems * 16;   // TMEM base, abort flag, any
  static constexpr uint32_t oPlace = oMisc + 32;        // of two items
  static constexpr uint32_t kSmem = oPlace + 2 * sizeof(Place);
  static_assert(3 * kRPiece <= kSBytes, "R in the state's place");
  static_assert(oJump4 % 16 == 0 && oBar % 8 == 0 && oBad % 16 == 0 && oRedoX % 16 == 0, "alignment");
  static_assert(kSmem <= 232448, "shared memory of one CTA");
};

enum Bar { QK = 0, ST = 1 /* , 2 */, SC = 3, X, COEF, RP, ACC, TAB, kNumBars };

// Products of pieces in the order in which they are issued, small ones first: a piece of A in bits 0..1, of B in 2..3
template <int NA, int NB> struct Order;
template <> struct Order<3, 3> { static constexpr int n = 6; static constexpr uint32_t code = 0x014825u; };
template <> struct Order<1, 3> { static constexpr int n = 3; static constexpr uint32_t code = 0x048u; };
template <> struct Order<3, 1> { static constexpr int n = 3; static constexpr uint32_t code = 0x012u; };
template <> struct Order<1, 1> { static constexpr int n = 1; static constexpr uint32_t code = 0x0u; };

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 r;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a) : "memory");
  return r;
}
__device__ __forceinline__ float4 ldg_stream(const float* p) {
  float4 r;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p) : "memory");
  return r;
}
// kUp times a pair of fp32 as three words of two bf16: every piece rounded to nearest, every remainder exact, for any
// number that the factor does not take past fp32's range (infinite or NaN pieces there).
__device__ __forceinline__ void split3(Pair x, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  const Pair minus = pack(-1.f, -1.f);
  x = mul2(x, pack(kUp, kUp));
  float2 v = unpack(x);
  hi = pack_sat(v.x, v.y);
  x = fma2(pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), minus, x);
  v = unpack(x);
  mid = pack_sat(v.x, v.y);
  x = fma2(pack(__uint_as_float(mid << 16), __uint_as_float(mid & 0xffff0000u)), minus, x);
  v = unpack(x);
  lo = pack_rn(v.x, v.y);
}
// NaN where x or y is not finite, else s unchanged
__device__ __forceinline__ Pair watch(Pair s, Pair x) { return fma2(x, pack(0.f, 0.f), s); }
__device__ __forceinline__ bool spotted(Pair s) {
  const float2 v = unpack(s);
  return !(v.x + v.y == 0.f);
}

// Rows that a value that is not finite reaches, by the recurrence's own terms: the dense products lose track of whose it was.
// `bad`: nodes whose value reaches all nodes below them, two words, then nodes of their own row only.  The whole item is worked
// out again in fp32 by the worker warps, in the pipeline's shared memory (4 x 4 tiles a thread for the products, a thread per
// column for U), and the rows in question are stored.  No such value is expected; a poisoned request should still not hold
// up a batch: 512 items of 64 nodes, 32 of them NaN, f32 delta 145 us, all of them 430 (row by row from global memory 840
// and 3270; without any 56, general kernel 111), bf16 chains 245 and 825 (1065 and 4140; 52, 127).
template <bool BF16, bool DELTA, int DK, int DVC>
__device__ __forceinline__ void redo_rows(const VerifyArgs& a, int item, int v_first, const uint32_t* bad, unsigned char* sm,
                                          float2* link, float* be_s, float* P_s, uint64_t* mask_s, int tid) {
  using C = Cfg<BF16, DELTA, DK, DVC>;
  constexpr int LD = C::kRedoLd, kT = 32 * kWorkers;
  float* const rows_s = reinterpret_cast<float*>(sm);                     // q rows, then k rows
  float* const state_s = reinterpret_cast<float*>(sm + C::oRedoS);        // 64 value columns of the state
  float* const coef_s = state_s;                                          // later: C, then G
  float* const x_s = reinterpret_cast<float*>(sm + C::oRedoX);            // [Q ; K] S^T; then R and U in the k rows
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kT) : "memory"); };
  // worked out again for every part: kept through all of them, they would take registers from the whole kernel
  auto place = [&] {
    asm volatile("" : "+r"(item));
    return tv_item_rows(a.tree, a.lay, item, a.B, a.H, a.Hk, a.T, DK, a.dv);
  };
  ItemRows rows = place();
  const int n = rows.n;
  if (tid < n) {
    mask_s[tid] = a.tree.anc[(rows.meta0 + tid) * 2];
    link[tid].x = a.alpha[rows.g0 + (size_t)tid * rows.g_rs];
    be_s[tid] = DELTA ? a.beta[rows.g0 + (size_t)tid * rows.g_rs] : 1.f;
  }
  auto four = [&](const void* x, size_t i) {
    if (!BF16) return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(x) + i);
    const uint2 w = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(x) + i);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
  };
#pragma unroll 1
  for (int x = tid; x < n * (DK / 4); x += kT) {
    const int r = x / (DK / 4), c = x % (DK / 4) * 4;
    const size_t at = rows.qk0 + (size_t)((int64_t)r * rows.qk_rs) + c;
    *reinterpret_cast<float4*>(rows_s + r * LD + c) = four(a.q, at);
    *reinterpret_cast<float4*>(rows_s + (kNodes + r) * LD + c) = four(a.k, at);
  }
  // products of the 128 rows with 64 value columns of the state after the other, and with the k rows
  constexpr int kChunks = DVC / 64, R = DELTA ? 4 : 2;   // (gated rule: q rows only)
  using Vec = std::conditional_t<BF16, float2, float4>;   // (fewer registers where this is compiled in line, see kRedoCall)
  constexpr int VW = sizeof(Vec) / 4;
#pragma unroll 1
  for (int ch = 0; ch <= kChunks; ++ch) {
    const bool coef = ch == kChunks;
    if (!coef) {
      const float* S = a.S_pre + ((size_t)item * a.dv + v_first + 64 * ch) * DK;
#pragma unroll 1
      for (int x = tid; x < 64 * (DK / 4); x += kT)
        *reinterpret_cast<float4*>(state_s + x / (DK / 4) * LD + x % (DK / 4) * 4) = *reinterpret_cast<const float4*>(S + 4 * x);
    }
    sync();
    const float* ra = rows_s + (tid >> 4) * LD;                                           // rows tid / 16 + 0, 32, ..
    const float* rb = (coef ? rows_s + kNodes * LD : state_s) + (tid & 15) * LD;          // columns tid % 16 + 0, 16, 32, 48
    float acc[R][4] = {};
#pragma unroll 1
    for (int x = 0; x < DK; x += VW) {
      Vec l[R];
#pragma unroll
      for (int e = 0; e < R; ++e) l[e] = *reinterpret_cast<const Vec*>(ra + 32 * e * LD + x);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const Vec r = *reinterpret_cast<const Vec*>(rb + 16 * f * LD + x);
#pragma unroll
        for (int w = 0; w < VW; ++w)
#pragma unroll
          for (int e = 0; e < R; ++e)
            acc[e][f] = fmaf(reinterpret_cast<const float*>(&l[e])[w], reinterpret_cast<const float*>(&r)[w], acc[e][f]);
      }
    }
#pragma unroll
    for (int e = 0; e < R; ++e)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int r = (tid >> 4) + 32 * e, c = (tid & 15) + 16 * f;
        (coef ? coef_s + r * (kNodes + 1) : x_s + r * DVC + 64 * ch)[c] = acc[e][f];
      }
    sync();
  }
  // decay, from a node up its path: C in the first 64 rows, G in the others
  if (tid < (DELTA ? 2 : 1) * kNodes && (tid & (kNodes - 1)) < n) {
    const int i = tid & (kNodes - 1);
    const bool g = DELTA && tid >= kNodes;
    float* c = coef_s + tid * (kNodes + 1);
    float w = 1.f;
#pragma unroll 1
    for (int j = i; j >= 0;) {
      c[j] = g ? be_s[i] * (w * c[j]) : w * c[j];
      w *= link[j].x;
      const uint64_t m = mask_s[j];
      j = m ? 63 - __clzll((long long)m) : -1;
    }
    if (!g) P_s[i] = w;
  }
  sync();
  rows = place();
#pragma unroll 1
  for (int x = tid; x < n * DVC; x += kT) {
    const int i = x / DVC, c = x % DVC;
    const size_t at = rows.v0 + (size_t)((int64_t)i * rows.v_rs) + v_first + c;
    float u = BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.v)[at]) : reinterpret_cast<const float*>(a.v)[at];
    if (DELTA) u = be_s[i] * (u - P_s[i] * x_s[(kNodes + i) * DVC + c]);
    x_s[(kNodes + i) * DVC + c] = u;
  }
  sync();
  // sum over the nodes of m, from the deepest up, of their coefficients in a row times their entries of U in column c
  auto over = [&](const float* row, uint64_t m, int c) {
    float s = 0.f;
#pragma unroll 1
    while (m) {
      float w[4], u[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = 63 - __clzll((long long)m);
        w[e] = m ? row[j] : 0.f;
        u[e] = m ? x_s[(kNodes + j) * DVC + c] : 0.f;
        if (m) m ^= 1ull << j;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) s = fmaf(w[e], u[e], s);
    }
    return s;
  };
  if (DELTA) {
    if (tid < DVC)
#pragma unroll 1
      for (int i = 0; i < n; ++i) x_s[(kNodes + i) * DVC + tid] -= over(coef_s + (kNodes + i) * (kNodes + 1), mask_s[i], tid);
    sync();
  }
  rows = place();
  const uint64_t B = bad[0] | (uint64_t)bad[1] << 32, W = bad[2] | (uint64_t)bad[3] << 32;
#pragma unroll 1
  for (int x = tid; x < n * DVC; x += kT) {
    const int i = x / DVC, c = x % DVC;
    const uint64_t m = mask_s[i] | 1ull << i;
    if (!((m & B) || (W >> i & 1))) continue;
    const size_t to = rows.o0 + (size_t)((int64_t)i * rows.o_rs) + v_first + c;
    a.O[to] = P_s[i] * x_s[i * DVC + c] + over(coef_s + i * (kNodes + 1), m, c);
    if (a.U) a.U[to] = x_s[(kNodes + i) * DVC + c];
  }
  sync();
}

// All items of the CTA that have such rows.  Only the worker warps come back from here to barriers.
template <bool BF16, bool DELTA, int DK, int DVC>
__device__ __forceinline__ void redo_items(const VerifyArgs& a, int n_units, int n_split, unsigned char* sm) {
  using C = Cfg<BF16, DELTA, DK, DVC>;
  int tid;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  if (tid >= 32 * kWorkers) return;
  const uint32_t* bad = reinterpret_cast<const uint32_t*>(sm + C::oBad);
#pragma unroll 1
  for (int unit = (int)blockIdx.x; unit < n_units; unit += (int)gridDim.x, bad += 4) {
    if (!(bad[0] | bad[1] | bad[2] | bad[3])) continue;
    const int item = unit / n_split;
    redo_rows<BF16, DELTA, DK, DVC>(a, item, (unit - item * n_split) * DVC, bad, sm, reinterpret_cast<float2*>(sm + C::oLink),
                                    reinterpret_cast<float*>(sm + C::oBe), reinterpret_cast<float*>(sm + C::oP), reinterpret_cast<uint64_t*>(sm + C::oMask), tid);
  }
}

template <bool BF16, bool DELTA, int DK, int DVC>
__device__ __noinline__ void redo_items_call(const VerifyArgs& a, int n_units, int n_split, unsigned char* sm) {
  redo_items<BF16, DELTA, DK, DVC>(a, n_units, n_split, sm);
}

template <bool BF16, bool DELTA, int DK, int DVC, bool PATHS>
__global__ void __launch_bounds__(kThreads, 1)
verify_exact_kernel(const __grid_constant__ VerifyArgs a, int n_units, int n_split, int32_t* status) {
  using C = Cfg<BF16, DELTA, DK, DVC>;
  constexpr int KH = C::KH, CW = C::CW, SU = C::SU;
  constexpr int CK = DK / 4, RS = 32 * kWorkers / CK, U = kNodes / RS;   // f32 q and k: 16-byte chunks of a row, rows of a pass, passes
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw;
  const uint32_t sbase = smem_u32(sm);
  if (sbase & 1023u) {   // the swizzled tiles need this alignment; refuse rather than compute garbage
    if (threadIdx.x == 0 && status) atomicExch(status, (int)TV_ERR_CUDA);
    return;
  }
  float2* const link = reinterpret_cast<float2*>(sm + C::oLink);   // alpha and parent (int bits, -1 at a root child)
  float* const P_s = reinterpret_cast<float*>(sm + C::oP);
  float* const be_s = reinterpret_cast<float*>(sm + C::oBe);
  uint64_t* const mask_s = reinterpret_cast<uint64_t*>(sm + C::oMask);
  uint32_t* const bad_s = reinterpret_cast<uint32_t*>(sm + C::oBad);   // per item: [2] below, [2] own (see redo_rows)
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(sm + C::oMisc);
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(sm + C::oMisc + 4);
  volatile int* const any_bad = reinterpret_cast<volatile int*>(sm + C::oMisc + 8);
  auto bar = [&](int i) { return sbase + C::oBar + 8u * (uint32_t)i; };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // a unit of work: DVC value columns of an item; this CTA has every gridDim.x-th one
  const int n_it = (n_units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  auto unit_of = [&](int it) { return (int)blockIdx.x + it * (int)gridDim.x; };
  auto state_of = [&](int unit) {
    const int item = n_split == 1 ? unit : unit / n_split;
    return a.S_pre + ((size_t)item * a.dv + (unit - item * n_split) * DVC) * DK;
  };
  Place* const place_s = reinterpret_cast<Place*>(sm + C::oPlace);
  auto set_place = [&](int it) {
    const int unit = unit_of(it), item = n_split == 1 ? unit : unit / n_split, v_first = (unit - item * n_split) * DVC;
    const ItemRows rows = tv_item_rows(a.tree, a.lay, item, a.B, a.H, a.Hk, a.T, DK, a.dv);
    Place* const p = place_s + (it & 1);
    p->qk0 = rows.qk0;
    p->v0 = rows.v0 + v_first;
    p->g0 = rows.g0;
    p->o0 = rows.o0 + v_first;
    p->meta0 = rows.meta0;
    p->S = state_of(unit);
    p->n = rows.n;
  };

  // Operands on their way to pieces, in batches of SU (state) or U (f32 q or k) 16-byte chunks a thread: the one being
  // split and the one behind it.  The state is never the output of a kernel that releases its dependents early, so it
  // is requested before the dependency wait: bf16 to registers, f32, where q and k come first, to L2.
  constexpr int NU = SU > U ? SU : U;
  float4 cur[NU], next[NU];
  auto fetch_state = [&](const float* S, int h, float4 (&d)[NU]) {
    const float* Sg = S + (tid >> 4) * DK + h * 64 + (tid & 15) * 4;
#pragma unroll
    for (int u = 0; u < SU; ++u) d[u] = ldg_stream(Sg + u * 32 * DK);
  };
  if (warp < kWorkers) {
    if (BF16) {
      fetch_state(state_of(unit_of(0)), 0, cur);
      if (KH == 2) fetch_state(state_of(unit_of(0)), 1, next);
    } else if (tid < DVC * DK / 32) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(state_of(unit_of(0)) + tid * 32));
    }
  }
  if (tid < kMaxItems * 4) bad_s[tid] = 0;
  if (tid == 0) {
    *abort_flag = 0;
    *any_bad = 0;
    mbar_init(bar(QK), kWorkers);
    mbar_init(bar(ST), kWorkers);
    mbar_init(bar(ST + 1), kWorkers);
    mbar_init(bar(SC), 1);
    mbar_init(bar(X), 1);
    mbar_init(bar(COEF), kWorkers);
    mbar_init(bar(RP), kWorkers);
    mbar_init(bar(ACC), 1);
    mbar_init(bar(TAB), 3);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kWorkers) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(C::kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sc_col = tmem + 2 * DVC;
  grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) set_place(0);
  __syncthreads();

  if (warp < kWorkers) {   // (this branch first in the code: 512 f32 items of 64 nodes 61.3 -> 58.4 us)
    // ===================== workers =====================
    // A wait that runs out sets the abort flag, and every later one returns soon; the warps go on all the same, for
    // they meet at barriers of the CTA.
    set_registers_up<kWorkerRegs>();
    auto request_qk = [&](int it) {   // bf16: rows as they are
      const Place& pl = place_s[it & 1];
      const uint32_t set = (uint32_t)(it & 1) * C::kQKSet;
      constexpr int CB = DK / 8, RB = 32 * kWorkers / CB;   // 16-byte chunks of a row, rows of a pass
      const int c = tid % CB;
      const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q) + pl.qk0 + c * 8;
      const __nv_bfloat16* k = reinterpret_cast<const __nv_bfloat16*>(a.k) + pl.qk0 + c * 8;
#pragma unroll 1
      for (int row = tid / CB; row < pl.n; row += RB) {
        const uint32_t to = sbase + C::oQK + set + (uint32_t)(c >> 3) * C::kHalf + (uint32_t)row * 128u + (uint32_t)(((c & 7) ^ (row & 7)) << 4);
        cp_async16(to, q + (int64_t)row * a.lay.qk.t);
        cp_async16(to + 8192u, k + (int64_t)row * a.lay.qk.t);
      }
    };
    if (BF16) request_qk(0);
    const int tid0 = tid;
    const uint32_t sbase0 = sbase, tmem0 = tmem;
#pragma unroll 1
    for (int it = 0; it < n_it; ++it) {
      // What follows from the thread's place is worked out for each item: kept, it would not fit the registers.
      int tid = tid0;
      uint32_t sbase = sbase0, tmem = tmem0;
      asm volatile("" : "+r"(tid), "+r"(sbase), "+r"(tmem));
      const int warp = tid >> 5, lane = tid & 31;
      const uint32_t sc_col = tmem + 2 * DVC;
      const int quad = warp & 3, cg = warp >> 2;   // TMEM lanes of this warp; its quarter of the columns
      const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
      const int i = (quad & 1) * 32 + lane, b = i >> 4, r16 = i & 15;   // the thread's tile row: node, its block, its place there
      const bool key = quad >= 2;                                       // tile rows 64..127: k rows
      const int c0 = CW * cg;
      auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(32 * kWorkers) : "memory"); };
      auto arrive = [&](int n) {
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(n));
      };
      // block (rb, cb) of a triangular matrix, chunk of four columns of a row in it
      auto blk = [&](int mat, int rb, int cb) { return sbase + C::oTab + mat * C::kMat + (uint32_t)((rb * (rb + 1) >> 1) + cb) * 1024u; };
      auto chunk = [](int row, int q) { return (uint32_t)(row * 64 + ((q ^ ((row >> 1) & 3)) << 4)); };
      // four fp32 as pieces, `step` bytes from one to the next
      auto put4 = [&](uint32_t to, uint32_t step, const float4& x) {
        uint32_t h0, m0, l0, h1, m1, l1;
        split3(pack(x.x, x.y), h0, m0, l0);
        split3(pack(x.z, x.w), h1, m1, l1);
        sts64(to, h0, h1);
        sts64(to + step, m0, m1);
        sts64(to + 2 * step, l0, l1);
      };
      const uint32_t ph = it & 1;
      const Place& pl = place_s[ph];
      const int T = pl.n, nb = (T + 15) >> 4;
      const bool more = it + 1 < n_it, live = (quad & 1) * 32 < T;   // warp-uniform
      // ---- operands: q, k (f32) and the halves of the state, one batch after the other ----
      {
        const uint32_t s_at = sbase + C::oS + (uint32_t)(tid >> 4) * 128u + (uint32_t)((((tid & 15) >> 1) ^ ((tid >> 4) & 7)) << 4) + (uint32_t)(tid & 1) * 8u;
        const int c4 = tid % CK, qrow = tid / CK;
        const uint32_t q_at = sbase + C::oQK + (uint32_t)(c4 >> 4) * C::kHalf + (uint32_t)qrow * 128u + (uint32_t)((((c4 & 15) >> 1) ^ (qrow & 7)) << 4) + (uint32_t)(c4 & 1) * 8u;
        auto fetch_rows = [&](const void* x, float4 (&d)[NU]) {
          const float* from = reinterpret_cast<const float*>(x) + pl.qk0 + c4 * 4 + (int64_t)qrow * a.lay.qk.t;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (qrow + u * RS < T) d[u] = ldg_stream(from + (int64_t)(u * RS) * a.lay.qk.t);
        };
        if (BF16) {
          if (it > 0) {
            fetch_state(pl.S, 0, cur);
            if (KH == 2) fetch_state(pl.S, 1, next);
          }
          asm volatile("cp.async.wait_all;" ::: "memory");
          arrive(QK);
        } else {
          fetch_rows(a.q, cur);
          fetch_rows(a.k, next);
        }
#pragma unroll 1
        for (int x = BF16 ? 2 : 0; x < 2 + KH; ++x) {   // 0, 1: q, k; 2, 3: state
          const bool qk = !BF16 && x < 2;
          const uint32_t to = qk ? q_at + (uint32_t)x * 8192u : s_at + (uint32_t)(x - 2) * C::kSHalf;
          const uint32_t step = qk ? KH * C::kHalf : KH * C::kSHalf;
          const uint32_t down = qk ? RS * 128u : 32 * 128u;
#pragma unroll
          for (int u = 0; u < NU; ++u)
            if (qk ? u < U && qrow + u * RS < T : u < SU) put4(to + (uint32_t)u * down, step, cur[u]);
          if (x >= 1) arrive(x == 1 ? QK : ST + x - 2);
#pragma unroll
          for (int u = 0; u < NU; ++u) cur[u] = next[u];
          if (!BF16 && x < KH) fetch_state(pl.S, x, next);
        }
      }
      // v of the thread's node (k rows): requested where the registers allow it
      constexpr int NV = BF16 ? CW / 2 : CW;
      uint32_t vv[NV];
      auto fetch_v = [&] {
        if (!key || i >= T) return;
        const char* src = reinterpret_cast<const char*>(a.v) + (pl.v0 + (size_t)((int64_t)i * a.lay.v.t) + c0) * (BF16 ? 2 : 4);
#pragma unroll
        for (int e = 0; e < NV / 4; ++e) {
          const uint4 x = *reinterpret_cast<const uint4*>(src + 16 * e);
          vv[4 * e] = x.x; vv[4 * e + 1] = x.y; vv[4 * e + 2] = x.z; vv[4 * e + 3] = x.w;
        }
      };
      if (BF16) fetch_v();
      mbar_wait_warp(bar(TAB), ph, abort_flag);
      if (BF16 && more) request_qk(it + 1);   // the other set: read last by the item before
      // ---- C and G: sixteen columns of a row per thread ----
      mbar_wait_warp(bar(SC), ph, abort_flag);
      tc_fence_after();
      const uint32_t slots = (uint32_t)(key ? C::kMat : 0) + sbase + C::oTab + (uint32_t)i * 64u + (uint32_t)(((i >> 1) & 3) << 4);   // ^ 4 x depth
      uint4 depths = make_uint4(0u, 0u, 0u, 0u);   // PATHS: four times the depths of the thread's columns
      if (live && cg < nb && (DELTA || !key)) {
        if (PATHS) depths = lds128(sbase + C::oDepth + 16u * cg);
        uint32_t x[16], y[16];
        tmem_ld16(sc_col + lane_addr + 16u * cg, x);
        tmem_ld16(sc_col + lane_addr + 64u + 16u * cg, y);
        tmem_wait_ld();
        if (cg <= b) {
          uint64_t m = mask_s[i];
          if (!key && i < T) m |= 1ull << i;
          const uint32_t from = blk(2, b, cg), to = blk(key ? 1 : 0, b, cg), bits = (uint32_t)(m >> (16 * cg));
          const uint32_t dw[4] = {depths.x, depths.y, depths.z, depths.w};
          const float be = be_s[i];
          Pair seen = pack(0.f, 0.f);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 w4 = lds128(from + chunk(r16, q));
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float s = __uint_as_float(x[4 * q + e]);
              s += __uint_as_float(y[4 * q + e]);
              if (!BF16) s *= C::kXDown;   // (q and k both split)
              s *= __uint_as_float(w[e]);
              if (key) s *= be;
              v[e] = (bits >> (4 * q + e)) & 1 ? s : 0.f;   // select, never 0 * x
            }
            seen = watch(seen, pack(v[0], v[1]));
            seen = watch(seen, pack(v[2], v[3]));
            if (!PATHS) {
              sts128(to + chunk(r16, q), __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if ((bits >> (4 * q + e)) & 1)
                  asm volatile("st.shared.f32 [%0], %1;" ::"r"(slots ^ ((dw[q] >> (8 * e)) & 255u)), "f"(v[e]) : "memory");
            }
          }
          if (DELTA && key && spotted(seen)) {   // a row of G that is not finite: its node's subtree is redone
            atomicOr(&bad_s[4 * it + (i >> 5)], 1u << (i & 31));
            *any_bad = 1;
#pragma unroll 1
            for (int e = 0; e < 16; ++e) {
              const uint32_t at = !PATHS ? to + chunk(r16, e >> 2) + (uint32_t)(e & 3) * 4u : slots ^ sm[C::oDepth + 16 * cg + e];
              if ((bits >> e) & 1) asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(0.f) : "memory");
            }
          }
        }
      }
      sync();
      // The warps of the q rows solve x (I + G) = c_i or e_i for the rows of C N and of N; those of the k rows work out R.
      if (DELTA && PATHS && !key) {
        // ---- paths of at most 16 nodes, entries by depth: a row per thread, from its node upwards.  A node's row of G
        // is that of the same depths of every node below it. ----
        if (cg < 2 && (quad & 1) * 32 < T && i < T) {
          const uint4 pw = *reinterpret_cast<const uint4*>(sm + C::oPath + i * kPath);
          const uint32_t pword[4] = {pw.x, pw.y, pw.z, pw.w};
          const int d = __popcll(mask_s[i]);
          const bool of_n = cg == 1;
          float x[kPath], known[kPath];   // known: what the nodes below explain, summed from zero
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint4 c4 = make_uint4(0u, 0u, 0u, 0u);
            if (!of_n) c4 = lds128(slots ^ (uint32_t)(q << 4));
            const uint32_t cw[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              x[4 * q + e] = of_n ? (4 * q + e == d ? 1.f : 0.f) : 4 * q + e <= d ? __uint_as_float(cw[e]) : 0.f;
              known[4 * q + e] = 0.f;
            }
          }
#pragma unroll
          for (int t = kPath - 1; t > 0; --t) {
            if (t > d) continue;
            x[t] -= known[t];
            const uint32_t p = (pword[t >> 2] >> (8 * (t & 3))) & 255u;
            const uint32_t g = sbase + C::oTab + C::kMat + p * 64u + (((p >> 1) & 3u) << 4);
#pragma unroll
            for (int q = 0; q < (t + 3) / 4; ++q) {
              const uint4 g4 = lds128(g ^ (uint32_t)(q << 4));
              const uint32_t gw[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (4 * q + e < t) known[4 * q + e] = fmaf(x[t], __uint_as_float(gw[e]), known[4 * q + e]);
            }
          }
          x[0] -= known[0];
          const uint32_t to = slots + (of_n ? 2 * C::kMat : 0u);   // C N in the place of C, N in that of the decay ratios
#pragma unroll
          for (int q = 0; q < 4; ++q)
            sts128(to ^ (uint32_t)(q << 4), __float_as_uint(x[4 * q]), __float_as_uint(x[4 * q + 1]), __float_as_uint(x[4 * q + 2]), __float_as_uint(x[4 * q + 3]));
        }
      }
      if (DELTA && !PATHS && !key) {
        auto sync_q = [] { asm volatile("bar.sync 3, %0;" ::"n"(16 * kWorkers) : "memory"); };   // the eight warps of the q rows
        const int qw = 2 * cg + quad;   // 0..7 among them
        // ---- diagonal blocks of N in the place of G's: one row per thread ----
        if (qw < 2 && qw * 2 < nb) {
          const int d = qw * 2 + (lane >> 4), r = lane & 15;
          const uint32_t g = blk(1, d, d);
          float x[16];
          Pair sum[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) sum[k] = pack(0.f, 0.f);
          if (d < nb) {
#pragma unroll
            for (int t = 15; t >= 0; --t) {
              const float2 s2 = unpack(sum[t >> 1]);
              x[t] = (r == t ? 1.f : 0.f) - ((t & 1) ? s2.y : s2.x);
              const Pair xx = pack(x[t], x[t]);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                if (4 * c >= t) break;
                const uint4 gv = lds128(g + chunk(t, c));
                sum[2 * c] = fma2(xx, pack(__uint_as_float(gv.x), __uint_as_float(gv.y)), sum[2 * c]);
                if (4 * c + 2 < t) sum[2 * c + 1] = fma2(xx, pack(__uint_as_float(gv.z), __uint_as_float(gv.w)), sum[2 * c + 1]);
              }
            }
          }
          __syncwarp();
          if (d < nb)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              sts128(g + chunk(r, q), __float_as_uint(x[4 * q]), __float_as_uint(x[4 * q + 1]), __float_as_uint(x[4 * q + 2]), __float_as_uint(x[4 * q + 3]));
        }
        sync_q();
        // ---- rows of C N and of N: x (I + G) = c_i or e_i; a warp has 16 rows, a thread four columns of every block of
        // two of them.  Block cb: (c - sum over later blocks of x G) times the diagonal block of N; the sum starts from
        // zero. ----
        if ((qw & 3) < nb) {
          const int q = lane >> 3, r = lane & 7, rb = qw & 3;
          const bool of_n = qw >= 4;
          const int mat = of_n ? 2 : 0;
          // sum over t of x_t M[t][4 q .. 4 q + 3], rows r and r + 8
          auto times = [&](uint32_t x, uint32_t m, Pair (&s)[4]) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint4 x0 = lds128(x + chunk(r, c)), x1 = lds128(x + chunk(r + 8, c));
              const uint32_t xa[4] = {x0.x, x0.y, x0.z, x0.w}, xb[4] = {x1.x, x1.y, x1.z, x1.w};
              uint4 g[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) g[e] = lds128(m + chunk(4 * c + e, q));
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const Pair g0 = pack(__uint_as_float(g[e].x), __uint_as_float(g[e].y)), g1 = pack(__uint_as_float(g[e].z), __uint_as_float(g[e].w));
                const Pair a2 = pack(__uint_as_float(xa[e]), __uint_as_float(xa[e])), b2 = pack(__uint_as_float(xb[e]), __uint_as_float(xb[e]));
                s[0] = fma2(a2, g0, s[0]);
                s[1] = fma2(a2, g1, s[1]);
                s[2] = fma2(b2, g0, s[2]);
                s[3] = fma2(b2, g1, s[3]);
              }
            }
          };
          auto put = [&](uint32_t at, Pair s0, Pair s1) {
            const float2 u = unpack(s0), v = unpack(s1);
            sts128(at, __float_as_uint(u.x), __float_as_uint(u.y), __float_as_uint(v.x), __float_as_uint(v.y));
          };
#pragma unroll 1
          for (int cb = rb; cb >= 0; --cb) {
            const uint32_t own = blk(mat, rb, cb), at0 = own + chunk(r, q), at1 = own + chunk(r + 8, q);
            Pair s[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = pack(0.f, 0.f);
            if (of_n && cb == rb) {   // the diagonal block itself
              const uint32_t from = blk(1, rb, rb);
              const uint4 d0 = lds128(from + chunk(r, q)), d1 = lds128(from + chunk(r + 8, q));
              sts128(at0, d0.x, d0.y, d0.z, d0.w);
              sts128(at1, d1.x, d1.y, d1.z, d1.w);
            } else {
              // (the last product apart: both in one loop compile to a form that is 7 % slower on 64-node chains)
#pragma unroll 1
              for (int tb = cb + 1; tb <= rb; ++tb) times(blk(mat, rb, tb), blk(1, tb, cb), s);
              if (cb < rb) {
                const Pair minus = pack(-1.f, -1.f);
                uint4 y0 = make_uint4(0u, 0u, 0u, 0u), y1 = y0;
                if (!of_n) {
                  y0 = lds128(at0);
                  y1 = lds128(at1);
                }
                put(at0, fma2(s[0], minus, pack(__uint_as_float(y0.x), __uint_as_float(y0.y))), fma2(s[1], minus, pack(__uint_as_float(y0.z), __uint_as_float(y0.w))));
                put(at1, fma2(s[2], minus, pack(__uint_as_float(y1.x), __uint_as_float(y1.y))), fma2(s[3], minus, pack(__uint_as_float(y1.z), __uint_as_float(y1.w))));
#pragma unroll
                for (int e = 0; e < 4; ++e) s[e] = pack(0.f, 0.f);
                __syncwarp();
              }
              times(own, blk(1, cb, cb), s);
              __syncwarp();
              put(at0, s[0], s[1]);
              put(at1, s[2], s[3]);
            }
            __syncwarp();
          }
        }
      }
      // ---- R ----
      if (!BF16) fetch_v();
      mbar_wait_warp(bar(X), ph, abort_flag);
      tc_fence_after();
      // What the last product is added to -- q rows: the prefix term, k rows: R -- waits in the second accumulator's columns.
      if (live) {
        const uint32_t r_row = sbase + C::oS + (uint32_t)(c0 >> 6) * 8192u + (uint32_t)i * 128u, ch0 = (uint32_t)(c0 & 63) >> 3;
        const float P = P_s[i], be = be_s[i];
        const bool node = i < T;
        Pair seen = pack(0.f, 0.f);
#pragma unroll 1
        for (int c = 0; c < CW / 16; ++c) {   // 16 columns
          uint32_t x[16], y[16];
          if (DELTA || !key) {
            tmem_ld16(tmem + lane_addr + c0 + 16u * c, x);
            tmem_ld16(tmem + lane_addr + DVC + c0 + 16u * c, y);
            tmem_wait_ld();
          }
          if (!key) {
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              Pair s = add2(pack(__uint_as_float(x[e]), __uint_as_float(x[e + 1])), pack(__uint_as_float(y[e]), __uint_as_float(y[e + 1])));
              s = mul2(mul2(s, pack(C::kXDown, C::kXDown)), pack(P, P));
              const float2 s2 = unpack(s);
              y[e] = __float_as_uint(s2.x);
              y[e + 1] = __float_as_uint(s2.y);
            }
          } else {
#pragma unroll
            for (int g = 0; g < 2; ++g) {   // eight columns: 16 bytes of a piece
              uint32_t hi[4], mid[4], lo[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int n = 8 * g + 2 * e, w = 4 * g + e;
                Pair rr = BF16 ? pack(__uint_as_float(vv[w % NV] << 16), __uint_as_float(vv[w % NV] & 0xffff0000u))
                               : pack(__uint_as_float(vv[n % NV]), __uint_as_float(vv[(n + 1) % NV]));
                if (DELTA) {
                  Pair s = pack(__uint_as_float(x[n]), __uint_as_float(x[n + 1]));
                  s = mul2(add2(s, pack(__uint_as_float(y[n]), __uint_as_float(y[n + 1]))), pack(C::kXDown, C::kXDown));
                  rr = mul2(fma2(s, pack(-P, -P), rr), pack(be, be));
                }
                if (!node) rr = pack(0.f, 0.f);
                seen = watch(seen, rr);
                const float2 r2 = unpack(rr);
                y[n] = __float_as_uint(r2.x);
                y[n + 1] = __float_as_uint(r2.y);
                if (C::NR == 3) split3(rr, hi[e], mid[e], lo[e]);
                else hi[e] = pack_rn(r2.x, r2.y);
              }
              const uint32_t to = r_row + ((ch0 + 2u * c + g) ^ (uint32_t)(i & 7)) * 16u;
              sts128(to, hi[0], hi[1], hi[2], hi[3]);
              if (C::NR == 3) {
                sts128(to + C::kRPiece, mid[0], mid[1], mid[2], mid[3]);
                sts128(to + 2 * C::kRPiece, lo[0], lo[1], lo[2], lo[3]);
              }
            }
#pragma unroll
            for (int e = 0; e < NV / 2; ++e) vv[e] = vv[e + NV / 2];   // the next 16 columns (CW = 32)
          }
          __syncwarp();
          tmem_st16(tmem + lane_addr + DVC + c0 + 16u * c, y);
        }
        tmem_wait_st();
        if (key && spotted(seen)) {   // nothing of this row may meet another node's zero coefficient
          atomicOr(&bad_s[4 * it + (i >> 5)], 1u << (i & 31));
          *any_bad = 1;
#pragma unroll 1
          for (int p = 0; p < C::NR; ++p)
#pragma unroll
            for (uint32_t g = 0; g < CW / 8; ++g) sts128(r_row + (uint32_t)p * C::kRPiece + ((ch0 + g) ^ (uint32_t)(i & 7)) * 16u, 0u, 0u, 0u, 0u);
        }
      }
      tc_fence_before();
      arrive(RP);
      sync();
      // ---- C N and N - I as three pieces, the A operand of the last product, in the columns of the scores ----
      if (live && cg < nb && (DELTA || !key)) {
        uint64_t m = mask_s[i];   // k rows: strict ancestors, R itself is added where the rows leave
        if (!key && i < T) m |= 1ull << i;
        const uint32_t on = (uint32_t)(m >> (16 * cg));
        Pair x2[8];
        if (!PATHS) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (cg <= b) x = lds128(blk(key ? 2 : 0, b, cg) + chunk(r16, q));
            const uint32_t o = on >> (4 * q);
            x2[2 * q] = pack(o & 1 ? __uint_as_float(x.x) : 0.f, o & 2 ? __uint_as_float(x.y) : 0.f);
            x2[2 * q + 1] = pack(o & 4 ? __uint_as_float(x.z) : 0.f, o & 8 ? __uint_as_float(x.w) : 0.f);
          }
        } else {
          const uint32_t from = slots + (key ? C::kMat : 0u);
          const uint32_t dw[4] = {depths.x, depths.y, depths.z, depths.w};
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            float x[2] = {0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 2; ++e)
              if ((on >> (2 * k + e)) & 1)
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x[e]) : "r"(from ^ ((dw[k >> 1] >> (8 * (2 * (k & 1) + e))) & 255u)) : "memory");
            x2[k] = pack(x[0], x[1]);
          }
        }
        uint32_t hi[8], mid[8], lo[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) split3(x2[k], hi[k], mid[k], lo[k]);
        __syncwarp();
        tmem_st8(sc_col + lane_addr + 8u * cg, hi);
        tmem_st8(sc_col + lane_addr + 32u + 8u * cg, mid);
        tmem_st8(sc_col + lane_addr + 64u + 8u * cg, lo);
        tmem_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(COEF));
      // ---- outputs: 32 rows of the warp's columns through its own staging area, whole lines to memory ----
      mbar_wait_warp(bar(ACC), ph, abort_flag);
      tc_fence_after();
      float* const out = key ? a.U : a.O;
      if (live && out != nullptr) {
        constexpr int NC = CW / 4;   // 16-byte chunks of a staged row
        const uint32_t stage = sbase + C::oS + (uint32_t)warp * C::kStage;
        Pair seen = pack(0.f, 0.f);
#pragma unroll 1
        for (int c = 0; c < CW / 16; ++c) {
          uint32_t x[16], y[16];
          tmem_ld16(tmem + lane_addr + DVC + c0 + 16u * c, y);
          if (DELTA || !key) tmem_ld16(tmem + lane_addr + c0 + 16u * c, x);
          tmem_wait_ld();
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            Pair z[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int k = 4 * g + 2 * e;
              z[e] = pack(__uint_as_float(y[k]), __uint_as_float(y[k + 1]));
              if (DELTA || !key) z[e] = fma2(pack(__uint_as_float(x[k]), __uint_as_float(x[k + 1])), pack(C::kLastDown, C::kLastDown), z[e]);
              seen = watch(seen, z[e]);
            }
            const float2 z0 = unpack(z[0]), z1 = unpack(z[1]);
            // eight rows a wavefront: 128-byte rows are swizzled by row, 64-byte rows by pair of rows
            const uint32_t at = NC == 8 ? (uint32_t)((4 * c + g) ^ (lane & 7)) : (uint32_t)(g ^ ((lane >> 1) & 3));
            sts128(stage + (uint32_t)lane * (CW * 4u) + at * 16u, __float_as_uint(z0.x), __float_as_uint(z0.y),
                   __float_as_uint(z1.x), __float_as_uint(z1.y));
          }
        }
        tc_fence_before();
        __syncwarp();
        constexpr int RP_ = 32 / NC;   // rows of a pass
        const int r0 = lane / NC, cc = lane % NC, n = T - (quad & 1) * 32 - r0;   // of this lane's rows, those below n are nodes
        float* o = out + pl.o0 + (size_t)((int64_t)((quad & 1) * 32 + r0) * a.lay.out.t) + c0 + 4 * cc;
#pragma unroll
        for (int j = 0; j < 32 / RP_; ++j) {
          const int row = r0 + RP_ * j;
          const uint4 w = lds128(stage + (uint32_t)row * (CW * 4u) + (uint32_t)(NC == 8 ? cc ^ (row & 7) : cc ^ ((row >> 1) & 3)) * 16u);
          if (RP_ * j < n)
            asm volatile("st.global.L1::no_allocate.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(o + (int64_t)(RP_ * j) * a.lay.out.t),
                         "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w) : "memory");
        }
        if (i < T && spotted(seen)) {
          atomicOr(&bad_s[4 * it + 2 + (i >> 5)], 1u << (i & 31));
          *any_bad = 1;
        }
      }
      if (more) sync();   // the staged rows have been read
    }
  } else {
    set_registers_down<kServiceRegs>();
    if (warp == kWorkers) {
      // ===================== products =====================
      if (lane == 0) {
        const uint64_t dQK = desc_kmajor(sbase + C::oQK), dS = desc_kmajor(sbase + C::oS), dR = desc_mnmajor(sbase + C::oS, 8192);
        constexpr uint32_t kIdSc = idesc_bf16(kNodes, false), kIdX = idesc_bf16(DVC, false), kIdR = idesc_bf16(DVC, true);
        using OS = Order<C::NP, C::NP>;
        using OX = Order<C::NP, 3>;
        using OR = Order<3, C::NR>;
#pragma unroll 1
        for (int it = 0; it < n_it; ++it) {
          const uint32_t ph = it & 1, set = BF16 ? (ph * C::kQKSet) >> 4 : 0;
          // scores
          if (!mbar_wait(bar(QK), ph, abort_flag)) break;
          const int nb = (place_s[ph].n + 15) >> 4;
          tc_fence_after();
#pragma unroll 1
          for (uint32_t h = 0; h < 2; ++h)   // halves of the contraction: an accumulator each
#pragma unroll 1
            for (int o = 0; o < OS::n; ++o) {
              const uint32_t pa = (OS::code >> (4 * o)) & 3u, pb = (OS::code >> (4 * o + 2)) & 3u;
              const uint64_t dA = dQK + set + ((pa * KH * C::kHalf + h * C::kStep) >> 4), dB = dQK + set + ((pb * KH * C::kHalf + h * C::kStep + 8192u) >> 4);
#pragma unroll
              for (uint32_t k = 0; k < DK / 32; ++k)
                mma_bf16_ss(sc_col + 64u * h, dA + ((k * 32u) >> 4), dB + ((k * 32u) >> 4), kIdSc, o > 0 || k > 0);
            }
          tc_commit(bar(SC));
          // state product
          bool ok = true;
#pragma unroll 1
          for (uint32_t h = 0; h < 2; ++h) {
            if (h < KH && !(ok = mbar_wait(bar(ST + (int)h), ph, abort_flag))) break;
            tc_fence_after();
#pragma unroll 1
            for (int o = 0; o < OX::n; ++o) {
              const uint32_t pa = (OX::code >> (4 * o)) & 3u, pb = (OX::code >> (4 * o + 2)) & 3u;
              const uint64_t dA = dQK + set + ((pa * KH * C::kHalf + h * C::kStep) >> 4), dB = dS + ((pb * KH * C::kSHalf + h * (KH == 2 ? C::kSHalf : 64u)) >> 4);
#pragma unroll
              for (uint32_t k = 0; k < DK / 32; ++k)
                mma_bf16_ss(tmem + DVC * h, dA + ((k * 32u) >> 4), dB + ((k * 32u) >> 4), kIdX, o > 0 || k > 0);
            }
          }
          if (!ok) break;
          tc_commit(bar(X));
          // [C N ; N - I] R
          if (!mbar_wait(bar(COEF), ph, abort_flag) || !mbar_wait(bar(RP), ph, abort_flag)) break;
          tc_fence_after();
#pragma unroll 1
          for (int o = 0; o < OR::n; ++o) {
            const uint32_t pa = (OR::code >> (4 * o)) & 3u, pb = (OR::code >> (4 * o + 2)) & 3u;
            const uint32_t A = sc_col + pa * 32u;
            const uint64_t dB = dR + ((pb * C::kRPiece) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k) {   // 16 nodes
              if (k >= nb) break;
              mma_bf16_ts(tmem, A + k * 8u, dB + ((k * 2048u) >> 4), kIdR, o > 0 || k > 0);
            }
          }
          tc_commit(bar(ACC));
        }
      }
    } else if (warp < kWorkers + 3) {
      // ===================== tables: masks, gates and decay ratios, a node per thread =====================
      const int n = tid - 32 * (kWorkers + 1);
      float4* const jump4 = reinterpret_cast<float4*>(sm + C::oJump4);
      uint32_t* const up4 = reinterpret_cast<uint32_t*>(sm + C::oUp4);
#pragma unroll 1
      for (int it = 0; it < n_it; ++it) {
        const uint32_t ph = it & 1;
        // the tables of the item before have been read (and this one's place is known)
        if (it > 0) {
          mbar_wait_warp(bar(COEF), ph ^ 1, abort_flag);
          mbar_wait_warp(bar(RP), ph ^ 1, abort_flag);
        }
        const Place& pl = place_s[ph];
        const bool node = n < pl.n;
        uint64_t m = 0;
        float al = 1.f, be = 0.f;
        if (node) {
          m = a.tree.anc[(pl.meta0 + n) * 2];
          al = a.alpha[pl.g0 + (size_t)n * a.lay.gate.t];
          if (DELTA) be = a.beta[pl.g0 + (size_t)n * a.lay.gate.t];
        }
        link[n] = make_float2(al, __int_as_float(m ? 63 - __clzll((long long)m) : -1));
        mask_s[n] = m;
        be_s[n] = be;
        asm volatile("bar.sync 2, 64;" ::: "memory");
        // four steps up at a time: the ancestors and the products of alpha on the way to them
        {
          float w[4], acc = 1.f;
          uint32_t up = 0;
          int j = n;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (j >= 0) {
              const float2 y = link[j];
              acc *= y.x;
              j = __float_as_int(y.y);
            }
            w[e] = acc;
            up |= (uint32_t)(j & 255) << (8 * e);
          }
          jump4[n] = make_float4(w[0], w[1], w[2], w[3]);
          up4[n] = up;
        }
        asm volatile("bar.sync 2, 64;" ::: "memory");
        // the products of alpha from a node up to, not including, each node of its path
        const uint32_t row = sbase + C::oTab + 2 * C::kMat + (uint32_t)(((n >> 4) * ((n >> 4) + 1)) >> 1) * 1024u + (uint32_t)(n & 15) * 64u;
        const uint32_t swz = (uint32_t)((n & 15) >> 1) & 3u;
        auto put = [&](uint32_t col, float x) {
          asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + (col >> 4) * 1024u + ((((col & 15u) >> 2) ^ swz) << 4) + (col & 3u) * 4u), "f"(x) : "memory");
        };
        float w = 1.f;
        int j = node ? n : -1;
#pragma unroll 1
        while (j >= 0) {
          const float4 y = jump4[j];
          const uint32_t up = up4[j];
          put(j, w);
          if (!(up & 0x80u)) put(up & 255u, w * y.x);
          if (!(up & 0x8000u)) put((up >> 8) & 255u, w * y.y);
          if (!(up & 0x800000u)) put((up >> 16) & 255u, w * y.z);
          w *= y.w;
          j = (int32_t)up >> 24;
        }
        P_s[n] = w;
        if (PATHS) {
          const int depth = __popcll(m) & (kPath - 1);
          sm[C::oDepth + n] = (uint8_t)(4 * depth);
          j = n;
#pragma unroll 1
          for (int e = depth; e >= 0; --e) {
            sm[C::oPath + n * kPath + e] = (uint8_t)j;
            j = __float_as_int(link[j].y);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(TAB));
      }
    } else {
      // ===================== places; requests to L2: v of this item, all of the next =====================
      auto near = [](const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); };
      constexpr int ES = BF16 ? 2 : 4, QL = DK * ES / 128, VL = DVC * ES / 128;   // lines of a row
      auto near_v = [&](const Place& pl) {
        const char* v = reinterpret_cast<const char*>(a.v) + pl.v0 * ES;
        for (int x = lane; x < pl.n * VL; x += 32) near(v + (int64_t)(x / VL) * a.lay.v.t * ES + (x % VL) * 128);
      };
      near_v(place_s[0]);
#pragma unroll 1
      for (int it = 0; it < n_it; ++it) {
        mbar_wait_warp(bar(QK), it & 1, abort_flag);   // the item before is done with, this one's operands are here
        const bool more = it + 1 < n_it;
        if (more && lane == 0) set_place(it + 1);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(TAB));
        if (!more) break;
        const Place& pl = place_s[(it + 1) & 1];
        if (!BF16)   // bf16: requested by the workers, to shared memory
          for (int x = lane; x < pl.n * QL; x += 32) {
            const size_t at = (pl.qk0 + (size_t)((int64_t)(x / QL) * a.lay.qk.t)) * ES + (x % QL) * 128;
            near(reinterpret_cast<const char*>(a.q) + at);
            near(reinterpret_cast<const char*>(a.k) + at);
          }
        for (int x = lane; x < DVC * DK / 32; x += 32) near(pl.S + x * 32);
        near_v(pl);
      }
    }
  }

  // ---- teardown: every path comes here ----
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kWorkers)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kCols) : "memory");
  if (*abort_flag) {
    if (tid == 0 && status) atomicExch(status, (int)TV_ERR_DEVICE_TIMEOUT);
    return;
  }
  // (values of this part's own, so that none is kept through the pipeline for it)
  const VerifyArgs* args = &a;
  asm volatile("" : "+l"(args), "+l"(sm));
  if (*reinterpret_cast<volatile int*>(sm + C::oMisc + 8)) {   // any_bad
    if (!C::kRedoCall) redo_items<BF16, DELTA, DK, DVC>(*args, n_units, n_split, sm);
    else redo_items_call<BF16, DELTA, DK, DVC>(*args, n_units, n_split, sm);
  }
}

template <bool BF16, bool DELTA, int DK, int DVC, bool PATHS>
inline int prepare() {
  return allow_kernel(verify_exact_kernel<BF16, DELTA, DK, DVC, PATHS>, Cfg<BF16, DELTA, DK, DVC>::kSmem, 4 * kWorkerRegs + kServiceRegs, 5);
}

template <bool BF16, bool DELTA, int DK, int DVC, bool PATHS>
inline int launch(const VerifyArgs& a, int sms, int32_t* status, cudaStream_t stream) {
  static thread_local int configured_dev = -1;
  int dev = 0;
  TV_CUDA_TRY(cudaGetDevice(&dev));
  if (configured_dev != dev) {
    const int st = prepare<BF16, DELTA, DK, DVC, PATHS>();
    if (st != TV_OK) return st;
    configured_dev = dev;
  }
  const int n_split = a.dv / DVC;
  const int64_t units = (int64_t)a.L * a.B * a.H * n_split;
  if (units > 0x7fffffffLL) return TV_ERR_UNSUPPORTED;
  // One CTA per SM, more only where one would have more items than it keeps a record of: then the same number for every
  // SM, as no two run on one at the same time (4768 fp32 items of 33 nodes, 64 x 64: 462 us with 149 CTAs, 242 with 296).
  const int64_t waves = (units + (int64_t)kMaxItems * sms - 1) / ((int64_t)kMaxItems * sms);
  const int64_t grid = units < sms ? units : waves * sms;
  TV_CUDA_TRY(launch_dependent(verify_exact_kernel<BF16, DELTA, DK, DVC, PATHS>, (int)grid, kThreads,
                               Cfg<BF16, DELTA, DK, DVC>::kSmem, stream, a, (int)units, n_split, status));
  return TV_OK;
}

// bf16 operands at 128 x 128 come here for deep trees under the delta rule only: other kernels take the rest.
template <bool BF16, bool DELTA, bool PATHS>
constexpr bool kHasWide = !BF16 || (DELTA && !PATHS);

template <bool BF16, bool DELTA, bool PATHS>
inline int launch_width(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  const int sms = tv_sm_count();
  if (sms <= 0) return TV_ERR_CUDA;
  // 128 value columns in two halves where that leaves no SM with more than one of them
  const bool halves = a.dv == 64 || 2 * (int64_t)a.L * a.B * a.H <= sms;
  if (a.dk == 64)
    return halves ? launch<BF16, DELTA, 64, 64, PATHS>(a, sms, status, stream) : launch<BF16, DELTA, 64, 128, PATHS>(a, sms, status, stream);
  if (halves) return launch<BF16, DELTA, 128, 64, PATHS>(a, sms, status, stream);
  if constexpr (kHasWide<BF16, DELTA, PATHS>) return launch<BF16, DELTA, 128, 128, PATHS>(a, sms, status, stream);
  return TV_ERR_UNSUPPORTED;
}
template <bool BF16>
inline int launch_any(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  if (a.rule != TV_GATED_DELTA) return launch_width<BF16, false, false>(a, status, stream);
  return a.tree.max_depth_all < kPath ? launch_width<BF16, true, true>(a, status, stream) : launch_width<BF16, true, false>(a, status, stream);
}
template <bool BF16, bool DELTA, bool PATHS>
inline int prepare_width() {
  int st = prepare<BF16, DELTA, 64, 64, PATHS>();
  if (st == TV_OK) st = prepare<BF16, DELTA, 64, 128, PATHS>();
  if (st == TV_OK) st = prepare<BF16, DELTA, 128, 64, PATHS>();
  if constexpr (kHasWide<BF16, DELTA, PATHS>)
    if (st == TV_OK) st = prepare<BF16, DELTA, 128, 128, PATHS>();
  return st;
}
// The callers of tv_prepare_verify_exact do not know the depth.
template <bool BF16>
inline int prepare_any() {
  const int st = prepare_width<BF16, false, false>();
  return st == TV_OK ? prepare_width<BF16, true, false>() : st;
}

}  // namespace tvexact
