// Tree verification, general fp32 kernels (any T <= 128, dk, dv <= 128, f32 or bf16 operands, gated
// and delta rules).  All arithmetic is fp32 FMA, so they serve every shape that the tensor-core kernels
// refuse, the calls where they are ahead of the one of fp32 accuracy (tv_verify_exact.cu), and TV_IMPL_SIMT.
//
// One CTA per (layer, request, head) and chunk of value columns, following Theorem 1 (Eq. 2) in the
// factorised form of Eq. 4 / Lemma 2 (Eq. 5):
//   state    [Q; K] S_pre^T:  B0 = D_P Q S_pre^T,  R = D_beta (V - D_P K S_pre^T)  (gated: U = V)
//   scores   C_ij = (P_i / P_j) q_i.k_j and G_ij = beta_i (P_i / P_j) k_i.k_j on the tree's paths; the
//            decay ratio is a running product of alpha along the path, never a division
//   solve    delta rule: (I + G) U = R, which is triangular in topological order (Lemma 2)
//   readout  O = B0 + C U
// The sums over a path start from zero and meet R or B0 once, at the end: a term added to R itself rounds at
// R's size, which on a chain of 128 nodes left U with an error of 2.1e-7 where this leaves 0.7e-7.
// The state product is the same for every tree.  The rest has two forms:
//   paths    (at most 15 ancestors per node: every drafted tree) only the pairs that exist: eight
//            lanes walk up from a node and leave its coefficients in a table of 16 entries; nodes of
//            equal depth are solved together.  A tree of 63 nodes and depth 8 has about 300 pairs.
//   blocks   (deeper: chains) dense products [Q; K] K^T masked by the ancestor sets; block forward
//            substitution, 16 nodes at a time: one thread per column for the diagonal block, a
//            product over all threads for the rows below.
// The form is chosen per CTA from the masks (trees of up to 64 nodes), by the launcher from the depth it
// knows (up to 128 nodes, two row blocks), or per CTA of two launches where it does not.  In both, a node's
// sums run over the nodes of its path, whatever their coefficients are: a non-finite value stays on the
// paths through its node, and a zero gate, key or query below it does not hide it (0 x NaN and 0 x inf are
// NaN).
//
// What bounds it: fp32 FMA issue in the state product, and the latency of the short phases behind it
// with eight warps on an SM.  T = 63, 128 items, f32, delta: 27 us, of them 13 in the state product (8.6
// at the FMA rate); the one-item-per-CTA walk over global memory that was here before took 85.  A chain
// of 40 nodes, 256 items: 47 us against 490.  Products are accumulated in pairs over k
// (fma.rn.f32x2: even and odd k in one register pair, added at the end) and operands are read as
// 16-byte rows along k, so neither side is transposed and no value is duplicated.  A 16-byte read by
// a warp costs two shared-memory wavefronts where lanes (i, i ^ 1) or (i, i ^ 2) share an address and
// four otherwise: the thread grid below is laid out for the former.
#pragma once
#include <cuda_bf16.h>

#include "tv_internal.h"
#include "tv_tc_common.cuh"

namespace {

constexpr int kLD = TV_MAX_DIM + 4;  // floats between operand rows: 33 16-byte words, 8 consecutive rows miss each other's banks
constexpr int kMaskParts = 8;         // 16-bit parts of a node's mask of 128 bits
constexpr int kPath = 16;            // entries of a node's coefficient table: itself and 15 ancestors

// 4 consecutive elements starting at idx (idx % 4 == 0) widened to float.
template <bool BF16>
__device__ __forceinline__ float4 load4(const void* base, size_t idx) {
  if (BF16) {
    const uint2 r = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(base) + idx);
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
  }
  return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + idx);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// acc.lo += a.lo * b.lo, acc.hi += a.hi * b.hi
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float pair_sum(uint64_t x) {
  return __uint_as_float((uint32_t)x) + __uint_as_float((uint32_t)(x >> 32));
}

// `nodes` rows of an operand, from element `first` on and `rs` elements apart, widened to float.
template <bool BF16, int WARPS>
__device__ __forceinline__ void load_rows(float* dst, const void* src, size_t first, int64_t rs, int nodes, int dk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (BF16) {
    // two rows per warp and pass, eight elements per lane; four passes in flight
    const int c = (lane & 15) * 8, r0 = warp * 2 + (lane >> 4);
    if (c >= dk) return;
    const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(src) + first + c;
    for (int r = r0; r < nodes; r += 8 * WARPS) {
      uint4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r + u * 2 * WARPS < nodes) x[u] = *reinterpret_cast<const uint4*>(p + (int64_t)(r + u * 2 * WARPS) * rs);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (r + u * 2 * WARPS >= nodes) break;
        float4* d = reinterpret_cast<float4*>(dst + (r + u * 2 * WARPS) * kLD + c);
        d[0] = make_float4(__uint_as_float(x[u].x << 16), __uint_as_float(x[u].x & 0xffff0000u),
                           __uint_as_float(x[u].y << 16), __uint_as_float(x[u].y & 0xffff0000u));
        d[1] = make_float4(__uint_as_float(x[u].z << 16), __uint_as_float(x[u].z & 0xffff0000u),
                           __uint_as_float(x[u].w << 16), __uint_as_float(x[u].w & 0xffff0000u));
      }
    }
  } else {
    const int c = lane * 4;
    if (c >= dk) return;
    const float* p = reinterpret_cast<const float*>(src) + first + c;
    for (int r = warp; r < nodes; r += WARPS) cp_async16(tvtc::smem_u32(dst + r * kLD + c), p + (int64_t)r * rs);
  }
}

// acc[r][n] = x_r . y_n over dk channels: rows r < MT are 16 rows apart from x on, rows r >= MT the same
// from x + x2 on; columns are CT rows apart from y on.  SKIP: the lower triangle of a diagonal block
// (row tile m ends at row 16 m + 15, column tile n starts at row CT n).
template <int MT, int RT, int NT, int CT, bool SKIP>
__device__ __forceinline__ void product(uint64_t (&acc)[RT][NT], const float* x, int x2, const float* y, int dk) {
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[r][n] = 0;
#pragma unroll (RT * NT >= 32 ? 1 : 4)   // a large tile hides its own reads; unrolled, 8 x 8 is 5 % slower
  for (int k = 0; k < dk; k += 4) {
    ulonglong2 yv[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) yv[n] = *reinterpret_cast<const ulonglong2*>(y + n * CT * kLD + k);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const int m = r % MT;
      const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(x + (r / MT) * x2 + 16 * m * kLD + k);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        if (SKIP && CT * n > 16 * m + 15) continue;
        fma2(acc[r][n], xv.x, yv[n].x);
        fma2(acc[r][n], xv.y, yv[n].y);
      }
    }
  }
}

__device__ __forceinline__ void fma4(float4& o, float s, const float4& u) {
  o.x = fmaf(s, u.x, o.x);
  o.y = fmaf(s, u.y, o.y);
  o.z = fmaf(s, u.z, o.z);
  o.w = fmaf(s, u.w, o.w);
}

__device__ __forceinline__ float4 add4(const float4& a, const float4& b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 sub4(const float4& a, const float4& b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}

// out[m][h] += the sum over the nodes j of one block of 16 that lie on the row's path: w_m[j] * U[j][column
// quad h], for the row tiles m >= m0.  w_m: row tile m of a coefficient matrix (16 rows of `wld` floats apart);
// on: the block's part of the path mask of the thread's first row.
template <int MT, int NC>
__device__ __forceinline__ void accumulate16(float4 (&out)[MT][NC], int m0, const float* w, int wld, const uint16_t* on,
                                             const float* U, int ustride, int hstep) {
  uint32_t path[MT];
#pragma unroll
  for (int m = 0; m < MT; ++m) path[m] = m < m0 ? 0u : on[16 * m * kMaskParts];
#pragma unroll (MT > 2 ? 2 : 1)   // MT = 2, unrolled: the kernel, at its limit of 128 registers, is 8 % slower
  for (int j = 0; j < 16; j += 4) {
    float4 u[4][NC];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int h = 0; h < NC; ++h) u[x][h] = *reinterpret_cast<const float4*>(U + (j + x) * ustride + h * hstep);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      if (m < m0) continue;
      const float4 c = *reinterpret_cast<const float4*>(w + 16 * m * wld + j);
      const float cj[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if ((path[m] >> (j + x)) & 1) {   // whatever U and the coefficients hold off the path stays out
#pragma unroll
          for (int h = 0; h < NC; ++h) fma4(out[m][h], cj[x], u[x][h]);
        }
    }
  }
}

// Forward substitution of one diagonal block of 16 nodes, one thread per column.  on: the block's part of
// the path mask of its first node.
__device__ __forceinline__ void solve16(float* u, int ustride, const float* g, int gld, const uint16_t* on) {
  float r[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = u[i * ustride];
#pragma unroll
  for (int i = 1; i < 16; ++i) {
    const uint32_t path = on[i * kMaskParts];
    float known = 0.f;
#pragma unroll
    for (int j = 0; j < i; j += 4) {
      const float4 w = *reinterpret_cast<const float4*>(g + i * gld + j);
      const float wj[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (j + x < i && ((path >> (j + x)) & 1)) known = fmaf(wj[x], r[j + x], known);
    }
    r[i] -= known;
  }
#pragma unroll
  for (int i = 1; i < 16; ++i) u[i * ustride] = r[i];
}

// Tables of an item in shared memory, entries past the tree included (no path, alpha = beta = 0).
struct Tables {
  float2* link;     // alpha and the parent (int bits, -1 at a root child) of every node
  float* beta;
  uint64_t* path;   // [2] per node: the node and its ancestors
  // Part b of node i's mask: nodes 16 b .. 16 b + 15.
  __device__ __forceinline__ const uint16_t* on(int i, int b) const {
    return reinterpret_cast<const uint16_t*>(path) + i * kMaskParts + b;
  }
};

// One node per thread: reads masks and gates, fills the tables, returns the node's ancestor count.
template <bool DELTA>
__device__ __forceinline__ int load_meta(const VerifyArgs& a, const ItemRows& rows, int entries, const Tables& t) {
  const int tid = threadIdx.x;
  if (tid >= entries) return 0;
  uint64_t m0 = 0, m1 = 0;
  float al = 0.f, be = 0.f;
  if (tid < rows.n) {
    m0 = a.tree.anc[(rows.meta0 + tid) * 2];
    m1 = a.tree.anc[(rows.meta0 + tid) * 2 + 1];
    al = a.alpha[rows.g0 + (size_t)tid * rows.g_rs];
    if (DELTA) be = a.beta[rows.g0 + (size_t)tid * rows.g_rs];
  }
  const int parent = m1 ? 127 - __clzll((long long)m1) : m0 ? 63 - __clzll((long long)m0) : -1;
  const uint64_t self = tid < rows.n ? 1ull << (tid & 63) : 0;
  t.path[2 * tid] = tid < 64 ? m0 | self : m0;
  t.path[2 * tid + 1] = tid < 64 ? m1 : m1 | self;
  t.link[tid] = make_float2(al, __int_as_float(parent));
  t.beta[tid] = be;
  return __popcll(m0) + __popcll(m1);
}

// Block form.  jump[i]: the product of alpha over the 16 nodes from i upwards and the node after them
// (-1 past the root), by pointer doubling; P[i] from whole jumps.  All threads.
__device__ __forceinline__ void build_jumps(const Tables& t, float2* jump, float* P, int n) {
  const int tid = threadIdx.x;
  if (tid < n) jump[tid] = t.link[tid];
  __syncthreads();
#pragma unroll 1
  for (int r = 0; r < 4; ++r) {
    float2 x = make_float2(0.f, 0.f);
    if (tid < n) {
      x = jump[tid];
      const int up = __float_as_int(x.y);
      if (up >= 0) {
        const float2 y = jump[up];
        x = make_float2(x.x * y.x, y.y);
      }
    }
    __syncthreads();
    if (tid < n) jump[tid] = x;
    __syncthreads();
  }
  if (tid < n) {
    float2 x = jump[tid];
    float p = x.x;
    for (int up = __float_as_int(x.y); up >= 0; up = __float_as_int(x.y)) {
      x = jump[up];
      p *= x.x;
    }
    P[tid] = p;
  }
}

// Block form: multiplies the entries of rows i0 .. i0 + nb - 1 of C (and G) by the decay ratio (G: also by
// beta).  A task is 16 steps of a node's path; it gets to its first node by jumps.
template <bool DELTA, int THREADS>
__device__ __forceinline__ void scale_rows(const Tables& t, const float2* jump, float* C_s, float* G_s, int gld, int i0,
                                           int nb, int segments) {
  for (int x = threadIdx.x; x < nb * segments; x += THREADS) {
    const int i = x % nb;
    int j = i0 + i;
    float w = 1.f;
    for (int u = x / nb; u > 0 && j >= 0; --u) {
      const float2 y = jump[j];
      w *= y.x;
      j = __float_as_int(y.y);
    }
    const float be = DELTA ? t.beta[i0 + i] : 0.f;
    float* c = C_s + i * gld;
    float* g = G_s + i * gld;
    for (int u = 0; u < 16 && j >= 0; ++u) {
      c[j] *= w;
      if (DELTA) g[j] *= w * be;
      const float2 y = t.link[j];
      w *= y.x;
      j = __float_as_int(y.y);
    }
  }
}

// The chunk of the state: row 4 c + n of every 4 * CT rows goes to place n * CT + c, so that threads
// of neighbouring columns read neighbouring rows and each owns four consecutive columns.
template <int CT, int DVC, int WARPS>
__device__ __forceinline__ void load_state(float* S_s, const float* Sg, int n_rows, int dk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane * 4 >= dk) return;
  for (int r = warp; r < DVC && r < n_rows; r += WARPS) {
    const int q = r % (4 * CT), place = r - q + (q & 3) * CT + (q >> 2);
    cp_async16(tvtc::smem_u32(S_s + place * kLD + lane * 4), Sg + (size_t)r * dk + lane * 4);
  }
}

// The tree of a work item.
__device__ __forceinline__ int tree_of(const VerifyArgs& a, int item) {
  return a.tree.n_trees == 1 ? 0 : item / a.H % a.B;
}

// BF16, DELTA: operand type and rule.  MT: a thread's node rows (16 MT nodes in a row block).
// CT, NC: column threads and column quads of a thread (4 CT NC value columns in the CTA's chunk, 16 CT
// threads).  NBLK: row blocks (two: path form only).
template <int MT, int CT, int NC, int NBLK>
struct Cfg {
  static constexpr int kThreads = 16 * CT, kWarps = kThreads / 32;
  static constexpr int NB = 16 * MT;              // nodes of a row block
  static constexpr int N = NB * NBLK;
  static constexpr int DVC = 4 * CT * NC;         // value columns of the CTA
  static constexpr bool kBlockForm = NBLK == 1 && N > kPath;   // 16 nodes have at most 15 ancestors
  // One row block: U and B0 take the state's place, C and G (block form) that of the operand rows.
  // Two: U takes the k rows' place and B0 the q rows', block by block.
  // shared memory, in floats: q rows and k rows of block 0 (, of block 1), state, tables
  static constexpr int oS = 2 * N * kLD;
  static constexpr int oC = oS + DVC * kLD;          // path form: C entries [N][kPath], from the node upwards
  static constexpr int oG = oC + kPath * N;          // and G entries
  static constexpr int oIdx = oG + kPath * N;        // uint8 [N][kPath]: their nodes
  static constexpr int oDep = oIdx + kPath * N / 4;  // uint8 [N]: depths
  static constexpr int oOrd = oDep + N / 4;          // uint8 [N]: nodes by depth
  static constexpr int oLev = oOrd + N / 4;          // int [kPath + 1]: first place of every depth
  static constexpr int oMask = oLev + 20;
  static constexpr int oLink = oMask + 4 * N;
  static constexpr int oP = oLink + 2 * N;
  static constexpr int oBe = oP + N;
  static constexpr size_t kSmem = sizeof(float) * (oBe + N);
  static_assert(NBLK == 2 || 2 * N * DVC <= DVC * kLD, "U and B0 fit the state's place");
  static_assert(NBLK == 1 || DVC <= kLD, "U and B0 rows fit the operands' place");
  static_assert(NBLK == 2 || NB % CT == 0, "whole score columns");
  static_assert(kSmem <= 232448, "shared memory of one CTA");
  static_assert(kThreads >= N, "one thread per node");
  // CTAs per SM: what shared memory and registers hold (the tiles of 6 x 8 and 8 x 8 pair accumulators
  // take up to 255, the smaller ones 128)
  static constexpr int kBySmem = (int)(233472 / (kSmem + 1024));
  static constexpr int kByRegs = (MT * NC > 4 ? 256 : 512) / kThreads;
  static constexpr int kCtas = NBLK == 2 ? 1 : kBySmem < kByRegs ? kBySmem : kByRegs;
  __device__ static __forceinline__ int q_row(int i) { return NBLK == 1 ? i : i + (i / NB) * NB; }
  __device__ static __forceinline__ int k_row(int i) { return q_row(i) + NB; }
  __device__ static __forceinline__ float* U(float* sm, int i) {
    return NBLK == 1 ? sm + oS + i * DVC : sm + k_row(i) * kLD;
  }
  __device__ static __forceinline__ float* B0(float* sm, int i) {
    return NBLK == 1 ? sm + oS + (N + i) * DVC : sm + q_row(i) * kLD;
  }
};

template <bool BF16, bool DELTA, int MT, int CT, int NC, int NBLK>
__global__ void __launch_bounds__(16 * CT, Cfg<MT, CT, NC, NBLK>::kCtas)
verify_simt_kernel(const __grid_constant__ VerifyArgs a, int n_split) {
  using C = Cfg<MT, CT, NC, NBLK>;
  constexpr int RT = DELTA ? 2 * MT : MT;   // a thread's rows of the products: q (and k) of its nodes
  extern __shared__ __align__(16) float sm[];
  float* const X = sm;
  float* const S_s = sm + C::oS;
  float* const Cp_s = sm + C::oC;
  float* const Gp_s = sm + C::oG;
  uint8_t* const idx_s = reinterpret_cast<uint8_t*>(sm + C::oIdx);
  uint8_t* const dep_s = reinterpret_cast<uint8_t*>(sm + C::oDep);
  uint8_t* const ord_s = reinterpret_cast<uint8_t*>(sm + C::oOrd);
  int* const lev_s = reinterpret_cast<int*>(sm + C::oLev);
  const Tables tab = {reinterpret_cast<float2*>(sm + C::oLink), sm + C::oBe, reinterpret_cast<uint64_t*>(sm + C::oMask)};
  float* const P_s = sm + C::oP;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a warp covers 8 node rows x 4 column groups of the thread grid of 16 x CT
  const int rt = (warp & 1) * 8 + ((lane >> 1) & 7), ct = (warp >> 1) * 4 + (lane & 1) + (lane >> 4) * 2;
  const int dk = a.dk, dv = a.dv;
  const int item = blockIdx.x / n_split, v_first = (blockIdx.x - item * n_split) * C::DVC;

  if (NBLK == 2 && a.max_depth != nullptr) {   // of unknown depth: the deeper trees are the kernel's below
    tvtc::grid_dependency_wait();
    if (a.max_depth[tree_of(a, item)] >= kPath) return;
  }
  // The state is never the output of a kernel that releases its dependents early: its chunk is
  // requested before the dependency wait.
  load_state<CT, C::DVC, C::kWarps>(S_s, a.S_pre + ((size_t)item * dv + v_first) * dk, dv - v_first, dk);
  // Dependent launch on both sides: everything else -- the tree metadata may come from the kernel in
  // front -- is read after that kernel is done; the kernel behind this one may set itself up from
  // then on (the library's kernels read nothing this one writes before their own wait, and a
  // dependent released after the wait never runs beside anything older than this grid).
  tvtc::grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const ItemRows rows = tv_item_rows(a.tree, a.lay, item, a.B, a.H, a.Hk, a.T, dk, dv);
  const int T = rows.n;   // real nodes of this item (the whole slab unless the forest is packed)

#pragma unroll
  for (int I = 0; I < NBLK; ++I) {
    const size_t first = rows.qk0 + (size_t)((int64_t)(I * C::NB) * rows.qk_rs);
    const int n = min(T - I * C::NB, C::NB);
    load_rows<BF16, C::kWarps>(X + 2 * I * C::NB * kLD, a.q, first, rows.qk_rs, n, dk);
    load_rows<BF16, C::kWarps>(X + (2 * I + 1) * C::NB * kLD, a.k, first, rows.qk_rs, n, dk);
  }
  // the V rows are needed after the state product: bring them near
  {
    const int es = BF16 ? 2 : 4, per_row = C::DVC * es / 128 > 0 ? C::DVC * es / 128 : 1;
    for (int x = tid; x < T * per_row; x += C::kThreads) {
      const int i = x / per_row, c = (x - i * per_row) * (128 / es);
      if (v_first + c < dv)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(
            reinterpret_cast<const char*>(a.v) + (rows.v0 + (size_t)((int64_t)i * rows.v_rs) + v_first + c) * es));
    }
  }
  if (tid < kPath + 2) lev_s[tid] = 0;
  const int n_anc = load_meta<DELTA>(a, rows, C::N, tab);
  if (tid < C::N) dep_s[tid] = tid < T ? (uint8_t)n_anc : 255;
  const bool deep = __syncthreads_or(n_anc >= kPath) && C::kBlockForm;

  if (!deep) {
    // path form: every node's thread lists its path with the decay ratios, and the nodes by depth
    if (tid < T) {
      float w = 1.f;
      int j = tid;
      for (int e = 0; e <= n_anc; ++e) {
        idx_s[tid * kPath + e] = (uint8_t)j;
        Cp_s[tid * kPath + e] = w;
        const float2 y = tab.link[j];
        w *= y.x;
        j = __float_as_int(y.y);
      }
      P_s[tid] = w;
      const uint32_t d4 = (uint32_t)n_anc * 0x01010101u;
      int lt = 0, eq = 0, before = 0;
#pragma unroll
      for (int x = 0; x < C::N / 4; ++x) {
        const uint32_t y = reinterpret_cast<const uint32_t*>(dep_s)[x], same = __vcmpeq4(y, d4);
        lt += __popc(__vcmpltu4(y, d4));
        eq += __popc(same);
        const int mine = tid - 4 * x;   // nodes of this word in front of this one
        before += __popc(mine >= 4 ? same : mine > 0 ? same & ((1u << (8 * mine)) - 1) : 0u);
      }
      ord_s[(lt + before) >> 3] = (uint8_t)tid;
      lev_s[n_anc] = lt >> 3;
      lev_s[n_anc + 1] = (lt + eq) >> 3;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // scores: eight lanes per node, 16 channels each, two entries at a time
    const int s = lane & 7;
    for (int r0 = 0; r0 < T; r0 += C::kThreads / 8) {
      const int r = r0 + (tid >> 3), i = ord_s[min(r, T - 1)], n = r < T ? dep_s[i] : 0;
      const float* qi = X + C::q_row(i) * kLD + 4 * s;
      const float* ki = X + C::k_row(i) * kLD + 4 * s;
      float4 q[4], k[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        q[t] = k[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (32 * t + 4 * s < dk) {
          q[t] = *reinterpret_cast<const float4*>(qi + 32 * t);
          if (DELTA) k[t] = *reinterpret_cast<const float4*>(ki + 32 * t);
        }
      }
      const float be = DELTA ? tab.beta[i] : 0.f;
      const int n_warp = __reduce_max_sync(0xffffffffu, n);
      for (int e = 0; e <= n_warp; e += 2) {
        float c[2], g[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const float* kj = X + C::k_row(idx_s[i * kPath + min(e + x, n)]) * kLD + 4 * s;
          float c0 = 0.f, c1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (32 * t + 4 * s < dk) {
              const float4 y = *reinterpret_cast<const float4*>(kj + 32 * t);
              c0 = fmaf(q[t].x, y.x, c0); c1 = fmaf(q[t].y, y.y, c1);
              c0 = fmaf(q[t].z, y.z, c0); c1 = fmaf(q[t].w, y.w, c1);
              if (DELTA) {
                g0 = fmaf(k[t].x, y.x, g0); g1 = fmaf(k[t].y, y.y, g1);
                g0 = fmaf(k[t].z, y.z, g0); g1 = fmaf(k[t].w, y.w, g1);
              }
            }
          c[x] = c0 + c1;
          g[x] = g0 + g1;
        }
        // sums over the eight lanes: the upper four end up with g, lanes 2, 3 mod 4 with entry e + 1
        float z0, z1;
        if (DELTA) {
          const bool up = s & 4;
          z0 = (up ? g[0] : c[0]) + __shfl_xor_sync(0xffffffffu, up ? c[0] : g[0], 4);
          z1 = (up ? g[1] : c[1]) + __shfl_xor_sync(0xffffffffu, up ? c[1] : g[1], 4);
        } else {
          z0 = c[0] + __shfl_xor_sync(0xffffffffu, c[0], 4);
          z1 = c[1] + __shfl_xor_sync(0xffffffffu, c[1], 4);
        }
        const bool odd = s & 2;
        float z = (odd ? z1 : z0) + __shfl_xor_sync(0xffffffffu, odd ? z0 : z1, 2);
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        const int ex = e + (odd ? 1 : 0), at = i * kPath + ex;
        const bool mine = !(s & 1) && r < T && ex <= n;
        const float w = mine ? Cp_s[at] : 0.f;   // the decay ratio
        __syncwarp();
        if (mine) {
          if (!(s & 4)) Cp_s[at] = w * z;
          else if (DELTA) Gp_s[at] = be * (w * z);
        }
      }
    }
  } else {
    build_jumps(tab, reinterpret_cast<float2*>(Cp_s), P_s, C::N);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }

  // state
#pragma unroll 1
  for (int I = 0; I < NBLK; ++I) {
    if (I * C::NB >= T) break;
    uint64_t acc[RT][4 * NC];
    product<MT, RT, 4 * NC, CT, false>(acc, X + (2 * I * C::NB + rt) * kLD, C::NB * kLD, S_s + ct * kLD, dk);
    float4 vv[MT][NC];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const int i = I * C::NB + rt + 16 * m;
#pragma unroll
      for (int h = 0; h < NC; ++h) {
        const int c = v_first + 4 * (ct + h * CT);
        vv[m][h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < T && c < dv) vv[m][h] = load4<BF16>(a.v, rows.v0 + (size_t)((int64_t)i * rows.v_rs) + c);
      }
    }
    __syncthreads();   // U and B0 take the place of what has been read now; P is complete
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const int i = I * C::NB + rt + 16 * m;
      const float P = i < T ? P_s[i] : 0.f, be = DELTA ? tab.beta[i] : 0.f;
#pragma unroll
      for (int h = 0; h < NC; ++h) {
        const int c = 4 * (ct + h * CT);
        float4 r = vv[m][h];
        if (DELTA && i < T) {   // rows past the tree hold whatever the memory held: their U is zero
          r.x = be * (r.x - P * pair_sum(acc[MT + m][4 * h]));
          r.y = be * (r.y - P * pair_sum(acc[MT + m][4 * h + 1]));
          r.z = be * (r.z - P * pair_sum(acc[MT + m][4 * h + 2]));
          r.w = be * (r.w - P * pair_sum(acc[MT + m][4 * h + 3]));
        }
        *reinterpret_cast<float4*>(C::U(sm, i) + c) = r;
        *reinterpret_cast<float4*>(C::B0(sm, i) + c) =
            make_float4(P * pair_sum(acc[m][4 * h]), P * pair_sum(acc[m][4 * h + 1]), P * pair_sum(acc[m][4 * h + 2]),
                        P * pair_sum(acc[m][4 * h + 3]));
      }
    }
  }

  if (!deep) {
    // solve and readout, path form: DVC / 4 lanes per node
    constexpr int LN = C::DVC / 4, NN = C::kThreads / LN;   // lanes per node, nodes at a time
    const int n0 = tid / LN, c = 4 * (tid % LN);
    // entries first .. n of node i times the U rows they belong to
    auto along = [&](const float* w, int i, int first, int n) {
      float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
      const uint4 iv = *reinterpret_cast<const uint4*>(idx_s + i * kPath);
      const uint32_t word[4] = {iv.x, iv.y, iv.z, iv.w};
#pragma unroll
      for (int e4 = 0; e4 < kPath / 4; ++e4) {
        if (4 * e4 > n) break;
        const float4 x = *reinterpret_cast<const float4*>(w + i * kPath + 4 * e4);
        const float xe[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * e4 + e >= first && 4 * e4 + e <= n)
            fma4(sum, xe[e], *reinterpret_cast<const float4*>(C::U(sm, (word[e4] >> (8 * e)) & 255) + c));
      }
      return sum;
    };
    if (DELTA) {
      for (int lev = 1; lev < kPath; ++lev) {
        const int begin = lev_s[lev], end = lev_s[lev + 1];
        if (end <= begin) break;
        __syncthreads();   // the level above
        for (int r = begin + n0; r < end; r += NN) {
          const int i = ord_s[r];
          float4* const at = reinterpret_cast<float4*>(C::U(sm, i) + c);
          const float4 rhs = *at;
          *at = sub4(rhs, along(Gp_s, i, 1, lev));
        }
      }
    }
    __syncthreads();
    for (int r = n0; r < T; r += NN) {
      const int i = ord_s[r];
      const float4 b0 = *reinterpret_cast<const float4*>(C::B0(sm, i) + c);
      const float4 o = add4(b0, along(Cp_s, i, 0, dep_s[i]));
      if (v_first + c < dv) {
        const size_t at = rows.o0 + (size_t)((int64_t)i * rows.o_rs) + v_first + c;
        *reinterpret_cast<float4*>(a.O + at) = o;
        if (a.U) *reinterpret_cast<float4*>(a.U + at) = *reinterpret_cast<const float4*>(C::U(sm, i) + c);
      }
    }
    return;
  }

  if constexpr (C::kBlockForm) {
    constexpr int NTS = C::NB / CT;   // a thread's score columns
    constexpr int ULD = C::DVC, GLD = C::NB + 4;   // floats between rows of U; of C and G
    float* const C_s = X;
    float* const G_s = X + C::NB * GLD;
    float* const U_s = C::U(sm, 0);
    // scores, block form
    {
      uint64_t acc[RT][NTS];
      product<MT, RT, NTS, CT, true>(acc, X + rt * kLD, C::NB * kLD, X + (C::NB + ct) * kLD, dk);
      __syncthreads();   // C and G take the operand rows' place
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int i = rt + 16 * m;
#pragma unroll
        for (int n = 0; n < NTS; ++n) {
          const int j = ct + CT * n;
          C_s[i * GLD + j] = pair_sum(acc[m][n]);
          if (DELTA) G_s[i * GLD + j] = pair_sum(acc[MT + m][n]);
        }
      }
    }
    __syncthreads();
    scale_rows<DELTA, C::kThreads>(tab, reinterpret_cast<const float2*>(Cp_s), C_s, G_s, GLD, 0, C::NB, MT);
    __syncthreads();
    // solve, block form: tile by tile, each after the sum of what the tiles above it explain
    if (DELTA) {
      float4 known[MT][NC] = {};
#pragma unroll
      for (int b = 0; b < MT; ++b) {
        if (16 * b >= T) break;
        if (b > 0) {
          accumulate16<MT, NC>(known, b, G_s + rt * GLD + 16 * (b - 1), GLD, tab.on(rt, b - 1),
                               U_s + 16 * (b - 1) * ULD + 4 * ct, ULD, 4 * CT);
#pragma unroll
          for (int h = 0; h < NC; ++h) {
            float4* const at = reinterpret_cast<float4*>(U_s + (rt + 16 * b) * ULD + 4 * (ct + h * CT));
            *at = sub4(*at, known[b][h]);
          }
          __syncthreads();
        }
        if (tid < C::DVC) solve16(U_s + 16 * b * ULD + tid, ULD, G_s + 16 * b * GLD + 16 * b, GLD, tab.on(16 * b, b));
        __syncthreads();
      }
    }
    // readout, block form
    float4 o[MT][NC] = {};
#pragma unroll
    for (int b = 0; b < MT; ++b)
      accumulate16<MT, NC>(o, b, C_s + rt * GLD + 16 * b, GLD, tab.on(rt, b), U_s + 16 * b * ULD + 4 * ct, ULD, 4 * CT);
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int h = 0; h < NC; ++h) {
        const int i = rt + 16 * m, c = 4 * (ct + h * CT);
        if (i >= T || v_first + c >= dv) continue;
        const size_t at = rows.o0 + (size_t)((int64_t)i * rows.o_rs) + v_first + c;
        *reinterpret_cast<float4*>(a.O + at) = add4(*reinterpret_cast<const float4*>(C::B0(sm, i) + c), o[m][h]);
        if (a.U) *reinterpret_cast<float4*>(a.U + at) = *reinterpret_cast<const float4*>(U_s + i * ULD + c);
      }
  }
}

// Two row blocks of 16 MT nodes in the block form: deep trees of more than 64 nodes.  The second block's
// products with the first one's keys and corrections are full blocks.
template <bool DELTA, int MT>
struct DeepCfg {
  static constexpr int CT = 16, kThreads = 256, kWarps = 8, NB = 16 * MT, N = 2 * NB, DVC = 64;
  static constexpr int GLD = N + 4;
  // shared memory, in floats: q and k rows of the block, state (then block 0's keys), U, B0, C, G, tables
  static constexpr int oS = 2 * NB * kLD;
  static constexpr int oU = oS + DVC * kLD;
  static constexpr int oB0 = oU + N * DVC;
  static constexpr int oC = oB0 + NB * DVC;
  static constexpr int oG = oC + NB * GLD;
  static constexpr int oMask = oG + (DELTA ? NB * GLD : 0);
  static constexpr int oLink = oMask + 4 * N;
  static constexpr int oJump = oLink + 2 * N;
  static constexpr int oP = oJump + 2 * N;
  static constexpr int oBe = oP + N;
  static constexpr size_t kSmem = sizeof(float) * (oBe + N);
  static_assert(kSmem <= 232448 && NB <= DVC, "shared memory of one CTA; keys in the state's place");
};

template <bool BF16, bool DELTA, int MT>
__global__ void __launch_bounds__(256) verify_simt_deep_kernel(const __grid_constant__ VerifyArgs a, int n_split) {
  using C = DeepCfg<DELTA, MT>;
  constexpr int CT = C::CT, NB = C::NB, RT = DELTA ? 2 * MT : MT;
  extern __shared__ __align__(16) float sm[];
  float* const X = sm;
  float* const S_s = sm + C::oS;
  float* const U_s = sm + C::oU;
  float* const B0_s = sm + C::oB0;
  float* const C_s = sm + C::oC;
  float* const G_s = sm + C::oG;
  const Tables tab = {reinterpret_cast<float2*>(sm + C::oLink), sm + C::oBe, reinterpret_cast<uint64_t*>(sm + C::oMask)};
  float2* const jump_s = reinterpret_cast<float2*>(sm + C::oJump);
  float* const P_s = sm + C::oP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rt = (warp & 1) * 8 + ((lane >> 1) & 7), ct = (warp >> 1) * 4 + (lane & 1) + (lane >> 4) * 2;
  const int dk = a.dk, dv = a.dv;
  const int item = blockIdx.x / n_split, v_first = (blockIdx.x - item * n_split) * C::DVC;
  // launch order: as in the kernel above
  if (a.max_depth != nullptr) {
    tvtc::grid_dependency_wait();
    if (a.max_depth[tree_of(a, item)] < kPath) return;
  }
  load_state<CT, C::DVC, C::kWarps>(S_s, a.S_pre + ((size_t)item * dv + v_first) * dk, dv - v_first, dk);
  tvtc::grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const ItemRows rows = tv_item_rows(a.tree, a.lay, item, a.B, a.H, a.Hk, a.T, dk, dv);
  const int T = rows.n;
  load_meta<DELTA>(a, rows, C::N, tab);
  const int col = v_first + 4 * ct;   // the thread's four value columns
  for (int I = 0; I < 2 && I * NB < T; ++I) {
    const int i0 = I * NB;
    __syncthreads();   // tables; the first block's operand rows, C and G have been read
    {
      const size_t first = rows.qk0 + (size_t)((int64_t)i0 * rows.qk_rs);
      load_rows<BF16, C::kWarps>(X, a.q, first, rows.qk_rs, min(T - i0, NB), dk);
      load_rows<BF16, C::kWarps>(X + NB * kLD, a.k, first, rows.qk_rs, min(T - i0, NB), dk);
    }
    if (I == 0) build_jumps(tab, jump_s, P_s, C::N);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // state
    {
      uint64_t acc[RT][4];
      product<MT, RT, 4, CT, false>(acc, X + rt * kLD, NB * kLD, S_s + ct * kLD, dk);
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int i = i0 + rt + 16 * m;
        const float P = P_s[i];
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < T && col < dv) r = load4<BF16>(a.v, rows.v0 + (size_t)((int64_t)i * rows.v_rs) + col);
        if (DELTA && i < T) {
          const float be = tab.beta[i];
          r.x = be * (r.x - P * pair_sum(acc[MT + m][0]));
          r.y = be * (r.y - P * pair_sum(acc[MT + m][1]));
          r.z = be * (r.z - P * pair_sum(acc[MT + m][2]));
          r.w = be * (r.w - P * pair_sum(acc[MT + m][3]));
        }
        *reinterpret_cast<float4*>(U_s + i * C::DVC + 4 * ct) = r;
        *reinterpret_cast<float4*>(B0_s + (rt + 16 * m) * C::DVC + 4 * ct) = make_float4(
            P * pair_sum(acc[m][0]), P * pair_sum(acc[m][1]), P * pair_sum(acc[m][2]), P * pair_sum(acc[m][3]));
      }
    }
    // scores against the keys of this block and of the one before
    for (int J = 0; J <= I; ++J) {
      const float* Y = X + NB * kLD;
      if (J < I) {
        __syncthreads();   // the state has been read for the last time
        load_rows<BF16, C::kWarps>(S_s, a.k, rows.qk0, rows.qk_rs, NB, dk);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        Y = S_s;
      }
      uint64_t acc[RT][MT];
      product<MT, RT, MT, CT, false>(acc, X + rt * kLD, NB * kLD, Y + ct * kLD, dk);
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int i = rt + 16 * m;
#pragma unroll
        for (int n = 0; n < MT; ++n) {
          const int j = J * NB + ct + CT * n;
          C_s[i * C::GLD + j] = pair_sum(acc[m][n]);
          if (DELTA) G_s[i * C::GLD + j] = pair_sum(acc[MT + m][n]);
        }
      }
    }
    __syncthreads();
    scale_rows<DELTA, C::kThreads>(tab, jump_s, C_s, G_s, C::GLD, i0, NB, (I + 1) * MT);
    __syncthreads();
    // solve: what the first block explains of this one, then tile by tile as above
    if (DELTA) {
      float4 known[MT][1] = {};
      if (I > 0) {
#pragma unroll 1
        for (int b = 0; b < MT; ++b)
          accumulate16<MT, 1>(known, 0, G_s + rt * C::GLD + 16 * b, C::GLD, tab.on(i0 + rt, b),
                              U_s + 16 * b * C::DVC + 4 * ct, C::DVC, 0);
      }
#pragma unroll
      for (int b = 0; b < MT; ++b) {
        if (i0 + 16 * b >= T) break;
        if (b > 0)
          accumulate16<MT, 1>(known, b, G_s + rt * C::GLD + i0 + 16 * (b - 1), C::GLD, tab.on(i0 + rt, i0 / 16 + b - 1),
                              U_s + (i0 + 16 * (b - 1)) * C::DVC + 4 * ct, C::DVC, 0);
        if (I + b > 0) {
          float4* const at = reinterpret_cast<float4*>(U_s + (i0 + rt + 16 * b) * C::DVC + 4 * ct);
          *at = sub4(*at, known[b][0]);
          __syncthreads();
        }
        if (tid < C::DVC)
          solve16(U_s + (i0 + 16 * b) * C::DVC + tid, C::DVC, G_s + 16 * b * C::GLD + i0 + 16 * b, C::GLD,
                  tab.on(i0 + 16 * b, i0 / 16 + b));
        __syncthreads();
      }
    }
    // readout
    float4 o[MT][1] = {};
    if (I > 0) {
#pragma unroll 1
      for (int b = 0; b < MT; ++b)
        accumulate16<MT, 1>(o, 0, C_s + rt * C::GLD + 16 * b, C::GLD, tab.on(i0 + rt, b), U_s + 16 * b * C::DVC + 4 * ct,
                            C::DVC, 0);
    }
#pragma unroll
    for (int b = 0; b < MT; ++b)
      accumulate16<MT, 1>(o, b, C_s + rt * C::GLD + i0 + 16 * b, C::GLD, tab.on(i0 + rt, i0 / 16 + b),
                          U_s + (i0 + 16 * b) * C::DVC + 4 * ct, C::DVC, 0);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const int i = i0 + rt + 16 * m;
      if (i >= T || col >= dv) continue;
      const size_t at = rows.o0 + (size_t)((int64_t)i * rows.o_rs) + col;
      *reinterpret_cast<float4*>(a.O + at) =
          add4(*reinterpret_cast<const float4*>(B0_s + (rt + 16 * m) * C::DVC + 4 * ct), o[m][0]);
      if (a.U) *reinterpret_cast<float4*>(a.U + at) = *reinterpret_cast<const float4*>(U_s + i * C::DVC + 4 * ct);
    }
  }
}

int launch_kernel(void (*kern)(VerifyArgs, int), int threads, size_t smem, int dvc, int& configured_dev,
                  const VerifyArgs& a, cudaStream_t stream) {
  int dev = 0;
  TV_CUDA_TRY(cudaGetDevice(&dev));
  if (configured_dev != dev) {
    TV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    configured_dev = dev;
  }
  const int n_split = (a.dv + dvc - 1) / dvc;
  const int64_t grid = (int64_t)a.L * a.B * a.H * n_split;
  if (grid > 0x7fffffffLL) return TV_ERR_UNSUPPORTED;
  TV_CUDA_TRY(tvtc::launch_dependent(kern, (int)grid, threads, smem, stream, a, n_split));
  return TV_OK;
}

template <bool BF16, bool DELTA, int MT, int CT, int NC, int NBLK>
int launch(const VerifyArgs& a, cudaStream_t stream) {
  using C = Cfg<MT, CT, NC, NBLK>;
  static thread_local int configured_dev = -1;
  return launch_kernel(verify_simt_kernel<BF16, DELTA, MT, CT, NC, NBLK>, C::kThreads, C::kSmem, C::DVC, configured_dev,
                       a, stream);
}

template <bool BF16, bool DELTA, int MT>
int launch_deep(const VerifyArgs& a, cudaStream_t stream) {
  using C = DeepCfg<DELTA, MT>;
  static thread_local int configured_dev = -1;
  return launch_kernel(verify_simt_deep_kernel<BF16, DELTA, MT>, C::kThreads, C::kSmem, C::DVC, configured_dev, a, stream);
}

// Up to 64 nodes.  Every chunk of value columns computes the item's scores again, so a chunk is all 128
// columns where there are enough items to fill the SMs, else 64 or 32 (T = 64, f32, delta: 128 items
// 27.9 us in whole columns, 32.9 in halves; 64 items 25 us in halves).
template <bool BF16, bool DELTA, int MT>
int launch_one(const VerifyArgs& a, int sms, cudaStream_t stream) {
  const int64_t items = (int64_t)a.L * a.B * a.H;
  if (a.dv <= 32 || items * ((a.dv + 31) / 32) <= sms) return launch<BF16, DELTA, MT, 8, 1, 1>(a, stream);
  if (a.dv <= 64 || items * ((a.dv + 63) / 64) <= sms) return launch<BF16, DELTA, MT, 8, 2, 1>(a, stream);
  return launch<BF16, DELTA, MT, 16, 2, 1>(a, stream);
}

template <bool BF16, bool DELTA, int MT>
int launch_two(const VerifyArgs& a, int sms, cudaStream_t stream) {
  const int64_t items = (int64_t)a.L * a.B * a.H;
  if (a.dv <= 32 || items * ((a.dv + 31) / 32) <= sms) return launch<BF16, DELTA, MT, 8, 1, 2>(a, stream);
  if (a.dv <= 64 || items * ((a.dv + 63) / 64) <= sms) return launch<BF16, DELTA, MT, 16, 1, 2>(a, stream);
  return launch<BF16, DELTA, MT, 16, 2, 2>(a, stream);
}

template <bool BF16, bool DELTA>
int launch_nodes(const VerifyArgs& a, cudaStream_t stream) {
  const int sms = tv_sm_count();
  if (sms == 0) return TV_ERR_CUDA;
  if (a.T <= 16) return launch_one<BF16, DELTA, 1>(a, sms, stream);
  if (a.T <= 32) return launch_one<BF16, DELTA, 2>(a, sms, stream);
  if (a.T <= 48) return launch_one<BF16, DELTA, 3>(a, sms, stream);
  if (a.T <= 64) return launch_one<BF16, DELTA, 4>(a, sms, stream);
  // two row blocks of 48 or 64 nodes
  if (a.tree.max_depth_all < kPath)
    return a.T <= 96 ? launch_two<BF16, DELTA, 3>(a, sms, stream) : launch_two<BF16, DELTA, 4>(a, sms, stream);
  // Depths that only the device knows: the block form serves every tree.  Under the gated rule with more items
  // than SMs its dense scores cost a shallow tree more than a second launch, in which such trees take the path
  // form (f32, depth 8, 160 / 512 items: 65 nodes 45 / 93 us against 68 / 167, 128 nodes 64 / 131 against 92 /
  // 225), and a deep tree loses nothing by it (chains of 128 nodes, 512 items: 256 us against 255).  Elsewhere
  // deep trees would: 65 nodes, 4 items 25.6 -> 27.3 us, delta rule, 512 items of 128 nodes 469 -> 475.
  VerifyArgs b = a;
  if (!DELTA && a.max_depth != nullptr && (int64_t)a.L * a.B * a.H > sms) {
    const int st = a.T <= 96 ? launch_two<BF16, DELTA, 3>(a, sms, stream) : launch_two<BF16, DELTA, 4>(a, sms, stream);
    if (st != TV_OK) return st;
  } else {
    b.max_depth = nullptr;   // every tree in one launch
  }
  return a.T <= 96 ? launch_deep<BF16, DELTA, 3>(b, stream) : launch_deep<BF16, DELTA, 4>(b, stream);
}

// Loads a kernel and allows its shared memory on the current device.
int prepare_kernel(void (*kern)(VerifyArgs, int), size_t smem) {
  TV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return TV_OK;
}
template <bool BF16, bool DELTA, int MT, int CT, int NC, int NBLK>
int prepare() {
  return prepare_kernel(verify_simt_kernel<BF16, DELTA, MT, CT, NC, NBLK>, Cfg<MT, CT, NC, NBLK>::kSmem);
}
template <bool BF16, bool DELTA, int MT>
int prepare_one() {
  int st = prepare<BF16, DELTA, MT, 8, 1, 1>();
  if (st == TV_OK) st = prepare<BF16, DELTA, MT, 8, 2, 1>();
  if (st == TV_OK) st = prepare<BF16, DELTA, MT, 16, 2, 1>();
  return st;
}
template <bool BF16, int MT>
int prepare_two() {
  int st = prepare<BF16, false, MT, 8, 1, 2>();
  if (st == TV_OK) st = prepare<BF16, false, MT, 16, 1, 2>();
  if (st == TV_OK) st = prepare<BF16, false, MT, 16, 2, 2>();
  return st;
}
template <bool BF16, bool DELTA>
int prepare_all() {
  int st = prepare_one<BF16, DELTA, 1>();
  if (st == TV_OK) st = prepare_one<BF16, DELTA, 2>();
  if (st == TV_OK) st = prepare_one<BF16, DELTA, 3>();
  if (st == TV_OK) st = prepare_one<BF16, DELTA, 4>();
  // the callers of tv_prepare_verify_simt do not know the depth: of the kernels for more than 64
  // nodes they reach the block form and, under the gated rule, the path form
  if (st == TV_OK) st = prepare_kernel(verify_simt_deep_kernel<BF16, DELTA, 3>, DeepCfg<DELTA, 3>::kSmem);
  if (st == TV_OK) st = prepare_kernel(verify_simt_deep_kernel<BF16, DELTA, 4>, DeepCfg<DELTA, 4>::kSmem);
  if constexpr (!DELTA) {
    if (st == TV_OK) st = prepare_two<BF16, 3>();
    if (st == TV_OK) st = prepare_two<BF16, 4>();
  }
  return st;
}

}  // namespace
