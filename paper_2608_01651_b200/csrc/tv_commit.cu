// Accepted-path commit (Section IV-D Eq. 10; Lemma 1 Eq. 3).
//
//   S_new[v][k] = P_a S_pre[v][k] + sum_{j in P(a)} (P_a/P_j) u_j[v] k_j[k]
//
// One CTA streams one (layer, request, head) state of dv x dk floats through
// registers exactly once: 16-byte loads issued back to back, the rank-len
// update applied from shared memory, 16-byte stores.  HBM-bound: 8 dk dv bytes
// per state against (1 + len) FMAs per element.
//
// The accepted path needs no parent walk: node indices grow along a
// root-to-node path, so the set bits of the 128-bit ancestor mask of a, plus a
// itself, are the path in topological order.
//
// Every kernel takes its tensors layer by layer from a table in its parameters (Section IV-D /
// V-B: all linear layers are committed by one launch, whether they are stacked in one allocation
// or own their caches separately); work item -> (layer, request, head), tensors of that layer,
// rows addressed through the layout's strides within the layer.
#include <cuda_bf16.h>

#include "tv_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kPathChunk = 16;  // path rows staged in shared memory at a time
constexpr int kMaxVec = 16;     // float4 per thread: dk*dv <= 16384

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* base, size_t idx) {
  if (BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[idx]);
  return reinterpret_cast<const float*>(base)[idx];
}

// Work item -> layer and item within the layer.
struct LayerItem {
  int l, it;   // layer of this launch, (request, head) item inside the layer
  int b;       // request
};
__device__ __forceinline__ LayerItem layer_item(const CommitArgs& a, int item) {
  LayerItem r;
  const int bh = a.B * a.H;
  r.l = item / bh;
  r.it = item - r.l * bh;
  r.b = r.it / a.H;
  return r;
}
__device__ __forceinline__ ItemRows rows_of(const CommitArgs& a, int it_in_layer) {
  return tv_item_rows(a.tree, a.lay, it_in_layer, a.B, a.H, a.Hk, a.T, a.dk, a.dv);
}

// Fills path_s[0..len) (topological order), w_s[p] = P_a / P_path[p] and *Pa_s.
// al_s is scratch for the T decay gates (loaded by T threads in parallel so that
// the serial suffix product below never waits on global memory).
__device__ __forceinline__ int build_path(const TreeDev& tree, size_t meta0, int T, int acc,
                                          const float* alpha, size_t g0, int64_t g_rs, int* path_s, float* w_s,
                                          float* al_s, float* Pa_s) {
  const uint64_t* m = tree.anc + (meta0 + acc) * 2;
  const int t = threadIdx.x;
  if (t < T) al_s[t] = alpha[g0 + (size_t)t * g_rs];
  uint64_t m0 = m[0], m1 = m[1];
  if (acc < 64) m0 |= 1ull << acc; else m1 |= 1ull << (acc - 64);
  const int len = __popcll(m0) + __popcll(m1);
  if (t < 128) {
    const uint64_t w = t < 64 ? m0 : m1;
    const int bit = t & 63;
    if ((w >> bit) & 1) {
      int pos = __popcll(w & ((1ull << bit) - 1));
      if (t >= 64) pos += __popcll(m0);
      path_s[pos] = t;
    }
  }
  __syncthreads();
  if (t == 0) {
    float w = 1.f;
    for (int p = len - 1; p >= 0; --p) {
      w_s[p] = w;
      w *= al_s[path_s[p]];
    }
    *Pa_s = w;
  }
  __syncthreads();
  return len;
}

// Streaming 16-byte load / store: the state is touched exactly once.
__device__ __forceinline__ float4 ld_stream(const float4* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ void st_stream(float4* p, const float4& v) {
  asm volatile("st.global.L1::no_allocate.v4.f32 [%0], {%1,%2,%3,%4};"
               :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// Commit from given correction rows u_j: U (float) when given, else v.
template <bool BF16>
__global__ void __launch_bounds__(kThreads)
commit_factored_kernel(const CommitArgs a, const __grid_constant__ CommitLayers tb) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // dependent launch: nothing is read before the kernel in front is done
  __shared__ int path_s[TV_MAX_NODES];
  __shared__ float w_s[TV_MAX_NODES];
  __shared__ float Pa_s;
  __shared__ float al_s[TV_MAX_NODES];
  __shared__ __align__(16) float k_s[kPathChunk][TV_MAX_DIM];
  __shared__ float cu_s[kPathChunk][TV_MAX_DIM];

  const LayerItem li = layer_item(a, blockIdx.x);
  const int tid = threadIdx.x;
  const int dk = a.dk, dv = a.dv;
  const ItemRows rows = rows_of(a, li.it);
  const int T = rows.n;
  const int n4 = dv * dk / 4;
  const size_t sbase = (size_t)li.it * dv * dk;
  const float4* src = reinterpret_cast<const float4*>(tb.S_pre[li.l] + sbase);
  float4* dst = reinterpret_cast<float4*>(tb.S_new[li.l] + sbase);
  const void* kg = tb.k[li.l];
  const void* vg = tb.v[li.l];
  const float* Ug = tb.U[li.l];

  int acc = a.accepted[li.b];
  if (acc >= T) acc = -1;
  if (acc < 0) {
    if (!a.in_place)
      for (int i = tid; i < n4; i += kThreads) st_stream(dst + i, ld_stream(src + i));
    return;
  }
  // The whole state goes in flight first; the path is worked out under its latency.
  float4 s[kMaxVec];
#pragma unroll
  for (int e = 0; e < kMaxVec; ++e) {
    const int i = tid + e * kThreads;
    if (i < n4) s[e] = ld_stream(src + i);
  }
  const int len = build_path(a.tree, rows.meta0, T, acc, tb.alpha[li.l], rows.g0, rows.g_rs, path_s, w_s, al_s, &Pa_s);
  const float Pa = Pa_s;
#pragma unroll
  for (int e = 0; e < kMaxVec; ++e) {
    s[e].x *= Pa; s[e].y *= Pa; s[e].z *= Pa; s[e].w *= Pa;
  }
  const int dk4 = dk >> 2;
  for (int c0 = 0; c0 < len; c0 += kPathChunk) {
    const int nc = min(kPathChunk, len - c0);
    __syncthreads();
    for (int i = tid; i < nc * dk; i += kThreads) {
      const int p = i / dk, kk = i - p * dk;
      k_s[p][kk] = load_elem<BF16>(kg, rows.qk0 + (size_t)path_s[c0 + p] * rows.qk_rs + kk);
    }
    for (int i = tid; i < nc * dv; i += kThreads) {
      const int p = i / dv, vv = i - p * dv;
      const float u = a.has_U ? Ug[rows.o0 + (size_t)path_s[c0 + p] * rows.o_rs + vv]
                              : load_elem<BF16>(vg, rows.v0 + (size_t)path_s[c0 + p] * rows.v_rs + vv);
      cu_s[p][vv] = w_s[c0 + p] * u;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kMaxVec; ++e) {
      const int i = tid + e * kThreads;
      if (i < n4) {
        const int row = i / dk4, c4 = i - row * dk4;
        for (int p = 0; p < nc; ++p) {
          const float cu = cu_s[p][row];
          const float4 kv = *reinterpret_cast<const float4*>(&k_s[p][c4 * 4]);
          s[e].x = fmaf(cu, kv.x, s[e].x);
          s[e].y = fmaf(cu, kv.y, s[e].y);
          s[e].z = fmaf(cu, kv.z, s[e].z);
          s[e].w = fmaf(cu, kv.w, s[e].w);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < kMaxVec; ++e) {
    const int i = tid + e * kThreads;
    if (i < n4) st_stream(dst + i, s[e]);
  }
}

// dk = 64 and 128.  A CTA of 4 warps owns 4 * RPT * SUB consecutive rows (value channels) of one
// state; DK / 4 lanes own one float4 column each (SUB = 128 / DK rows side by side in a warp), so every
// load and store of a warp is whole rows of 256 or 512 bytes and the key row k_j[4 c .. 4 c + 3] stays in
// registers across the thread's RPT rows.  All its loads are in flight before anything else happens.
// Behind them is one chain of three dependent reads -- accepted node, its mask, the path's rows -- and
// nothing in it is serial over the path: the thread of a node finds the node's place by counting mask
// bits, a warp scan turns the gates into weights while the rows of up to 16 path nodes are on their way.
// A chain that loaded those rows one by one and scanned the gates with one thread took 23.5 us where this
// takes 21.7 (1024 items of 128 x 128, 20.5 at the copy peak), 4.2 against 2.3 at 16 items, and 24.1
// against 16.8 on paths of 40 nodes (256 items).  A persistent form of it with double-buffered rows was
// the slower one at every size too: 347 against 336 us on 16384 items.
constexpr int kRowThreads = 128;

// Four elements of a row, widened to float.
template <bool BF16>
__device__ __forceinline__ float4 widen4(const uint4& r) {
  if (BF16)
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
  return make_float4(__uint_as_float(r.x), __uint_as_float(r.y), __uint_as_float(r.z), __uint_as_float(r.w));
}
template <bool BF16>
__device__ __forceinline__ uint4 load_raw4(const void* base, size_t idx) {
  if (BF16) {
    const uint2 r = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(base) + idx);
    return make_uint4(r.x, r.y, 0u, 0u);
  }
  return *reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(base) + idx);
}

template <bool BF16, int DK, int RPT, int CTAS>
__global__ void __launch_bounds__(kRowThreads, CTAS)
commit_rows_kernel(const CommitArgs a, const __grid_constant__ CommitLayers tb) {
  constexpr int LPR = DK / 4, SUB = 32 / LPR, ROWS = 4 * RPT * SUB;
  constexpr int KQ = kPathChunk * LPR / kRowThreads;              // a thread's key quads of a chunk
  constexpr int UQ = kPathChunk * (ROWS / 4) / kRowThreads > 0 ? kPathChunk * (ROWS / 4) / kRowThreads : 1;
  __shared__ int path_s[TV_MAX_NODES];
  __shared__ __align__(16) float w_s[TV_MAX_NODES];
  __shared__ __align__(16) float al_s[TV_MAX_NODES];
  __shared__ float Pa_s;
  __shared__ __align__(16) float k_s[kPathChunk][DK];
  __shared__ __align__(16) float cu_s[kPathChunk][ROWS];

  const int dv = a.dv;
  const int n_part = (dv + ROWS - 1) / ROWS;
  const int item = blockIdx.x / n_part, part = blockIdx.x - item * n_part;
  const LayerItem li = layer_item(a, item);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int first = part * ROWS;                                  // of the CTA
  const int own = (warp * SUB + lane / LPR) * RPT;                // of the thread, within the CTA
  const int row0 = first + own;
  const size_t sbase = (size_t)li.it * dv * DK;
  const float4* src = reinterpret_cast<const float4*>(tb.S_pre[li.l] + sbase) + (size_t)row0 * LPR + lane % LPR;
  float4* dst = reinterpret_cast<float4*>(tb.S_new[li.l] + sbase) + (size_t)row0 * LPR + lane % LPR;

  int acc = a.accepted[li.b];
  if (acc >= a.T) acc = -1;
  // A request rejected in place has nothing to do, but not before the kernel in front is done: if every
  // request is rejected these are all the grid's threads, and the kernel behind -- an upload, a convolution --
  // waits for this grid only before it overwrites what the kernel in front (verify) may still be reading.
  float4 s[RPT];
  if (acc >= 0 || !a.in_place) {
#pragma unroll
    for (int e = 0; e < RPT; ++e)
      if (row0 + e < dv) s[e] = ld_stream(src + e * LPR);
  }
  // Dependent launch: this grid may have started under the tail of the kernel in front of it
  // (a verify kernel, or the tree-metadata kernel when no verify call sits in between).  S_pre
  // and the accepted nodes are older than either; everything those kernels write -- U, and the
  // tree metadata including the request offsets of a packed forest -- is read, and everything
  // they read that we write (S in place) is written, after this point.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const ItemRows rows = rows_of(a, li.it);
  const int T = rows.n;
  if (acc >= T) acc = -1;   // packed forest: beyond this request's node count
  if (acc < 0) {
    if (a.in_place) return;
#pragma unroll
    for (int e = 0; e < RPT; ++e)
      if (row0 + e < dv) st_stream(dst + e * LPR, s[e]);
    return;
  }
  const void* kg = tb.k[li.l];
  const void* vg = tb.v[li.l];
  const float* Ug = tb.U[li.l];

  // the path: thread t is node t
  int len;
  {
    const uint64_t* m = a.tree.anc + (rows.meta0 + acc) * 2;
    const float al = tid < T ? tb.alpha[li.l][rows.g0 + (size_t)tid * rows.g_rs] : 1.f;
    uint64_t m0 = m[0], m1 = m[1];
    if (acc < 64) m0 |= 1ull << acc; else m1 |= 1ull << (acc - 64);
    len = __popcll(m0) + __popcll(m1);
    const uint64_t w = tid < 64 ? m0 : m1, bit = 1ull << (tid & 63);
    const int pos = __popcll(w & (bit - 1)) + (tid < 64 ? 0 : __popcll(m0));
    if (w & bit) {
      path_s[pos] = tid;
      al_s[pos] = al;
    }
    if (tid >= len) al_s[tid] = 1.f;
  }
  __syncthreads();

  for (int c0 = 0; c0 < len; c0 += kPathChunk) {
    const int nc = min(kPathChunk, len - c0);
    uint4 kr[KQ], ur[UQ];
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
      const int i = tid + q * kRowThreads, p = i / LPR;
      if (p < nc) kr[q] = load_raw4<BF16>(kg, rows.qk0 + (size_t)((int64_t)path_s[c0 + p] * rows.qk_rs) + (i % LPR) * 4);
    }
#pragma unroll
    for (int q = 0; q < UQ; ++q) {
      const int i = tid + q * kRowThreads, p = i / (ROWS / 4), v = first + (i % (ROWS / 4)) * 4;
      ur[q] = make_uint4(0u, 0u, 0u, 0u);
      if (p < nc && v < dv)
        ur[q] = a.has_U ? load_raw4<false>(Ug, rows.o0 + (size_t)((int64_t)path_s[c0 + p] * rows.o_rs) + v)
                        : load_raw4<BF16>(vg, rows.v0 + (size_t)((int64_t)path_s[c0 + p] * rows.v_rs) + v);
    }
    if (c0 == 0) {
      if (warp == 0) {   // weights P_a / P_j: the product of the gates behind a position, four positions per lane
        const float4 x = *reinterpret_cast<const float4*>(&al_s[4 * lane]);
        const float x3 = x.w, x2 = x.z * x3, x1 = x.y * x2, x0 = x.x * x1;
        float behind = x0;   // product from this lane on
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float y = __shfl_down_sync(0xffffffffu, behind, o);
          if (lane + o < 32) behind *= y;
        }
        if (lane == 0) Pa_s = behind;
        float next = __shfl_down_sync(0xffffffffu, behind, 1);
        if (lane == 31) next = 1.f;
        *reinterpret_cast<float4*>(&w_s[4 * lane]) = make_float4(x1 * next, x2 * next, x3 * next, next);
      }
      __syncthreads();
      const float Pa = Pa_s;   // the first use of the state: its loads have had the path to land
#pragma unroll
      for (int e = 0; e < RPT; ++e) {
        s[e].x *= Pa; s[e].y *= Pa; s[e].z *= Pa; s[e].w *= Pa;
      }
    } else {
      __syncthreads();   // the chunk before has been read
    }
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
      const int i = tid + q * kRowThreads, p = i / LPR;
      if (p < nc) *reinterpret_cast<float4*>(&k_s[p][(i % LPR) * 4]) = widen4<BF16>(kr[q]);
    }
#pragma unroll
    for (int q = 0; q < UQ; ++q) {
      const int i = tid + q * kRowThreads, p = i / (ROWS / 4);
      if (p < nc) {
        const float w = w_s[c0 + p];
        const float4 u = a.has_U ? widen4<false>(ur[q]) : widen4<BF16>(ur[q]);
        *reinterpret_cast<float4*>(&cu_s[p][(i % (ROWS / 4)) * 4]) = make_float4(w * u.x, w * u.y, w * u.z, w * u.w);
      }
    }
    __syncthreads();
    for (int p = 0; p < nc; ++p) {
      const float4 kv = *reinterpret_cast<const float4*>(&k_s[p][(lane % LPR) * 4]);
#pragma unroll
      for (int q = 0; q < RPT / 4; ++q) {
        const float4 cu = *reinterpret_cast<const float4*>(&cu_s[p][own + q * 4]);
        const float c[4] = {cu.x, cu.y, cu.z, cu.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float4& x = s[q * 4 + t];
          x.x = fmaf(c[t], kv.x, x.x);
          x.y = fmaf(c[t], kv.y, x.y);
          x.z = fmaf(c[t], kv.z, x.z);
          x.w = fmaf(c[t], kv.w, x.w);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < RPT; ++e)
    if (row0 + e < dv) st_stream(dst + e * LPR, s[e]);
}

// Delta rule without stored corrections: every row v of the [dv][dk] state
// evolves independently along the accepted path,
//   s <- alpha_j s;  u = beta_j (v_j[v] - s . k_j);  s <- s + u k_j,
// which is the sequential rule restricted to one value channel.  A warp owns a
// row at a time (NPL consecutive floats per lane, dk = 32 NPL); the dot
// product is a shuffle reduction.
template <bool BF16, int NPL>
__global__ void __launch_bounds__(kThreads)
commit_delta_rows_kernel(const CommitArgs a, const __grid_constant__ CommitLayers tb) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // dependent launch: nothing is read before the kernel in front is done
  constexpr int DK = 32 * NPL;
  constexpr int kRowsPerWarp = TV_MAX_DIM / (kThreads / 32);  // 16
  __shared__ int path_s[TV_MAX_NODES];
  __shared__ float w_s[TV_MAX_NODES];
  __shared__ float Pa_s;
  __shared__ __align__(16) float k_s[kPathChunk][DK];
  __shared__ float v_s[kPathChunk][TV_MAX_DIM];
  __shared__ float alc_s[kPathChunk], be_s[kPathChunk];
  __shared__ float al_s[TV_MAX_NODES];

  const LayerItem li = layer_item(a, blockIdx.x);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dv = a.dv;
  const ItemRows rows = rows_of(a, li.it);
  const int T = rows.n;
  const size_t sbase = (size_t)li.it * dv * DK;
  const int n4 = dv * DK / 4;
  const float* Sp = tb.S_pre[li.l] + sbase;
  float* Sn = tb.S_new[li.l] + sbase;
  const void* kg = tb.k[li.l];
  const void* vg = tb.v[li.l];
  const float* beta = tb.beta[li.l];

  int acc = a.accepted[li.b];
  if (acc >= T) acc = -1;
  if (acc < 0) {
    if (!a.in_place) {
      const float4* src = reinterpret_cast<const float4*>(Sp);
      float4* dst = reinterpret_cast<float4*>(Sn);
      for (int i = tid; i < n4; i += kThreads) dst[i] = src[i];
    }
    return;
  }
  const int len = build_path(a.tree, rows.meta0, T, acc, tb.alpha[li.l], rows.g0, rows.g_rs, path_s, w_s, al_s, &Pa_s);

  float s[kRowsPerWarp][NPL];
#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r) {
    const int row = warp + r * (kThreads / 32);
    if (row < dv) {
      const float* p = Sp + (size_t)row * DK + lane * NPL;
      if (NPL == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        s[r][0] = t.x; s[r][1] = t.y; s[r][2 % NPL] = t.z; s[r][3 % NPL] = t.w;
      } else {
        const float2 t = *reinterpret_cast<const float2*>(p);
        s[r][0] = t.x; s[r][1] = t.y;
      }
    }
  }
  for (int c0 = 0; c0 < len; c0 += kPathChunk) {
    const int nc = min(kPathChunk, len - c0);
    __syncthreads();
    for (int i = tid; i < nc * DK; i += kThreads) {
      const int p = i / DK, kk = i - p * DK;
      k_s[p][kk] = load_elem<BF16>(kg, rows.qk0 + (size_t)path_s[c0 + p] * rows.qk_rs + kk);
    }
    for (int i = tid; i < nc * dv; i += kThreads) {
      const int p = i / dv, vv = i - p * dv;
      v_s[p][vv] = load_elem<BF16>(vg, rows.v0 + (size_t)path_s[c0 + p] * rows.v_rs + vv);
    }
    if (tid < nc) {
      alc_s[tid] = al_s[path_s[c0 + tid]];
      be_s[tid] = beta[rows.g0 + (size_t)path_s[c0 + tid] * rows.g_rs];
    }
    __syncthreads();
    for (int p = 0; p < nc; ++p) {
      float kr[NPL];
#pragma unroll
      for (int x = 0; x < NPL; ++x) kr[x] = k_s[p][lane * NPL + x];
      const float al = alc_s[p], be = be_s[p];
#pragma unroll
      for (int r = 0; r < kRowsPerWarp; ++r) {
        const int row = warp + r * (kThreads / 32);
        if (row < dv) {
          float dot = 0.f;
#pragma unroll
          for (int x = 0; x < NPL; ++x) {
            s[r][x] *= al;
            dot = fmaf(s[r][x], kr[x], dot);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
          const float u = be * (v_s[p][row] - dot);
#pragma unroll
          for (int x = 0; x < NPL; ++x) s[r][x] = fmaf(u, kr[x], s[r][x]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r) {
    const int row = warp + r * (kThreads / 32);
    if (row < dv) {
      float* p = Sn + (size_t)row * DK + lane * NPL;
      if (NPL == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(s[r][0], s[r][1], s[r][2 % NPL], s[r][3 % NPL]);
      } else {
        *reinterpret_cast<float2*>(p) = make_float2(s[r][0], s[r][1]);
      }
    }
  }
}

// Programmatic dependent launch behind the verify kernel (which releases its dependents once the
// tree metadata it waited for is complete): the commit grid is scheduled as SMs drain, and every
// thread of every kernel launched this way passes griddepcontrol.wait before it ends, so that a commit
// never ends before the kernel in front of it.  Behind any other kernel this is an ordinary launch.
cudaError_t launch_after_verify(void (*kernel)(const CommitArgs, const CommitLayers), int ctas, cudaStream_t stream,
                                const CommitArgs& a, const CommitLayers& tb, int threads = kRowThreads) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a, tb);
}

// Rows per thread.  Four (and no limit on registers) while that puts at most four CTAs on an SM: nothing
// but the chain counts there (16 items of 128 x 128: 2.3 us, 3.1 with sixteen rows).  Four, eight CTAs per
// SM, while all of them are resident (128 items: 4.6 us against 5.2 with eight rows).  Beyond that
// 64 rows per CTA -- sixteen per thread, eight for dk = 64: fewest paths to work out per byte (a round of
// 1024 items 53.2 us against 55.8 with half as many rows, of 512 items 40.4 against 41.1).  The register
// limits of the dk = 64 kernels (8 CTAs per SM, 7 with f32 keys) cost up to 24 bytes of spills.
template <bool BF16, int DK>
cudaError_t launch_rows(const CommitArgs& a, const CommitLayers& tb, int items, int sms, cudaStream_t stream) {
  constexpr int kRpt = DK == 128 ? 16 : 8, kCtas = DK == 128 ? 4 : BF16 ? 8 : 7;   // 64 rows per CTA
  constexpr int rows4 = 16 * (128 / DK), rows = 64;
  const int64_t ctas4 = (int64_t)items * ((a.dv + rows4 - 1) / rows4);
  if (ctas4 <= 4 * sms) return launch_after_verify(commit_rows_kernel<BF16, DK, 4, 4>, (int)ctas4, stream, a, tb);
  if (ctas4 <= 8 * sms) return launch_after_verify(commit_rows_kernel<BF16, DK, 4, 8>, (int)ctas4, stream, a, tb);
  const int ctas = items * ((a.dv + rows - 1) / rows);
  // From 30 CTAs per SM on an ordinary launch: most CTAs start long after the kernel in front is done, and
  // the dependent launch is the slower one.  Rounds of 64-node trees, dependent against ordinary: 128 x 128
  // states (two CTAs each) 1024 items 52.4 / 55.4 us, 2048 107.6 / 105.7, 4096 220 / 214, 24576 1290 / 1240;
  // 64 x 64 states (one CTA each) 2048 items 47.6 / 50.8, 4096 94.1 / 95.6, 8192 186 / 183, 24576 552 / 533.
  if (ctas >= 30 * sms) {
    commit_rows_kernel<BF16, DK, kRpt, kCtas><<<ctas, kRowThreads, 0, stream>>>(a, tb);
    return cudaSuccess;   // the caller asks for the launch's error
  }
  return launch_after_verify(commit_rows_kernel<BF16, DK, kRpt, kCtas>, ctas, stream, a, tb);
}

}  // namespace

int tv_launch_commit(const CommitArgs& a, const CommitLayers& tb, cudaStream_t stream) {
  if (a.L < 1 || a.L > kCommitMaxLayers) return TV_ERR_BAD_ARG;
  const int items = a.L * a.B * a.H;
  if ((size_t)a.dk * a.dv > (size_t)kMaxVec * kThreads * 4) return TV_ERR_UNSUPPORTED;
  const bool recompute = a.rule == TV_GATED_DELTA && !a.has_U;
  const int sms = tv_sm_count();
  if (sms == 0) return TV_ERR_CUDA;
  if (!recompute && a.dk == 128) {
    TV_CUDA_TRY((a.bf16 ? launch_rows<true, 128> : launch_rows<false, 128>)(a, tb, items, sms, stream));
  } else if (!recompute && a.dk == 64) {
    TV_CUDA_TRY((a.bf16 ? launch_rows<true, 64> : launch_rows<false, 64>)(a, tb, items, sms, stream));
  } else if (!recompute) {
    TV_CUDA_TRY(a.bf16 ? launch_after_verify(commit_factored_kernel<true>, items, stream, a, tb, kThreads)
                       : launch_after_verify(commit_factored_kernel<false>, items, stream, a, tb, kThreads));
  } else if (a.dk == 128) {
    TV_CUDA_TRY(a.bf16 ? launch_after_verify(commit_delta_rows_kernel<true, 4>, items, stream, a, tb, kThreads)
                       : launch_after_verify(commit_delta_rows_kernel<false, 4>, items, stream, a, tb, kThreads));
  } else if (a.dk == 64) {
    TV_CUDA_TRY(a.bf16 ? launch_after_verify(commit_delta_rows_kernel<true, 2>, items, stream, a, tb, kThreads)
                       : launch_after_verify(commit_delta_rows_kernel<false, 2>, items, stream, a, tb, kThreads));
  } else {
    return TV_ERR_UNSUPPORTED;
  }
  TV_CUDA_TRY(cudaGetLastError());
  return TV_OK;
}
