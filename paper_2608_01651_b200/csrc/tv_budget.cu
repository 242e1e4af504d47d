// Batch-wide utility allocation (Section V-A): score every candidate node by the drafter's
// probability of its whole path, keep the root of every tree plus the highest-scoring nodes of the
// whole batch up to a fixed budget, count per request, and pack the kept nodes into the padded
// parent slabs and offsets of a packed forest (Section V-B) -- all on the device, with fixed
// shapes, so the selection can sit inside a GPU-resident round.
//
// Up to 2048 candidates in at most as many requests as the GPU has SMs: two small launches, each dependent
// on the one in front of it:
//   budget_rho_kernel     one CTA per request: rho_i = rho_parent * p_i in float32, level by level
//                         (parent before child, one rounding per edge), and a 32-bit sort key
//   budget_choose_kernel  one CTA per request: every CTA finds the budget-th largest key of the batch
//                         for itself (all keys in its registers, two bits of the threshold per step,
//                         until exactly as many keys reach it as are wanted), counts what the requests in
//                         front of its own keep, then compacts its own request in order and renumbers the
//                         parents; ties go in (request, node) order
// Everything else takes three launches:
//   budget_rho_kernel, then
//   budget_select_kernel  one CTA: 4-pass radix select of the budget-th largest key, then per-request
//                         counts and their prefix sums
//   budget_pack_kernel    one CTA per request: order-preserving compaction and parent renumbering
// The sizes are tiny (at most a few 10^4 candidates): what counts is the chain of launches and of
// steps inside them.  A whole device-built round of 2048 candidates (32 requests, budget 1234) took 69.8 us
// with three ordinary launches, 61.2 us with these two and 60.0 us since the search ends early.  The search
// is steps of compares, one reduction and one barrier (some 0.25 us each): 16 of them to the last bit, 9 for 2048 spread
// probabilities, all 16 where ties decide.  Four warps of 16 keys a thread, three counts in one word and so one
// reduction a step, against eight warps with two reductions and all steps: 7.6 -> 5.45 us a selection of 2048 candidates
// in 16 or 32 requests, 7.3 -> 4.8 of 64 in one, 7.7 -> 7.7 where ties decide.  The early end is all of it: without
// it the four warps take 7.6 us, and 7.2 on 64 in one request.  One launch for everything, every CTA
// working out all scores, was slower: 8.7 us, and 37 on chains (7.6 and 12.4).
// Every request's CTA of the two-launch form searches all keys: its work is requests x candidates.  Device
// time of a selection of about 2000 candidates, two launches against three: 160 / 200 / 256 / 300 / 400 / 512 / 1024
// requests 7.2 / 6.5 / 6.6 / 8.7 / 10.7 / 11.5 / 12.9 us against 9.6 / 10.9 / 10.7 / 10.7 / 10.7 / 10.2 / 10.6, where ties
// decide 256 / 400 / 1024 requests 8.6 / 14.9 / 20.7 against 10.6 / 10.9 / 10.8.  The line is at one CTA per SM,
// where it was set when the search took all its steps (7.7 / 11.5 us on 148 / 300 requests against 10.9 / 10.3); since
// the shorter search two CTAs per SM would still be ahead, by 2 to 4 us, and nobody has moved it.  With 32
// keys per thread, which 2049 to 8192 candidates need, it was slower at any number of requests (on eight warps, searching
// to the last bit): 4096 candidates in 32 / 1024 requests 14.5 / 64 us against 11.4 / 11.4.
#include "tv_internal.h"
#include "tv_tc_common.cuh"

namespace {

constexpr int kSelThreads = 1024;

__global__ void __launch_bounds__(TV_MAX_NODES)
budget_rho_kernel(const int32_t* __restrict__ parent, const float* __restrict__ p, int32_t Tc,
                  float* __restrict__ rho, uint32_t* __restrict__ key, int32_t* status) {
  __shared__ int32_t par_s[TV_MAX_NODES];
  __shared__ float rho_s[TV_MAX_NODES];
  __shared__ int maxd_s;
  const int b = blockIdx.x, i = threadIdx.x;
  // Dependent launch on both sides: the candidates may be the output of the kernel in front, and an
  // earlier selection may still be reading the keys.
  tvtc::grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (i == 0) maxd_s = 0;
  int par = -1;
  float pi = 0.f;
  if (i < Tc) {
    par = parent[(size_t)b * Tc + i];
    pi = p[(size_t)b * Tc + i];
    if (par < -1 || par >= i || (i == 0 && par != -1)) {   // cannot be checked on the host
      par = -1;
      if (status) atomicExch(status, (int)TV_ERR_INVALID_TREE);
    }
    par_s[i] = par;
  }
  __syncthreads();
  int depth = 0;
  if (i < Tc) {
    for (int j = par; j >= 0 && depth < Tc; j = par_s[j]) ++depth;
    atomicMax(&maxd_s, depth);
  }
  __syncthreads();
  const int maxd = maxd_s;
  for (int d = 0; d <= maxd; ++d) {
    if (i < Tc && depth == d) rho_s[i] = par < 0 ? pi : __fmul_rn(rho_s[par], pi);
    __syncthreads();
  }
  if (i < Tc) {
    const float r = rho_s[i];
    rho[(size_t)b * Tc + i] = r;
    // non-negative floats order like their bit patterns; roots rank above everything
    key[(size_t)b * Tc + i] = i == 0 ? 0xffffffffu : (r >= 0.f ? __float_as_uint(r) : 0u);
  }
}

// Exclusive prefix sum of one int per thread over the CTA (kSelThreads threads).
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = warp_tot[lane];
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += up;
    }
    warp_tot[lane] = wi - w;   // exclusive over warps
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  return warp_tot[warp] + incl - v;
}

constexpr int kChooseThreads = 128, kChooseWarps = kChooseThreads / 32;
constexpr int KPT = 16;   // keys per thread, consecutive ones

__global__ void __launch_bounds__(kChooseThreads)
budget_choose_kernel(const uint32_t* __restrict__ key, const int32_t* parent, int32_t N, int32_t K,
                     int32_t B, int32_t Tc, int32_t budget, int32_t* __restrict__ counts, int32_t* __restrict__ offsets,
                     int32_t* parent_packed, int32_t* __restrict__ node_id) {
  static_assert(KPT * 32 < 1024 && KPT * kChooseThreads <= 2048, "counts of a warp in 10 bits, of the CTA in 12");
  static_assert(kChooseThreads == TV_MAX_NODES && kChooseWarps == 4, "a thread per node; four words are read at once");
  __shared__ __align__(16) uint32_t turn_s[2][kChooseWarps];
  __shared__ __align__(16) uint32_t front_s[2][kChooseWarps];
  __shared__ __align__(16) unsigned ballot_s[2][kChooseWarps];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  tvtc::grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int i0 = tid * KPT;
  uint32_t k[KPT];
#pragma unroll
  for (int x = 0; x < KPT; x += 4) {   // (keys lie on 16-byte boundaries)
    if (i0 + x + 4 <= N) {
      const uint4 y = *reinterpret_cast<const uint4*>(key + i0 + x);
      k[x] = y.x, k[x + 1] = y.y, k[x + 2] = y.z, k[x + 3] = y.w;
    } else {
#pragma unroll
      for (int z = 0; z < 4; ++z) k[x + z] = i0 + x + z < N ? key[i0 + x + z] : 0u;
    }
  }
  const bool node = tid < Tc;
  const uint32_t own = node ? key[(size_t)b * Tc + tid] : 0u;
  int par = node ? parent[(size_t)b * Tc + tid] : -1;   // (parent_packed may be the same buffer: read before any write)
  if (par < -1 || par >= tid) par = -1;

  // the largest tau that at least K keys reach, or any that exactly K reach: from the top, two bits at a
  // time (the places past N hold zero and every candidate is at least one).  Three counts share a word.
  uint32_t tau = 0;
#pragma unroll 1
  for (int shift = 30; shift >= 0; shift -= 2) {
    const uint32_t c1 = tau | 1u << shift, c2 = tau | 2u << shift, c3 = tau | 3u << shift;
    uint32_t n = 0;
#pragma unroll
    for (int x = 0; x < KPT; ++x) n += (k[x] >= c1 ? 1u : 0u) + (k[x] >= c2 ? 1u << 10 : 0u) + (k[x] >= c3 ? 1u << 20 : 0u);
    n = __reduce_add_sync(0xffffffffu, n);
    uint32_t* turn = turn_s[(shift >> 1) & 1];   // used again two steps on: one barrier per step is enough
    if (lane == 0) turn[warp] = n;
    __syncthreads();
    const uint4 w = *reinterpret_cast<const uint4*>(turn);
    const int n1 = (int)((w.x & 1023u) + (w.y & 1023u) + (w.z & 1023u) + (w.w & 1023u));
    const int n2 = (int)((w.x >> 10 & 1023u) + (w.y >> 10 & 1023u) + (w.z >> 10 & 1023u) + (w.w >> 10 & 1023u));
    const int n3 = (int)((w.x >> 20) + (w.y >> 20) + (w.z >> 20) + (w.w >> 20));
    tau = n3 >= K ? c3 : n2 >= K ? c2 : n1 >= K ? c1 : tau;
    if (n3 == K || n2 == K || n1 == K) break;   // (then tau is that one, and no lower bit changes the set)
  }
  // keys above tau, in the batch and in front of this request; keys equal to it in front of this request
  uint32_t above = 0, ties = 0;
  const int first = b * Tc;
#pragma unroll
  for (int x = 0; x < KPT; ++x) {
    const bool front = i0 + x < first;
    above += k[x] > tau ? (front ? 0x10001u : 1u) : 0u;
    ties += k[x] == tau && front ? 1u : 0u;
  }
  above = __reduce_add_sync(0xffffffffu, above);
  ties = __reduce_add_sync(0xffffffffu, ties);
  const bool tie = node && own == tau;
  const unsigned tie_ballot = __ballot_sync(0xffffffffu, tie);
  if (lane == 0) {
    front_s[0][warp] = above;
    front_s[1][warp] = ties;
    ballot_s[0][warp] = tie_ballot;
  }
  __syncthreads();
  above = ties = 0;
#pragma unroll
  for (int w = 0; w < kChooseWarps; ++w) {
    above += front_s[0][w];
    ties += front_s[1][w];
  }
  const int need = K - (int)(above & 0xffffu);      // keys equal to tau to take, in index order
  const int offset = (int)(above >> 16) + min(need, (int)ties);

  // this request's nodes
  int before = (int)ties + __popc(tie_ballot & ((1u << lane) - 1u));
#pragma unroll
  for (int w = 0; w < kChooseWarps; ++w)
    if (w < warp) before += __popc(ballot_s[0][w]);
  const bool flag = node && (own > tau || (tie && before < need));
  const unsigned ballot = __ballot_sync(0xffffffffu, flag);
  if (lane == 0) ballot_s[1][warp] = ballot;
  __syncthreads();
  int rank = __popc(ballot & ((1u << lane) - 1u)), count = 0, above_par = 0;
  unsigned par_word = 0;
#pragma unroll
  for (int w = 0; w < kChooseWarps; ++w) {
    const unsigned kept = ballot_s[1][w];
    const int c = __popc(kept);
    if (w < warp) rank += c;
    if (w < par >> 5) above_par += c;
    if (w == par >> 5) par_word = kept;
    count += c;
  }
  if (flag) {
    const unsigned bit = 1u << (par & 31);   // (-1 has no word: it stays without a parent, as one that was dropped)
    parent_packed[(size_t)b * Tc + rank] = par_word & bit ? above_par + __popc(par_word & (bit - 1u)) : -1;
    node_id[offset + rank] = b * Tc + tid;
  }
  if (node && tid >= count) parent_packed[(size_t)b * Tc + tid] = -1;    // padding of the slab
  if (tid == 0) {
    counts[b] = count;
    offsets[b] = offset;
    if (b == B - 1) offsets[B] = K;
  }
  if (b == 0)
    for (int j = K + tid; j < budget; j += kChooseThreads) node_id[j] = -1;   // rows past the forest
}

__global__ void __launch_bounds__(kSelThreads)
budget_select_kernel(const uint32_t* __restrict__ key, int32_t N, int32_t K, int32_t B, int32_t Tc,
                     uint8_t* __restrict__ keep, int32_t* __restrict__ counts, int32_t* __restrict__ offsets) {
  __shared__ int hist[256];
  __shared__ uint32_t prefix_s;
  __shared__ int need_s;
  __shared__ int warp_tot[32];
  __shared__ int total_s;
  __shared__ int cnt_s[kSelThreads];   // kept nodes per request (B <= kSelThreads)
  const int tid = threadIdx.x;
  cnt_s[tid] = 0;
  if (tid == 0) {
    prefix_s = 0;
    need_s = K;
  }
  // ---- the K-th largest key, one byte at a time from the top ----
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const uint32_t prefix = prefix_s;
    for (int i = tid; i < N; i += kSelThreads) {
      const uint32_t k = key[i];
      if (pass == 0 || (k >> (shift + 8)) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1);
    }
    __syncthreads();
    // the digit whose bucket holds the need-th largest key: thread t looks at digit 255 - t and
    // at the number of keys in the higher buckets (a prefix sum over the CTA, not a serial walk)
    {
      const int need = need_s;
      const int mine = tid < 256 ? hist[255 - tid] : 0;
      const int above = block_exclusive_scan(mine, warp_tot, &total_s);
      if (tid < 256 && above < need && above + mine >= need) {
        prefix_s = (prefix << 8) | (uint32_t)(255 - tid);
        need_s = need - above;   // how many keys with this prefix still have to be taken
      }
    }
    __syncthreads();
  }
  const uint32_t tau = prefix_s;   // the threshold key
  const int need = need_s;         // number of keys == tau to take, in index order
  // ---- flags: everything above the threshold, and the first `need` keys equal to it ----
  const int chunk = (N + kSelThreads - 1) / kSelThreads;
  const int i0 = tid * chunk, i1 = min(N, i0 + chunk);
  int ties = 0;
  for (int i = i0; i < i1; ++i) ties += key[i] == tau;
  int before = block_exclusive_scan(ties, warp_tot, &total_s);
  for (int i = i0; i < i1; ++i) {
    const uint32_t k = key[i];
    bool take = k > tau;
    if (k == tau) take = before++ < need;
    keep[i] = take ? 1 : 0;
    if (take) atomicAdd(&cnt_s[i / Tc], 1);
  }
  __syncthreads();
  // ---- per-request counts and their exclusive prefix sums (B <= kSelThreads) ----
  const int c = tid < B ? cnt_s[tid] : 0;
  const int off = block_exclusive_scan(c, warp_tot, &total_s);
  if (tid < B) {
    counts[tid] = c;
    offsets[tid] = off;
  }
  if (tid == 0) offsets[B] = total_s;
}

__global__ void __launch_bounds__(TV_MAX_NODES)
budget_pack_kernel(const int32_t* __restrict__ parent, const uint8_t* __restrict__ keep,
                   const int32_t* __restrict__ offsets, int32_t B, int32_t Tc, int32_t budget,
                   int32_t* __restrict__ parent_packed, int32_t* __restrict__ node_id) {
  __shared__ int rank_s[TV_MAX_NODES];
  __shared__ int warp_tot[4];
  const int b = blockIdx.x, i = threadIdx.x, lane = i & 31, warp = i >> 5;
  const bool flag = i < Tc && keep[(size_t)b * Tc + i] != 0;
  const unsigned ballot = __ballot_sync(0xffffffffu, flag);
  if (lane == 0) warp_tot[warp] = __popc(ballot);
  __syncthreads();
  int rank = __popc(ballot & ((1u << lane) - 1u));
  for (int w = 0; w < warp; ++w) rank += warp_tot[w];
  const int count = warp_tot[0] + warp_tot[1] + warp_tot[2] + warp_tot[3];
  rank_s[i] = flag ? rank : -1;
  __syncthreads();
  if (flag) {
    int par = parent[(size_t)b * Tc + i];
    if (par < -1 || par >= i) par = -1;
    parent_packed[(size_t)b * Tc + rank] = par < 0 ? -1 : rank_s[par];   // -1 also if the parent was dropped
    node_id[offsets[b] + rank] = b * Tc + i;
  }
  if (i >= count && i < Tc) parent_packed[(size_t)b * Tc + i] = -1;       // padding of the slab
  if (b == 0)
    for (int j = offsets[B] + i; j < budget; j += TV_MAX_NODES) node_id[j] = -1;   // rows past the forest
}

}  // namespace

#define TV_API __attribute__((visibility("default")))

extern "C" {

TV_API size_t tv_budget_workspace_bytes(int32_t n_req, int32_t n_cand) {
  if (n_req < 1 || n_cand < 1) return 0;
  const size_t N = (size_t)n_req * n_cand;
  return ((N * sizeof(uint32_t) + 255) & ~(size_t)255) + ((N + 255) & ~(size_t)255);
}

TV_API int tv_budget_select(const int32_t* parent, const float* p_draft, int32_t n_req, int32_t n_cand,
                            int32_t budget, float* rho, int32_t* counts, int32_t* offsets,
                            int32_t* parent_packed, int32_t* node_id, void* workspace, int32_t* status,
                            void* stream) {
  if (!parent || !p_draft || !rho || !counts || !offsets || !parent_packed || !node_id || !workspace)
    return TV_ERR_BAD_ARG;
  if (n_req < 1 || n_cand < 1 || budget < n_req) return TV_ERR_BAD_ARG;
  if (n_cand > TV_MAX_NODES || n_req > kSelThreads) return TV_ERR_UNSUPPORTED;
  if (((uintptr_t)parent | (uintptr_t)p_draft | (uintptr_t)rho | (uintptr_t)counts | (uintptr_t)offsets |
       (uintptr_t)parent_packed | (uintptr_t)node_id | (uintptr_t)status) & 3)
    return TV_ERR_BAD_ARG;
  if ((uintptr_t)workspace & 15) return TV_ERR_BAD_ARG;
  const int32_t N = n_req * n_cand;
  const int32_t K = budget < N ? budget : N;
  uint32_t* key = reinterpret_cast<uint32_t*>(workspace);
  uint8_t* keep = reinterpret_cast<uint8_t*>(workspace) + (((size_t)N * sizeof(uint32_t) + 255) & ~(size_t)255);
  cudaStream_t s = (cudaStream_t)stream;
  const int sms = tv_sm_count();
  if (sms == 0) return TV_ERR_CUDA;
  TV_CUDA_TRY(tvtc::launch_dependent(budget_rho_kernel, n_req, TV_MAX_NODES, 0, s, parent, p_draft, n_cand, rho, key,
                                     status));
  if (N <= KPT * kChooseThreads && n_req <= sms) {
    TV_CUDA_TRY(tvtc::launch_dependent(budget_choose_kernel, n_req, kChooseThreads, 0, s, (const uint32_t*)key, parent, N,
                                       K, n_req, n_cand, budget, counts, offsets, parent_packed, node_id));
    return TV_OK;
  }
  budget_select_kernel<<<1, kSelThreads, 0, s>>>(key, N, K, n_req, n_cand, keep, counts, offsets);
  TV_CUDA_TRY(cudaGetLastError());
  budget_pack_kernel<<<n_req, TV_MAX_NODES, 0, s>>>(parent, keep, offsets, n_req, n_cand, budget, parent_packed,
                                                   node_id);
  TV_CUDA_TRY(cudaGetLastError());
  return TV_OK;
}

}  // extern "C"
