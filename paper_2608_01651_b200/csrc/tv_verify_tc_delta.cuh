// Tree verification of the gated delta rule on the tensor cores (tcgen05 + TMEM + TMA).
//
// Shapes: bf16 q/k/v, fp32 state, dk = dv = 128, tree depth <= 15, dense batches (any strides) and
// packed forests.  NB = 1: up to 64 nodes, NB = 2: up to 128, worked on as two row blocks of 64.
//
// Algebra (Theorem 1, Eq. 2; Lemma 2/3).  With N = (I+G)^-1, A = N D_beta, W = C A, and
// V' = V - D_P K S_pre^T (the part of the correction that the old state does not hold already):
//     O = D_P Q S_pre^T + W V',     U = A V'
// so the state is contracted once, with the raw [Q ; K], and nothing of that product waits for the
// triangular systems.  G, C, N, A, W are T x T but ancestor-sparse: row i has entries only on the
// root-to-node path p_0 < ... < p_d = i of node i, and slot s of node i and of any descendant refer
// to the same node p_s.  Row i of W and of A come from ONE back-substitution each on the
// path-restricted unit triangular system (w L = c, x L = e_d; L = I + G on the path).  All decay
// factors are products of alpha over a stretch of the row's own path, never a quotient of two
// numbers that may both underflow.
//
// One half of a tile's 128 rows carries the O problem of the block's nodes (q rows), the other the U
// problem (k rows):
//     Sc  = [Q_b ; K_b] K^T                   scores, columns = all nodes up to the block's last
//     X   = [Q_b ; K_b] [S_hi + S_lo]^T       q/k exact, state as two bf16 (16 mantissa bits and more)
//     q rows of X *= P_i,  V' = V - P_i (k rows of X) -> bf16 hi + lo, then those rows = 0
//     X  += [W ; A]_hi V'_hi + [W ; A]_lo V'_hi + [W ; A]_hi V'_lo     q rows: O, k rows: U
// Block 0 has the q rows in front, block 1 the k rows: in memory Q_0 K_0 K_1 Q_1, so that K_0 K_1 is one
// operand of block 1's scores.
//
// What bounds it and how it is laid out.  At the copy rate an SM's share of the memory moves an item
// of 64 nodes in 4.1 us and one of 128 in 6.6; the dependent chain of one item is two to three times
// that.  So the chain is cut between five groups of four warps, each busy for less than that time and
// each working on a different item or block:
//     warps 0..3    TMA producer | MMAs of scores and readout | metadata (paths, gates, P of the items to
//                   come) | MMAs of the state product
//     warps 4..7    state rows split in place into bf16 hi + lo
//     warps 8..11   thread = tile row: scores of its path, back-substitution, row of [W ; A]
//     warps 12..15  finished rows of X to memory
//     warps 16..19  V' and the scaling of X
// and nothing of it is staged in a buffer that the next item needs: the coefficient rows are the A
// operand in tensor memory, in the columns of the scores they came from; the state arrives in a ring
// of four quarters of k (a quarter's fp32 rows of 128 bytes become [hi | lo] rows of the same bytes,
// so one 128-wide tile feeds the hi and the lo product); outputs pass through 2 or 4 KiB per warp.
// The state product has an issuing thread of its own, so that no product waits for another one's operands; one
// thread that polled for all three needed 150 ns per MMA.  Loops over columns stay rolled: all roles run at once
// and share one instruction cache (unrolled, 512 items of 24 / 128 nodes took 22.2 / 43.1 us, rolled 20.6 / 41.2).
//
// Measured, back to back / in rounds of upload, verify and commit, before (one chain of phases over eight warps,
// state as tf32, operand tiles and staged outputs sharing buffers) and now, us:
//     items x nodes   512 x 24       512 x 64       2048 x 64       512 x 128      2048 x 128
//     before          22.7 /  34.1   28.6 /  40.5   90.3 / 140.1    68.3 /  81.4   220 / 275
//     now             20.1 /  31.4   23.9 /  36.0   74.1 / 132.7    41.4 /  54.7   132 / 205
// Error against 64 bits 3e-4 before, 4.4e-6 now.  What is left: the four hops of an item (state product, V',
// readout, stores) over three or two sets of columns, with shared memory half busy.  Parts left out in a scratch
// build, all waits intact, 512 x 64 / 512 x 128: the output group's reads, staging and stores 19.9 / 32.9 us, its
// global stores alone 21.5 / 38.6, V' 22.1 / 38.7, scores and path systems 20.9 / 37.7.
//
// Values that are not finite: a gate's reaches the rows of its node's subtree (see the metadata warp); a q row's its own
// output row; a k or v row's or a state entry's every node of the (request, head), the entry's in its value column.
// Every wait is a bounded mbarrier wait (status word on expiry); every TMA load is a plain per-CTA copy.
#pragma once
#include "tv_tc_common.cuh"

namespace tvdelta {

using namespace tvtc;

constexpr int kThreads = 640;
constexpr int kSlots = 16;     // path slots per node: depth <= 15
constexpr int kBlk = 64;       // nodes per row block
constexpr int kLd = 17;        // row stride of the table of G (floats): conflict-free per slot
constexpr int kUnits = 4;      // quarters of k, ring slots of the state
// registers a thread, by group, out of 96 at launch; the V' group keeps its 96
constexpr int kServiceRegs = 64, kSplitRegs = 64, kPathRegs = 144, kOutRegs = 112;

template <int NB>
struct Map {
  static constexpr int kNodes = kBlk * NB;
  static constexpr int kMeta = NB == 1 ? 3 : 2;      // metadata buffers (items ahead of the slowest group)
  // bytes from the 1024-aligned base
  // NB = 1: two items, each 2 k halves of [Q ; K], [128][64] bf16.  NB = 2: 2 k halves of [Q_0 ; K_0 ; K_1 ; Q_1]
  static constexpr uint32_t kOffQK = 0;
  static constexpr uint32_t kBlkQK = NB == 1 ? 2 * kTile : kTile;    // from one block's operand to the next
  static constexpr uint32_t kHalfQK = NB == 1 ? kTile : 2 * kTile;   // from one k half to the next
  static constexpr uint32_t kOffS = 4 * kTile;       // four units [128 v][32] fp32, after the split [128 v][32 hi | 32 lo] bf16
  static constexpr uint32_t kOffV = 8 * kTile;       // V, then V'_hi in its place, and V'_lo: dv halves of [nodes][64] (NB = 1: two items)
  // Sets of columns of X: blocks between their state product and their stores.  NB = 1, two sets, with [Q ; K] copied
  // to tensor memory instead: 79.3 / 133 us on 2048 items of 64 nodes, with three 75.2 / 128.5.
  static constexpr uint32_t kXBufs = NB == 1 ? 3 : 2;
  static constexpr uint32_t kVHalf = kNodes * 128;   // one dv half
  static constexpr uint32_t kVItem = 4 * kVHalf;     // hi, lo
  static constexpr uint32_t kOffRow = 12 * kTile;    // 64 bytes per tile row, private to its thread (warps 8..11)
  static constexpr uint32_t kOffOut = kOffRow + 8192;   // staging of the outputs, per warp (warps 12..15)
  static constexpr int kOutRows = NB == 1 ? 32 : 16;    // rows of 32 floats that an output warp stages at a time
  static constexpr uint32_t kOffGs = kOffOut + 4 * kOutRows * 128;    // float Gs[kNodes][kLd]: rows of G, by path slot
  static constexpr uint32_t kOffPath = kOffGs + kNodes * kLd * 4;          // kMeta x uint8[kNodes][16], path in slot order
  static constexpr uint32_t kOffDepth = kOffPath + kMeta * kNodes * 16;    // kMeta x int8[kNodes], -1 = no node
  static constexpr uint32_t kOffTab = kOffDepth + kMeta * kNodes;          // kMeta x {{alpha, beta}[kNodes], P[kNodes]}
  static constexpr uint32_t kOffItem = kOffTab + kMeta * kNodes * 12;      // kMeta x {nodes, first output element (2 words), -}
  static constexpr uint32_t kOffLink = kOffItem + kMeta * 16;              // {alpha, parent}[kNodes], metadata warp only
  static constexpr uint32_t kOffBar = kOffLink + kNodes * 8;
  static constexpr uint32_t kOffMisc = kOffBar + 8 * 48;
  static constexpr uint32_t kSmemBytes = kOffMisc + 32;
  static_assert(kOffBar % 8 == 0 && kSmemBytes <= 232448, "shared memory of one CTA");
};

// [2]: block g of the CTA (item * NB + row block) uses entry g & 1, in its phase g >> 1
enum Bar {
  QK_FULL = 0, QK_FREE = 2, GD = 4, SC_FREE = 6, COEF = 8,
  V_FULL = 10, V_FREE = 12,          // [2]: NB = 1 as above, NB = 2 entry 0 per item
  VP = 14, X_FREE = 17, ACC = 20, X_DONE = 23,   // [kXBufs]: set of columns of X, phase = its use
  S_FULL = 26, S_SPLIT = 30, S_FREE = 34,   // [4]: unit, phase = item
  META_FULL = 38, META_FREE = 41,    // [kMeta]
  E1_SYNC = 44,
  kNumBars = 45
};
static_assert(kNumBars <= 48, "barrier area");

// TMEM columns: X from 0 on (three or two sets of 128), then the scores, which become the coefficients (NB = 1: two
// sets of 64; NB = 2: 64 for block 0, 128 for block 1)

struct Params {
  TreeDev tree;
  int32_t n_items, B, H, T;
  int32_t Hk;  // q/k heads (grouped key heads); H when not grouped
  const float* alpha;
  const float* beta;
  int32_t* status;
  float* O;
  float* U;                  // null: corrections not wanted
  const int32_t* offsets;    // packed forest only: row offsets of the requests, rows per (layer, head) plane
  int32_t capacity;
  ItemDiv div;               // divisions by H, B, H / Hk as multiply-shift
  Str3 gate, out;            // strides of alpha / beta and of O / U (dense layouts)
  // The q, k, v maps are 4-D, (channel, node, head, layer*request) or (channel, head, node, ...)
  // whichever has ascending strides: bit 0 / 1 set = q,k / v take the node coordinate first.
  int32_t node_first;
};

// A pair of fp32 as bf16 hi (rounded to nearest, within bf16's range) and lo (the exact remainder, rounded to nearest)
__device__ __forceinline__ void split_pair(Pair x, uint32_t& hi, uint32_t& lo) {
  const float2 v = unpack(x);
  hi = pack_sat(v.x, v.y);
  const float2 r = unpack(fma2(pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), pack(-1.f, -1.f), x));
  lo = pack_rn(r.x, r.y);
}

// DMAX: compile-time bound on the tree depth (8 covers draft trees, 15 the rest), so that the
// per-row triangular solve is straight-line code whose loads all issue up front.
// PACKED = packed forest: request b owns rows offsets[b] .. offsets[b+1]-1 of every plane; loads take
// 64-row boxes at the request's offset.  Rows past the request's node count may hold anything: their
// V' is set to zero, their scores are never selected and their outputs never stored.
template <int NB, int DMAX, bool PACKED>
__global__ void __launch_bounds__(kThreads, 1)
verify_tc_delta_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmS,
                       const Params p) {
  using M = Map<NB>;
  constexpr int kNodes = M::kNodes;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw;
  const uint32_t sbase = smem_u32(sm);
  if (sbase & 1023u) {   // the swizzled tiles need this alignment; refuse rather than compute garbage
    if (threadIdx.x == 0 && p.status) atomicExch(p.status, (int)TV_ERR_CUDA);
    return;
  }
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + M::kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + M::kOffMisc + 4);
  auto bar = [&](int i) { return sbase + M::kOffBar + 8u * (uint32_t)i; };
  auto tab_of = [&](uint32_t buf) { return reinterpret_cast<float*>(sm + M::kOffTab) + buf * (3 * kNodes); };
  auto item_of = [&](uint32_t buf) { return reinterpret_cast<int32_t*>(sm + M::kOffItem) + buf * 4; };
  auto sc_col = [](int g) -> uint32_t { return M::kXBufs * 128u + (uint32_t)(g & 1) * 64u; };
  // set of X of block g, and the parity of that use
  auto x_set = [](uint32_t g) -> uint32_t { return NB == 1 ? g % 3u : g & 1u; };
  auto x_par = [](uint32_t g) -> uint32_t { return (NB == 1 ? g / 3u : g >> 1) & 1u; };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int T = p.T;
  const bool want_U = p.U != nullptr;
  const uint32_t n_it = (int)blockIdx.x < p.n_items
                            ? ((uint32_t)p.n_items - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u;

  if (warp == 0) {
    if (lane == 0) {
      abort_flag[0] = 0;
      abort_flag[1] = 0;
      prefetch_map(&tmQ);
      prefetch_map(&tmK);
      prefetch_map(&tmS);
      prefetch_map(&tmV);
    }
    for (int i = lane; i < kNumBars; i += 32) {   // arrivals of a phase: one thread, unless it is four warps
      const bool warps4 = (i >= COEF && i < V_FULL) || (i >= VP && i < ACC) || (i >= S_SPLIT && i < S_FREE) || i == E1_SYNC;
      const bool qk = i >= QK_FREE && i < GD, meta = i >= META_FREE && i < E1_SYNC;
      mbar_init(bar(i), qk ? 2 : meta ? 12 : warps4 ? 4 : 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // registers: 96 per thread at launch, moved to where the long rows are held
  if (warp < 4) {
    set_registers_down<kServiceRegs>();
    if (warp == 0 && lane == 0) {
      // ===================== TMA producer =====================
      grid_dependency_wait();   // inputs may come from the kernel in front (dependent launch)
      uint32_t n_qk = 0, n_v = 0, n_s = 0;   // loads issued: blocks, items, units
      // Box coordinates: q/k head, v head, outermost index (layer*request, or the layer of a packed
      // forest) and the first node row.
      struct Coord {
        int item, hq, h, z, y0;
      };
      auto coord_of = [&](uint32_t it) {
        Coord c;
        c.item = (int)(blockIdx.x + it * gridDim.x);
        const int lb = (int)fdiv((uint32_t)c.item, p.div.dH);
        c.h = c.item - lb * p.H;
        c.hq = (int)fdiv((uint32_t)c.h, p.div.dG);
        c.z = lb;
        c.y0 = 0;
        if constexpr (PACKED) {
          c.z = (int)fdiv((uint32_t)lb, p.div.dB);
          c.y0 = __ldg(p.offsets + (lb - c.z * p.B));
        }
        return c;
      };
      const bool nf_qk = p.node_first & 1, nf_v = p.node_first & 2;
      auto load_qk = [&](uint32_t it, const Coord& co) -> bool {
        for (int b = 0; b < NB; ++b) {
          const uint32_t g = it * NB + b, gb = g & 1;
          if (!mbar_wait(bar(QK_FREE + gb), ((g >> 1) & 1) ^ 1, abort_flag)) return false;
          mbar_expect_tx(bar(QK_FULL + gb), 4 * 8192);
#pragma unroll 1
          for (int i = 0; i < 4; ++i)   // k half i >> 1; Q rows, then K rows
            load_box(sbase + M::kOffQK + gb * M::kBlkQK + (uint32_t)(i >> 1) * M::kHalfQK + (uint32_t)((i & 1) ^ b) * 8192u,
                     (i & 1) ? &tmK : &tmQ, bar(QK_FULL + gb), nf_qk, 64 * (i >> 1), co.y0 + kBlk * b, co.hq, co.z);
          ++n_qk;
        }
        return true;
      };
      auto load_v = [&](uint32_t it, const Coord& co) -> bool {
        const uint32_t vb = NB == 1 ? it & 1 : 0, vph = NB == 1 ? it >> 1 : it;
        if (!mbar_wait(bar(V_FREE + vb), (vph & 1) ^ 1, abort_flag)) return false;
        mbar_expect_tx(bar(V_FULL + vb), 2 * M::kVHalf);
#pragma unroll 1
        for (int i = 0; i < 2 * NB; ++i)   // dv half i & 1, row block i >> 1
          load_box(sbase + M::kOffV + vb * M::kVItem + (uint32_t)(i & 1) * M::kVHalf + (uint32_t)(i >> 1) * 8192u, &tmV,
                   bar(V_FULL + vb), nf_v, 64 * (i & 1), co.y0 + kBlk * (i >> 1), co.h, co.z);
        ++n_v;
        return true;
      };
      auto load_s = [&](uint32_t it, const Coord& co) -> bool {
#pragma unroll 1
        for (int u = 0; u < kUnits; ++u) {
          if (!mbar_wait(bar(S_FREE + u), (it & 1) ^ 1, abort_flag)) return false;
          mbar_expect_tx(bar(S_FULL + u), kTile);
          tma_load_3d(sbase + M::kOffS + (uint32_t)u * kTile, &tmS, bar(S_FULL + u), 32 * u, 0, co.item);
          ++n_s;
        }
        return true;
      };
      for (uint32_t it = 0; it < n_it; ++it) {
        const Coord co = coord_of(it);
        if (!load_qk(it, co) || !load_s(it, co) || !load_v(it, co)) break;   // in the order in which they come free
      }
      if (*abort_flag) {
        // Leave no copy of ours in flight: wait (bounded) for the last load issued into each buffer.
        for (uint32_t g = n_qk > 2 ? n_qk - 2 : 0; g < n_qk; ++g) mbar_wait(bar(QK_FULL + (g & 1)), (g >> 1) & 1, abort_flag + 1);
        for (uint32_t i = n_v > 2 ? n_v - 2 : 0; i < n_v; ++i)
          mbar_wait(bar(V_FULL + (NB == 1 ? i & 1 : 0)), (NB == 1 ? i >> 1 : i) & 1, abort_flag + 1);
        for (uint32_t i = n_s > 4 ? n_s - 4 : 0; i < n_s; ++i)
          mbar_wait(bar(S_FULL + (i & 3)), (i >> 2) & 1, abort_flag + 1);
      }
    } else if (warp == 1 && lane == 0) {
      // ===================== MMAs: scores, readout =====================
      constexpr uint32_t kIdGram = idesc_bf16(64, false), kIdGram2 = idesc_bf16(128, false), kIdAV = idesc_bf16(128, true);
      const uint32_t n_g = n_it * NB;
      uint32_t ig = 0, ia = 0;   // next block's scores, next block's readout
      const uint64_t dQK = desc_kmajor(sbase + M::kOffQK);
      const uint64_t dV = desc_mnmajor(sbase + M::kOffV, M::kVHalf);
      long long t_idle = clock64();
      uint32_t spin = 0;
      while (ia < n_g) {
        bool progress = false;
        // X += [W ; A] V' of block ia
        if (mbar_test(bar(VP + x_set(ia)), x_par(ia)) && mbar_test(bar(COEF + (ia & 1)), (ia >> 1) & 1)) {
          tc_fence_after();
          const uint32_t b = NB == 1 ? 0u : ia & 1;
          const uint32_t acc = tmem + x_set(ia) * 128u, chi = tmem + sc_col((int)ia), clo = chi + 32u * (b + 1);
          const uint64_t dvi = dV + (NB == 1 ? ((ia & 1) * M::kVItem) >> 4 : 0u);
          const int n = item_of((ia / NB) % M::kMeta)[0];   // the block's last steps may hold no node
#pragma unroll 1
          for (uint32_t hb = 0; hb <= b; ++hb)   // 64 ancestors
#pragma unroll
            for (uint32_t s = 0; s < 4; ++s) {   // 16 ancestors per step
              if ((int)(64u * hb + 16u * s) >= n) break;
              const uint64_t hi = dvi + ((hb * 8192u + s * 2048u) >> 4), lo = hi + ((2 * M::kVHalf) >> 4);
              const uint32_t c = hb * 32u + s * 8u;
              mma_bf16_ts(acc, chi + c, hi, kIdAV, 1);
              mma_bf16_ts(acc, clo + c, hi, kIdAV, 1);
              mma_bf16_ts(acc, chi + c, lo, kIdAV, 1);
            }
          tc_commit(bar(ACC + x_set(ia)));
          tc_commit(bar(SC_FREE + (ia & 1)));
          if (NB == 1) tc_commit(bar(V_FREE + (ia & 1)));
          else if (b == 1) tc_commit(bar(V_FREE));
          ++ia;
          progress = true;
        }
        // Sc = [Q ; K] K^T of block ig
        if (ig < n_g && mbar_test(bar(QK_FULL + (ig & 1)), (ig >> 1) & 1) &&
            mbar_test(bar(SC_FREE + (ig & 1)), ((ig >> 1) & 1) ^ 1)) {
          tc_fence_after();
          const uint32_t b = NB == 1 ? 0u : ig & 1;
          const uint64_t dA = dQK + (((ig & 1) * M::kBlkQK) >> 4), dB = dQK + ((NB == 1 ? (ig & 1) * M::kBlkQK + 8192u : 8192u) >> 4);
#pragma unroll
          for (uint32_t i = 0; i < 8; ++i) {   // k half i >> 2, 32 bytes of k per step
            const uint32_t off = ((i >> 2) * M::kHalfQK + (i & 3u) * 32u) >> 4;
            mma_bf16_ss(tmem + sc_col((int)ig), dA + off, dB + off, b ? kIdGram2 : kIdGram, i);
          }
          tc_commit(bar(GD + (ig & 1)));
          if (NB == 1) {
            tc_commit(bar(QK_FREE + (ig & 1)));
          } else if (b == 1) {   // block 1's scores read both blocks' keys
            tc_commit(bar(QK_FREE));
            tc_commit(bar(QK_FREE + 1));
          }
          ++ig;
          progress = true;
        }
        if (progress) {
          t_idle = clock64();
          spin = 0;
        } else {
          __nanosleep(20);   // four working warps share this one's issue slots
          if ((++spin & 255u) == 0) {   // the same limit as every other wait of the kernel
            if (*abort_flag) break;
            if (clock64() - t_idle > kWaitLimitCycles) {
              *abort_flag = 1;
              break;
            }
          }
        }
      }
    } else if (warp == 3 && lane == 0) {
      // ===================== MMAs: state product =====================
      constexpr uint32_t kIdX = idesc_bf16(128, false);
      const uint64_t dQK = desc_kmajor(sbase + M::kOffQK), dS = desc_kmajor(sbase + M::kOffS);
      bool ok = true;
      for (uint32_t g = 0; ok && g < n_it * NB; ++g) {
        const uint32_t it = g / NB, gb = g & 1, xs = x_set(g), x = tmem + xs * 128u;
        if (!(ok = mbar_wait(bar(QK_FULL + gb), (g >> 1) & 1, abort_flag))) break;
        if (!(ok = mbar_wait(bar(X_FREE + xs), x_par(g) ^ 1, abort_flag))) break;   // what these columns held has been read out
#pragma unroll 1
        for (uint32_t u = 0; u < kUnits; ++u) {   // a quarter of k
          if (!(ok = mbar_wait(bar(S_SPLIT + u), it & 1, abort_flag))) break;
          tc_fence_after();
          const uint64_t dB = dS + ((u * kTile) >> 4);
          const uint64_t dA = dQK + ((gb * M::kBlkQK + (u >> 1) * M::kHalfQK + (u & 1) * 64u) >> 4);
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i)   // hi: k 0..15, 16..31 of the quarter; lo: the same
            mma_bf16_ss(x, dA + (((i & 1u) * 32u) >> 4), dB + ((i * 32u) >> 4), kIdX, u | i);
          if (NB == 1 || gb == 1) tc_commit(bar(S_FREE + u));
        }
        if (!ok) break;
        tc_commit(bar(X_DONE + xs));
        tc_commit(bar(QK_FREE + gb));
      }
    } else if (warp == 2) {
      // ===================== metadata =====================
      grid_dependency_wait();   // tree metadata and gates may come from the kernels in front
      // A lane has the nodes lane, lane + 32, ...; the next item's values are on their way while this
      // one's tables are written.
      constexpr int NN = 2 * NB;
      int n = 0, dep[NN], par[NN];
      float al[NN], be[NN];
      size_t o0 = 0;               // element offset of the item's first output row
      auto fetch = [&](uint32_t it) {
        const int item = (int)(blockIdx.x + it * gridDim.x);
        n = T;
        int tb = 0;
        int64_t g0, gstep = 1;     // first gate of the item, step between nodes
        if constexpr (PACKED) {
          const PackedItem pi = packed_item(p.offsets, p.B, p.H, p.Hk, item, p.div);
          n = pi.n;
          tb = pi.b;
          g0 = (int64_t)pi.plane_v * p.capacity + pi.row0;
          o0 = (size_t)g0 * 128;
        } else {
          const int lb = (int)fdiv((uint32_t)item, p.div.dH), h = item - lb * p.H;
          tb = p.tree.n_trees == 1 ? 0 : request_of(item, p.B, p.div);
          g0 = (int64_t)lb * p.gate.b + (int64_t)h * p.gate.h;
          gstep = p.gate.t;
          o0 = (size_t)((int64_t)lb * p.out.b + (int64_t)h * p.out.h);
        }
#pragma unroll
        for (int h = 0; h < NN; ++h) {
          const int nd = lane + 32 * h;
          dep[h] = -1;
          par[h] = -1;
          al[h] = 1.f;
          be[h] = 0.f;
          if (nd < n) {
            dep[h] = __ldg(p.tree.depth + (size_t)tb * T + nd);
            par[h] = __ldg(p.tree.parent + (size_t)tb * T + nd);
            al[h] = __ldg(p.alpha + g0 + nd * gstep);
            be[h] = __ldg(p.beta + g0 + nd * gstep);
          }
        }
      };
      float2* link = reinterpret_cast<float2*>(sm + M::kOffLink);
      if (n_it > 0) fetch(0);
      for (uint32_t it = 0; it < n_it; ++it) {
        const uint32_t buf = it % M::kMeta, use = it / M::kMeta;
        if (!mbar_wait_warp(bar(META_FREE + buf), (use & 1) ^ 1, abort_flag)) break;
        float* tab = tab_of(buf);
        uint8_t* paths = sm + M::kOffPath + (buf * kNodes) * 16;
        int8_t* depths = reinterpret_cast<int8_t*>(sm + M::kOffDepth) + buf * kNodes;
        int slot[NN], j[NN];
        float P[NN];
#pragma unroll
        for (int h = 0; h < NN; ++h) {
          const int nd = lane + 32 * h;
          reinterpret_cast<float2*>(tab)[nd] = make_float2(al[h], be[h]);
          link[nd] = make_float2(al[h], __int_as_float(par[h]));
          depths[nd] = (int8_t)dep[h];
          const uint32_t self = (uint32_t)nd * 0x01010101u;   // slots past the node's depth name the node itself
          *reinterpret_cast<uint4*>(paths + nd * 16) = make_uint4(self, self, self, self);
          slot[h] = dep[h];
          j[h] = nd;
          P[h] = 1.f;
        }
        if (lane == 0) {
          int32_t* im = item_of(buf);
          im[0] = n;
          im[1] = (int32_t)(o0 & 0xffffffffu);
          im[2] = (int32_t)(o0 >> 32);
        }
        __syncwarp();
        if (it + 1 < n_it) fetch(it + 1);
        // from every node up: the path in slot order, and P
#pragma unroll 1
        for (int e = 0; e <= DMAX; ++e) {
          bool more = false;
#pragma unroll
          for (int h = 0; h < NN; ++h) {
            if (slot[h] >= 0 && j[h] >= 0) {
              paths[(lane + 32 * h) * 16 + slot[h]] = (uint8_t)j[h];
              const float2 y = link[j[h]];
              P[h] *= y.x;
              j[h] = __float_as_int(y.y);
              --slot[h];
              more = more || slot[h] >= 0;
            }
          }
          if (!__any_sync(0xffffffffu, more)) break;
        }
        // V' holds P and meets every node of the item in a dense product, whose zero coefficients do not stop a NaN:
        // where a gate leaves P not finite, V' is zero instead (V' group) and the node's beta a NaN, which reaches
        // the rows of the node and of its descendants alone.
#pragma unroll
        for (int h = 0; h < NN; ++h) {
          tab[2 * kNodes + lane + 32 * h] = P[h];
          if (!isfinite(P[h])) tab[2 * (lane + 32 * h) + 1] = __int_as_float(0x7fffffff);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(META_FULL + buf));
      }
    }
  } else if (warp < 8) {
    // ===================== state split =====================
    set_registers_down<kSplitRegs>();
    const int row = (warp & 3) * 32 + lane;
    const uint32_t swz = (uint32_t)(row & 7);
    bool ok = true;
    for (uint32_t it = 0; ok && it < n_it; ++it) {
#pragma unroll 1
      for (int u = 0; u < kUnits; ++u) {
        if (!(ok = mbar_wait_warp(bar(S_FULL + u), it & 1, abort_flag))) break;
        // 32 fp32 of this row -> 32 bf16 hi | 32 bf16 lo in the same 128 bytes
        unsigned char* r = sm + M::kOffS + (uint32_t)u * kTile + (uint32_t)row * 128u;
        uint4 hi[4], lo[4];
#pragma unroll
        for (uint32_t c = 0; c < 4; ++c) {
          const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(r + (((2 * c) ^ swz) << 4));
          const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(r + (((2 * c + 1) ^ swz) << 4));
          split_pair(Pair{a.x}, hi[c].x, lo[c].x);
          split_pair(Pair{a.y}, hi[c].y, lo[c].y);
          split_pair(Pair{e.x}, hi[c].z, lo[c].z);
          split_pair(Pair{e.y}, hi[c].w, lo[c].w);
        }
#pragma unroll
        for (uint32_t c = 0; c < 4; ++c) {
          *reinterpret_cast<uint4*>(r + ((c ^ swz) << 4)) = hi[c];
          *reinterpret_cast<uint4*>(r + (((c + 4) ^ swz) << 4)) = lo[c];
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(S_SPLIT + u));
      }
    }
  } else if (warp < 12) {
    // ===================== path systems =====================
    set_registers_up<kPathRegs>();
    constexpr int NS = DMAX + 1;            // path slots in use
    const int quad = warp & 3, row = quad * 32 + lane;
    const int rn = row & 63;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    float* Gs = reinterpret_cast<float*>(sm + M::kOffGs);
    // 64 bytes of scratch per tile row, seen by its own thread only: values go in by column and come
    // out by path node, or the other way round (registers cannot be indexed).  Chunks of 16 bytes are
    // swizzled so that eight neighbouring rows cover all banks.
    unsigned char* srow = sm + M::kOffRow + row * 64;
    const uint32_t ssw = (uint32_t)(row >> 1) & 3u;
    auto word = [&](uint32_t j) -> uint32_t { return (((j >> 2) ^ ssw) << 4) + ((j & 3u) << 2); };   // byte of column j < 16
    bool ok = true;
    for (uint32_t it = 0; ok && it < n_it; ++it) {
      const uint32_t buf = it % M::kMeta;
      if (!(ok = mbar_wait_warp(bar(META_FULL + buf), (it / M::kMeta) & 1, abort_flag))) break;
      const float2* ab = reinterpret_cast<const float2*>(tab_of(buf));   // alpha, beta
      const int n = item_of(buf)[0];
#pragma unroll 1
      for (int b = 0; b < NB; ++b) {
        const uint32_t g = it * NB + b;
        const int nd = kBlk * b + rn;
        const int part = (row >> 6) ^ b;        // 0: O problem, 1: U problem
        const uint4 pw = *reinterpret_cast<const uint4*>(sm + M::kOffPath + (buf * kNodes + nd) * 16);
        const int depth = reinterpret_cast<const int8_t*>(sm + M::kOffDepth)[buf * kNodes + nd];   // -1: no node
        const bool rows_live = kBlk * b + (quad & 1) * 32 < n;     // warp-uniform: some row of the warp is a node
        const bool solves = rows_live && (part == 0 || want_U);    // warp-uniform: its rows carry problems
        // of every path slot: row of Gs, chunk of 16 score columns, place in the row's scratch
        int grow[NS], chunk[NS];
        uint32_t place[NS];
        float al[NS], bt[NS], vec[NS];
        {
          const uint32_t pword[4] = {pw.x, pw.y, pw.z, pw.w};
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            const int node = (int)((pword[s >> 2] >> ((s & 3) * 8)) & 127u);
            grow[s] = node * kLd;
            chunk[s] = node >> 4;
            place[s] = word((uint32_t)node & 15u);
            const float2 y = ab[node];
            al[s] = s <= depth ? y.x : 1.f;   // slots past the node count as no decay
            bt[s] = s <= depth ? y.y : 0.f;
            vec[s] = 0.f;
          }
        }
        // ---- scores on the path: q_i . k_{p_s} (incl. the node), k_i . k_{p_s} ----
        if (!(ok = mbar_wait_warp(bar(GD + (g & 1)), (g >> 1) & 1, abort_flag))) break;
        // every warp has finished the solve of the block before, which read Gs
        if (g > 0 && !(ok = mbar_wait_warp(bar(COEF + ((g - 1) & 1)), ((g - 1) >> 1) & 1, abort_flag))) break;
        tc_fence_after();
        const uint32_t col = tmem + lane_addr + sc_col((int)g);
        // ancestors have smaller numbers than the node: nothing to select past the warp's last node
        const int nch = 4 * b + (quad & 1) * 2 + 2;                // chunks of 16 columns
        if (rows_live) {
#pragma unroll 1
          for (int c = 0; c < nch; c += 2) {
            uint32_t r[32];
            tmem_ld32(col + 16u * c, r);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i)
                *reinterpret_cast<float4*>(srow + ((i ^ ssw) << 4)) =
                    make_float4(__uint_as_float(r[16 * e + 4 * i]), __uint_as_float(r[16 * e + 4 * i + 1]),
                                __uint_as_float(r[16 * e + 4 * i + 2]), __uint_as_float(r[16 * e + 4 * i + 3]));
#pragma unroll
              for (int s = 0; s < NS; ++s)
                if (chunk[s] == c + e) vec[s] = *reinterpret_cast<const float*>(srow + place[s]);
            }
          }
          // Decay from a path node down to this one: the product of alpha over the slots between, built up
          // from the node's own slot backwards.
          //   part 0: C_{i,p_s} = (P_i / P_{p_s}) q_i . k_{p_s}
          //   part 1: G_{i,p_s} = beta_i (P_i / P_{p_s}) k_i . k_{p_s}, a row of Gs for every row whose path
          //           leads through this node; its own system is x L = e_d
          const float be = part == 0 ? 1.f : ab[nd].y;
          float sfx = 1.f;
#pragma unroll
          for (int s = NS - 1; s >= 0; --s) {
            const float c = vec[s] * (be * sfx);
            sfx *= al[s];
            if (part == 1) Gs[nd * kLd + s] = c;
            vec[s] = part == 1 ? (s == depth ? 1.f : 0.f) : s <= depth ? c : 0.f;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(E1_SYNC));
        if (!(ok = mbar_wait_warp(bar(E1_SYNC), g & 1, abort_flag))) break;
        if (solves) {
          // w_s = c_s - sum_{t > s} w_t G_{p_t,p_s}; slots past the node's depth carry vec = 0
#pragma unroll
          for (int s = NS - 2; s >= 0; --s) {
            float acc = vec[s];
#pragma unroll
            for (int t = s + 1; t < NS; ++t) acc = fmaf(-vec[t], Gs[grow[t] + s], acc);
            if (s < depth) vec[s] = acc;
          }
          // ---- row of [W ; A] = (w or x) D_beta as bf16 hi and lo, into the columns of the scores ----
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            const float w = vec[s] * bt[s];
            const uint32_t h = pack_rn(w, 0.f);
            vec[s] = __uint_as_float(pack_rn(__uint_as_float(h << 16), w - __uint_as_float(h << 16)));   // hi | lo << 16, both exact roundings
          }
          const uint32_t lo_off = 32u * (b + 1);
          const int n_all = 4 * (b + 1);
#pragma unroll 1
          for (int c = 0; c < n_all; ++c) {
            uint32_t w[16];
            if (c < nch) {
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(srow + ((i ^ ssw) << 4)) = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
              for (int s = 0; s < NS; ++s)
                if (s <= depth && chunk[s] == c) *reinterpret_cast<uint32_t*>(srow + place[s]) = __float_as_uint(vec[s]);
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i) {
                const uint4 x = *reinterpret_cast<const uint4*>(srow + ((i ^ ssw) << 4));
                w[4 * i] = x.x; w[4 * i + 1] = x.y; w[4 * i + 2] = x.z; w[4 * i + 3] = x.w;
              }
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i) w[i] = 0u;
            }
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              hi[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
              lo[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
            }
            tmem_st8(col + 8u * c, hi);
            tmem_st8(col + lo_off + 8u * c, lo);
          }
          tmem_wait_st();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(COEF + (g & 1)));
      }
      if (ok && lane == 0) mbar_arrive(bar(META_FREE + buf));
    }
  } else if (warp >= 16) {
    // ===================== V', scaling of X =====================
    const int quad = warp & 3, row = quad * 32 + lane;   // TMEM lane
    const int rn = row & 63;                             // node of this tile row within its block
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t swz = (uint32_t)(row & 7);
    bool ok = true;
    for (uint32_t it = 0; ok && it < n_it; ++it) {
      const uint32_t buf = it % M::kMeta, vb = NB == 1 ? it & 1 : 0;
      if (!(ok = mbar_wait_warp(bar(META_FULL + buf), (it / M::kMeta) & 1, abort_flag))) break;
      if (!(ok = mbar_wait_warp(bar(V_FULL + vb), (NB == 1 ? it >> 1 : it) & 1, abort_flag))) break;
      const int n = item_of(buf)[0];
#pragma unroll 1
      for (int b = 0; b < NB; ++b) {
        const uint32_t g = it * NB + b;
        const int nd = kBlk * b + rn;
        const float P = tab_of(buf)[2 * kNodes + nd];
        const uint32_t xcol = tmem + lane_addr + x_set(g) * 128u;
        if (!(ok = mbar_wait_warp(bar(X_DONE + x_set(g)), x_par(g), abort_flag))) break;
        tc_fence_after();
        if (((quad >> 1) ^ b) == 0) {
          // O problem: the prefix term P_i q_i S_pre^T is where the accumulation starts
          if (kBlk * b + (quad & 1) * 32 < n) {
#pragma unroll 1
            for (int c = 0; c < 4; c += 2) {
              uint32_t x[64];
              tmem_ld32(xcol + 32u * c, x);
              tmem_ld32(xcol + 32u * c + 32u, x + 32);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 64; ++i) x[i] = __float_as_uint(P * __uint_as_float(x[i]));
              tmem_st32(xcol + 32u * c, x);
              tmem_st32(xcol + 32u * c + 32u, x + 32);
            }
          }
        } else {
          const bool alive = nd < n && isfinite(P);
          // rows are multiplied 16 at a time: past the last such group nothing reads them
          if (kBlk * b + (quad & 1) * 32 < n) {
            unsigned char* vrow = sm + M::kOffV + vb * M::kVItem + (uint32_t)nd * 128u;
            // 32 columns (half of dv half d): V is read before anything is stored, and the next columns
            // of X are on their way meanwhile
            auto part_of = [&](uint32_t (&x)[32], uint32_t (&next)[32], int d, uint32_t half, bool more) {
              unsigned char* r = vrow + (uint32_t)d * M::kVHalf;
              const uint32_t col = xcol + 64u * d + 32u * half;
              uint4 v[4];
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i)
                v[i] = *reinterpret_cast<const uint4*>(r + (((half * 4 + i) ^ swz) << 4));
              tmem_wait_ld(x);
              if (more) tmem_ld32(col + 32u, next);
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i) {
                const uint32_t vw[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
                uint32_t hi[4], lo[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  split_pair(fma2(pack(__uint_as_float(x[8 * i + 2 * e]), __uint_as_float(x[8 * i + 2 * e + 1])), pack(-P, -P),
                                  pack(__uint_as_float(vw[e] << 16), __uint_as_float(vw[e] & 0xffff0000u))),
                             hi[e], lo[e]);
                const uint32_t off = ((half * 4 + i) ^ swz) << 4;
                *reinterpret_cast<uint4*>(r + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(r + 2 * M::kVHalf + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
              }
#pragma unroll
              for (int i = 0; i < 32; ++i) x[i] = 0u;   // U problem: the accumulation starts from nothing
              tmem_st32(col, x);
            };
            uint32_t xa[32], xb[32];
            tmem_ld32(xcol, xa);
#pragma unroll 1   // the roles of a CTA share one instruction cache
            for (int d = 0; d < 2; ++d) {
              part_of(xa, xb, d, 0, true);
              part_of(xb, xa, d, 1, d == 0);
              tmem_wait_ld(xa);   // no load in flight from one pass to the next
            }
            if (!alive) {   // rows past the request may hold anything: 0 x that need not be 0 (nor 0 x P that is not finite)
              const uint4 z = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
              for (uint32_t i = 0; i < 8; ++i)
#pragma unroll
                for (uint32_t part = 0; part < 4; ++part)
                  *reinterpret_cast<uint4*>(vrow + part * M::kVHalf + ((i ^ swz) << 4)) = z;
            }
            __syncwarp();
          }
          fence_async_smem();
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(VP + x_set(g)));
      }
      if (!ok) break;
      if (lane == 0) mbar_arrive(bar(META_FREE + buf));
    }
  } else {
    // ===================== outputs =====================
    set_registers_up<kOutRegs>();
    const int quad = warp & 3;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    // 32 rows x 32 columns at a time, all or half of the rows through the warp's staging area: a store then
    // covers whole 128-byte lines (eight lanes per row) where a lane with a row of its own touches 32 lines.
    // In: lane = row, chunk i at i ^ (row & 7); out: rows (lane >> 3) + 4 i, chunk lane & 7.
    constexpr int kRows = M::kOutRows;
    const uint32_t stage = sbase + M::kOffOut + (uint32_t)(quad * kRows * 128);
    const uint32_t in0 = stage + (uint32_t)(lane % kRows) * 128u + ((uint32_t)(lane & 7) << 4);
    const uint32_t out0 = stage + (uint32_t)(lane >> 3) * 128u + (((uint32_t)lane & 7u) ^ ((uint32_t)lane >> 3)) * 16u;
    const uint32_t out1 = (out0 ^ 64u) + 512u;   // rows 4 further have the other half of the swizzle
    const int64_t step4 = 4 * (PACKED ? (int64_t)128 : p.out.t);
    grid_dependency_wait();   // O and U may still be read by a kernel in front
    // the commit kernel behind this one may be scheduled as SMs drain (it orders itself)
    if (warp == 12 && lane == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool ok = true;
    for (uint32_t it = 0; ok && it < n_it; ++it) {
      const uint32_t buf = it % M::kMeta;
      if (!(ok = mbar_wait_warp(bar(META_FULL + buf), (it / M::kMeta) & 1, abort_flag))) break;
      const int32_t* im = item_of(buf);
      const int n = im[0];
      const size_t o0 = (size_t)(uint32_t)im[1] | (size_t)(uint32_t)im[2] << 32;
#pragma unroll 1
      for (int b = 0; b < NB; ++b) {
        const uint32_t g = it * NB + b;
        const int part = (quad >> 1) ^ b;             // 0: O rows, 1: U rows
        const int nd0 = kBlk * b + (quad & 1) * 32;   // first node of this warp
        const uint32_t xcol = tmem + lane_addr + x_set(g) * 128u;
        if (!(ok = mbar_wait_warp(bar(ACC + x_set(g)), x_par(g), abort_flag))) break;
        tc_fence_after();
        const bool stores = nd0 < n && (part == 0 || want_U);   // warp-uniform
        const int rows = n - nd0 - (lane >> 3);                 // of this lane's rows, those below this are nodes
        float* o[8];                                            // rows 4 j of this lane
        o[0] = (part == 0 ? p.O : p.U) + o0 + (int64_t)(nd0 + (lane >> 3)) * (step4 >> 2) + 4 * (lane & 7);
#pragma unroll
        for (int j = 1; j < 8; ++j) o[j] = o[j - 1] + step4;
        auto put = [&](const uint32_t (&x)[32], int c) {
#pragma unroll
          for (int h = 0; h < 32 / kRows; ++h) {
            __syncwarp();
            if (lane / kRows == h) {
#pragma unroll
              for (uint32_t i = 0; i < 8; ++i)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(in0 ^ (i << 4)), "r"(x[4 * i]),
                             "r"(x[4 * i + 1]), "r"(x[4 * i + 2]), "r"(x[4 * i + 3]) : "memory");
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < kRows / 16; ++q) {
              uint4 o4[4];
#pragma unroll
              for (int i = 0; i < 4; ++i)
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(o4[i].x), "=r"(o4[i].y), "=r"(o4[i].z), "=r"(o4[i].w)
                             : "r"(((i & 1) ? out1 : out0) + (uint32_t)(q * 2 + (i >> 1)) * 1024u) : "memory");
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (16 * (h + q) + 4 * i < rows)   // not read here again; cached in L1, rounds of 512 x 64 / 128: 36.3 / 55.3 against 35.8 / 54.3 us
                  asm volatile("st.global.L1::no_allocate.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(o[4 * (h + q) + i] + 32 * c),
                               "r"(o4[i].x), "r"(o4[i].y), "r"(o4[i].z), "r"(o4[i].w) : "memory");
            }
          }
        };
        uint32_t xa[32], xb[32];   // the next columns are read under the stores of these
        auto release = [&]() {   // all of this warp's rows are in registers
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(X_FREE + x_set(g)));
        };
        if (!stores) {
          release();
          continue;
        }
        tmem_ld32(xcol, xa);
        tmem_wait_ld(xa);
#pragma unroll 1   // the roles of a CTA share one instruction cache
        for (int d = 0; d < 2; ++d) {
          tmem_ld32(xcol + 64u * d + 32u, xb);
          put(xa, 0);
          tmem_wait_ld(xb);
          if (d == 0) tmem_ld32(xcol + 64u, xa);
          else release();
          put(xb, 1);
          tmem_wait_ld(xa);   // no load in flight from one pass to the next
#pragma unroll
          for (int j = 0; j < 8; ++j) o[j] += 64;
        }
      }
      if (ok && lane == 0) mbar_arrive(bar(META_FREE + buf));
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
  if (tid == 0 && *abort_flag && p.status) atomicExch(p.status, (int)TV_ERR_DEVICE_TIMEOUT);
}

template <int NB>
inline bool supports(const VerifyArgs& a) {
  return a.bf16 && a.dk == 128 && a.dv == 128 && a.rule == TV_GATED_DELTA && a.T > kBlk * (NB - 1) && a.T <= kBlk * NB &&
         a.tree.max_depth_all < kSlots;
}

template <int NB>
inline int launch(const VerifyArgs& a, int32_t* status, cudaStream_t stream) {
  if (!supports<NB>(a)) return TV_ERR_UNSUPPORTED;
  const bool packed = a.tree.offsets != nullptr;
  const uint64_t items = (uint64_t)a.L * a.B * a.H;
  // 4-D views: dense / strided layouts from the resolved strides, packed forests as planes
  NodeView vq, vv;
  if (!packed) {
    const uint64_t lb = (uint64_t)a.L * a.B;
    vq = NodeView{128, (uint64_t)a.T, (uint64_t)a.Hk, lb, a.lay.qk.b, a.lay.qk.h, a.lay.qk.t};
    vv = NodeView{128, (uint64_t)a.T, (uint64_t)a.H, lb, a.lay.v.b, a.lay.v.h, a.lay.v.t};
  } else {
    const int64_t cap = a.tree.capacity;
    vq = NodeView{128, (uint64_t)cap, (uint64_t)a.Hk, (uint64_t)a.L, (int64_t)a.Hk * cap * 128, cap * 128, 128};
    vv = NodeView{128, (uint64_t)cap, (uint64_t)a.H, (uint64_t)a.L, (int64_t)a.H * cap * 128, cap * 128, 128};
  }
  // q, k, v in boxes of 64 rows x 64 columns (rows past the tensor read as zero), S_pre in quarters of k
  const MapSet* ms = cached_maps(MapKey{{a.q, a.k, a.v, a.S_pre}, {vq, vv}, items, a.T, 9}, [&](CUtensorMap* m) {
    return make_map4(&m[0], a.q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, vq, 64, 64) &&
           make_map4(&m[1], a.k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, vq, 64, 64) &&
           make_map4(&m[2], a.v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, vv, 64, 64) &&
           make_map(&m[3], a.S_pre, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, items, 128, 128, 32, 128);
  });
  if (!ms) return TV_ERR_CUDA;
  constexpr uint32_t smem = Map<NB>::kSmemBytes;
  static thread_local int configured_dev = -1;
  int dev = 0;
  TV_CUDA_TRY(cudaGetDevice(&dev));
  if (configured_dev != dev) {
    constexpr int shares = kServiceRegs + kSplitRegs + kPathRegs + kOutRegs;
    int st = allow_kernel(verify_tc_delta_kernel<NB, 8, false>, smem, shares, 4);
    if (st == TV_OK) st = allow_kernel(verify_tc_delta_kernel<NB, 15, false>, smem, shares, 4);
    if (st == TV_OK) st = allow_kernel(verify_tc_delta_kernel<NB, 8, true>, smem, shares, 4);
    if (st == TV_OK) st = allow_kernel(verify_tc_delta_kernel<NB, 15, true>, smem, shares, 4);
    if (st != TV_OK) return st;
    configured_dev = dev;
  }
  const int sm_count = tv_sm_count();
  if (sm_count <= 0) return TV_ERR_CUDA;
  Params p;
  p.tree = a.tree;
  p.n_items = (int32_t)items;
  p.B = a.B; p.H = a.H; p.T = a.T; p.Hk = a.Hk;
  p.alpha = a.alpha;
  p.beta = a.beta;
  p.status = status;
  p.O = a.O;
  p.U = a.U;
  p.offsets = a.tree.offsets;
  p.capacity = a.tree.capacity;
  p.div = make_item_div(a.B, a.H, a.Hk);
  p.gate = a.lay.gate;
  p.out = a.lay.out;
  p.node_first = (node_first_of(vq) ? 1 : 0) | (node_first_of(vv) ? 2 : 0);
  // One CTA per SM, or as many as give every one the same number of items: they share the memory system with fewer
  // others, and the commit behind finds SMs free.  With two items a CTA always, with three or four where that
  // leaves out few SMs, never with more (us, equal shares / all SMs):
  //     items, 64 nodes     160          200          260          300          400          512          600          800
  //     back to back        13.2 / 13.1  13.3 / 13.7  13.7 / 13.9  17.9 / 16.8  18.7 / 18.7  23.7 / 23.5  28.2 / 26.4  33.6 / 33.0
  //     in rounds           19.8 / 20.6  20.7 / 21.3  21.9 / 22.1  26.5 / 26.7  29.8 / 29.9  36.0 / 36.4  42.0 / 41.5  52.9 / 52.1
  //     items, 128 nodes
  //     back to back        23.2 / 22.5  23.2 / 23.1  23.7 / 23.9  32.5 / 30.8  32.3 / 32.4  41.2 / 41.2  49.9 / 47.8  59.0 / 58.5
  //     in rounds           30.0 / 30.6  30.7 / 31.5  31.9 / 32.6  40.5 / 41.1  44.4 / 44.8  54.3 / 54.8  64.9 / 65.2  83.1 / 82.5
  int grid = (int)(items < (uint64_t)sm_count ? items : (uint64_t)sm_count);
  const int each = (int)((items + sm_count - 1) / sm_count), even = (int)((items + each - 1) / each);
  if (each == 2 || (each <= 4 && 20 * even >= 17 * sm_count)) grid = even;
  const bool shallow = a.tree.max_depth_all <= 8;
  auto go = [&](auto kernel) {
    return launch_dependent(kernel, grid, kThreads, smem, stream, ms->map[0], ms->map[1], ms->map[2], ms->map[3], p);
  };
  if (packed)
    TV_CUDA_TRY(shallow ? go(verify_tc_delta_kernel<NB, 8, true>) : go(verify_tc_delta_kernel<NB, 15, true>));
  else
    TV_CUDA_TRY(shallow ? go(verify_tc_delta_kernel<NB, 8, false>) : go(verify_tc_delta_kernel<NB, 15, false>));
  TV_CUDA_TRY(cudaGetLastError());
  return TV_OK;
}

}  // namespace tvdelta
