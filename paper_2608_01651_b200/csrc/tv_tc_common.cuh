// Device and host helpers shared by the kernels: mbarrier, TMA, tcgen05 / TMEM wrappers (inline
// PTX for sm_100a), shared-memory matrix descriptors, tensor-map construction, division by launch
// constants and dependent launches.  The tensor-core verify kernels use all of it; the Stage 1
// kernel the mbarrier / TMA part; the metadata, SIMT and commit kernels the dependent launch.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "tv_internal.h"
#include "tv_map_cache.h"

namespace tvtc {

constexpr uint32_t kTile = 16384;  // one 128-row x 128-byte operand tile

// instruction descriptors: fp32 accumulate, M = 128
constexpr uint32_t idesc_bf16(uint32_t n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | (8u << 24) | (b_mn_major ? (1u << 16) : 0u);
}

constexpr long long kWaitLimitCycles = 1ll << 31;  // ~1 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// ---- mbarrier ---------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Non-blocking look at a barrier (try_wait may park the thread for a while when the phase is
// not complete; a loop that polls several barriers must not be parked at one of them).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false when the limit ran out or another role gave up.  Kept short (32-bit
// clock, one exit for both reasons): a kernel has dozens of these, all inlined, and their code
// competes with the working loops for the instruction cache.  The clock is first read after
// 1024 failed tries and then every 1024; `limit` is cut to 2^31 cycles.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          long long limit = kWaitLimitCycles) {
  const uint32_t limit32 = limit > (long long)0x7fffffff ? 0x7fffffffu : (uint32_t)limit;
  uint32_t spin = 0, t0 = 0;
  while (!mbar_try(bar, parity)) {
    if ((++spin & 1023u) == 0) {
      const uint32_t now = (uint32_t)clock();
      if (spin == 1024u) {
        t0 = now;
      } else if (*abort_flag || now - t0 > limit32) {
        *abort_flag = 1;
        return false;
      }
    }
  }
  return true;
}

// Same for a whole warp: every lane gets the same answer, so that the warp never
// splits around the warp-collective tcgen05 instructions that follow.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               long long limit = kWaitLimitCycles) {
  const bool ok = mbar_wait(bar, parity, abort_flag, limit);
  return __all_sync(0xffffffffu, ok);
}

// ---- TMA --------------------------------------------------------------------
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// Brings a tensor map near before its first use: fetched by the copy itself, it is on that copy's path.
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
// Untiled bulk copy global -> shared (16-byte aligned on both sides, a multiple of 16 bytes),
// completing on `bar` like a TMA box.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// The calling thread's earlier cp.async copies arrive on `bar` when they have landed (the arrival
// is one of the barrier's expected count).
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
      ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// A box of a 4-D map (channel, node | head, head | node, outermost): the two middle coordinates
// are ordered by stride when the map is built (make_map4), `node_first` says which way.
__device__ __forceinline__ void load_box(uint32_t dst, const CUtensorMap* m, uint32_t bar, bool node_first, int x,
                                         int y, int h, int z) {
  if (node_first) tma_load_4d(dst, m, bar, x, y, h, z);
  else tma_load_4d(dst, m, bar, x, h, y, z);
}
__device__ __forceinline__ void store_box(const CUtensorMap* m, uint32_t src, bool node_first, int x, int y, int h,
                                          int z) {
  if (node_first) tma_store_4d(m, src, x, y, h, z);
  else tma_store_4d(m, src, x, h, y, z);
}

__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ---- tcgen05 ----------------------------------------------------------------
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_bf16_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// the same with A in tensor memory
__device__ __forceinline__ void mma_bf16_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),
        "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
        "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
        "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The same for one load's registers, by name: nothing that uses or copies them can stand in front of the wait,
// also where the load was issued in an earlier pass of a loop.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :: "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Two fp32 in one register pair: one instruction for both, rounded as two scalar ones.
struct Pair {
  uint64_t v;
};
__device__ __forceinline__ Pair pack(float a, float b) {
  Pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack(Pair a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
  Pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b) {
  Pair r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ Pair add2(Pair a, Pair b) {
  Pair r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

// Two fp32 -> one word of two bf16, rounded to nearest even (first argument in the low half).
__device__ __forceinline__ uint32_t pack_rn(float lo_elem, float hi_elem) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi_elem), "f"(lo_elem));
  return r;
}
// The same, finite values never rounded to infinity: what is left over then stays for a second piece.
__device__ __forceinline__ uint32_t pack_sat(float lo_elem, float hi_elem) {
  uint32_t r;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi_elem), "f"(lo_elem));
  return r;
}

// Shared-memory matrix descriptors, 128-byte swizzle, 1024-byte swizzle atoms.
// K-major: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
// MN-major (V as the B operand, dv contiguous): 64-column blocks `lbo` bytes
// apart, 8-row k groups 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}


// ---------------------------------------------------------------------------
// Host side: tensor maps.
// ---------------------------------------------------------------------------
inline PFN_cuTensorMapEncodeTiled get_encode() {
  static PFN_cuTensorMapEncodeTiled fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) ==
            cudaSuccess && qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(ptr);
  }
  return fn;
}

// [items][rows][cols] tensor, box {box_cols, box_rows, 1}, 128-byte swizzle, zero fill.
inline bool make_map(CUtensorMap* map, const void* base, CUtensorMapDataType dt, int esize, uint64_t items,
              uint64_t rows, uint64_t cols, uint32_t box_cols, uint32_t box_rows = 128) {
  PFN_cuTensorMapEncodeTiled enc = get_encode();
  if (!enc) return false;
  const cuuint64_t gdim[3] = {cols, rows, items};
  const cuuint64_t gstr[2] = {cols * esize, rows * cols * esize};
  const cuuint32_t box[3] = {box_cols, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, dt, 3, const_cast<void*>(base), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


// [rows][cols] tensor, box {box_cols, box_rows} landing as dense rows (no swizzle), zero fill.
inline bool make_map2_plain(CUtensorMap* map, const void* base, CUtensorMapDataType dt, int esize, uint64_t rows,
                            uint64_t cols, uint32_t box_cols, uint32_t box_rows) {
  PFN_cuTensorMapEncodeTiled enc = get_encode();
  if (!enc) return false;
  const cuuint64_t gdim[2] = {cols, rows};
  const cuuint64_t gstr[1] = {cols * esize};
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(map, dt, 2, const_cast<void*>(base), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Box {box_cols, box_rows nodes, 1 head, 1}; 128-byte swizzle, zero fill past the extents.
inline bool make_map4(CUtensorMap* map, const void* base, CUtensorMapDataType dt, int esize, const NodeView& v,
                      uint32_t box_cols, uint32_t box_rows) {
  PFN_cuTensorMapEncodeTiled enc = get_encode();
  if (!enc) return false;
  const bool nf = node_first_of(v);
  const uint64_t e1 = nf ? v.T : v.Hx, e2 = nf ? v.Hx : v.T;
  uint64_t s1 = (uint64_t)(nf ? v.st : v.sh) * esize, s2 = (uint64_t)(nf ? v.sh : v.st) * esize,
           s3 = (uint64_t)v.sb * esize;
  // a dimension of extent 1 never advances: give it a stride that keeps the sequence ascending
  if (e2 == 1) s2 = s1 * e1;
  if (v.Z == 1) s3 = s2 * e2;
  const cuuint64_t gdim[4] = {v.d, e1, e2, v.Z};
  const cuuint64_t gstr[3] = {s1, s2, s3};
  const cuuint32_t box[4] = {box_cols, nf ? box_rows : 1u, nf ? 1u : box_rows, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(map, dt, 4, const_cast<void*>(base), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// (layer, request, head) of a work item and, for a packed forest, where its rows live: request b
// owns rows offsets[b] .. offsets[b+1]-1 of every (layer, head) plane.
// Division by a launch constant: quotient = (mulhi(n, mul) + n) >> sh for every n < 2^31
// (round-up method; sh = ceil(log2 d)).  The persistent kernels turn item numbers into
// (layer, request, head) in several roles; the generic 32-bit division is some twenty
// instructions at every one of those places.
struct FastDiv {
  uint32_t d, mul, sh;
};
inline FastDiv make_fastdiv(uint32_t d) {
  FastDiv f;
  f.d = d;
  f.sh = 0;
  while ((1ull << f.sh) < d) ++f.sh;
  f.mul = (uint32_t)((((1ull << f.sh) - d) << 32) / d + 1);
  return f;
}
__device__ __forceinline__ uint32_t fdiv(uint32_t n, const FastDiv& f) { return (__umulhi(n, f.mul) + n) >> f.sh; }

struct PackedItem {
  int b, plane_v, plane_qk, row0, n;
};
// Divisions by H, B and the q/k group size H / Hk as multiply-shift.
struct ItemDiv {
  FastDiv dH, dB, dG;
};
inline ItemDiv make_item_div(int B, int H, int Hk) {
  ItemDiv d;
  d.dH = make_fastdiv((uint32_t)H);
  d.dB = make_fastdiv((uint32_t)B);
  d.dG = make_fastdiv((uint32_t)(H / Hk));
  return d;
}
__device__ __forceinline__ PackedItem packed_item(const int32_t* offsets, int B, int H, int Hk, int item,
                                                  const ItemDiv& d) {
  PackedItem r;
  const int lb = (int)fdiv((uint32_t)item, d.dH), h = item - lb * H;
  const int l = (int)fdiv((uint32_t)lb, d.dB);
  r.b = lb - l * B;
  r.plane_v = l * H + h;
  r.plane_qk = l * Hk + (int)fdiv((uint32_t)h, d.dG);
  r.row0 = offsets[r.b];
  r.n = offsets[r.b + 1] - r.row0;
  return r;
}
// dense layout: the tree of the request that item `item` belongs to
__device__ __forceinline__ int request_of(int item, int B, const ItemDiv& d) {
  const int lb = (int)fdiv((uint32_t)item, d.dH);
  return lb - (int)fdiv((uint32_t)lb, d.dB) * B;
}

// Registers a thread of a group of four warps, from here on (all four warps together).
template <int N>
__device__ __forceinline__ void set_registers_down() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void set_registers_up() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
// Shared memory and registers of a kernel, settled before its first launch on a device.  An increase waits, without
// a limit, for registers that other groups give up, out of those the block was launched with: `shares` (of all
// groups, those that keep what they have left out) must not exceed what the compiler gave that many groups.
template <class Kernel>
inline int allow_kernel(Kernel kernel, uint32_t smem, int shares, int groups) {
  cudaFuncAttributes at;
  TV_CUDA_TRY(cudaFuncGetAttributes(&at, kernel));
  if (shares > groups * at.numRegs) {
    tv_set_cuda_error(cudaErrorLaunchOutOfResources);
    return TV_ERR_CUDA;
  }
  TV_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return TV_OK;
}

// Programmatic dependent launch: the kernel may start while the kernel in front of it on the
// stream is still running, provided that kernel released its dependents early; whatever reads
// that kernel's output first passes grid_dependency_wait().
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... KArgs, class... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), int grid, int block, size_t smem,
                                    cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

}  // namespace tvtc
