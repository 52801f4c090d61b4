// Device-side helpers shared by the attention kernels: PTX wrappers (mbarrier, bulk and
// tensor-map asynchronous copies, ldmatrix / mma), bf16 conversion, and the per-warp tile ring
// through which a warp streams K/V page tiles from the pool.
#pragma once

#include "qc_internal.h"

#include <math.h>

#include <utility>

namespace qc {
namespace {

constexpr int kWarps = kAttendWarps;
constexpr int kThreads = kWarps * 32;
constexpr uint32_t kSpinLimit = 1u << 22; // bounded mbarrier wait

// values of the device error word (QC_ERR_* of the public header)
constexpr int kErrTimeout = 6;
constexpr int kErrBadPage = 7;
constexpr int kErrPlan = 8;   // a work range did not fit the limits the host planned it for
constexpr uint32_t kDebugSpinLimit = 1u << 12;   // wait limit under the test hook that drops a tile copy

// ------------------------------------------------------------------------------------------
// PTX helpers
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// 1-D bulk copy global -> this CTA's shared memory, completion counted on an mbarrier.
// Source, destination and size are multiples of 16 bytes by construction (whole page tiles).
// K/V tiles are read once per step: they are fetched with the evict-first L2 policy, so that the
// stream of tiles does not push the page tables, the queries and the partial rows out of the L2.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst_smem, const void* src, uint32_t bytes, uint64_t* bar,
                                         uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          dst_smem),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
// 2-D tensor-map copy global -> this CTA's shared memory (the map applies the 128-byte
// swizzle).  x is a multiple of 8 elements (16 bytes) by construction: 0 or 64.
__device__ __forceinline__ void tensor_g2s_2d(uint32_t dst_smem, const void* tmap, int32_t x, int32_t y,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst_smem),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// 3-D, with an L2 cache policy
__device__ __forceinline__ void tensor_g2s_3d(uint32_t dst_smem, const void* tmap, int32_t x, int32_t y, int32_t z,
                                              uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, "
      "%3, %4}], [%5], %6;" ::"r"(dst_smem),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tensor_g2s_3d(uint32_t dst_smem, const void* tmap, int32_t x, int32_t y, int32_t z,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(dst_smem),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// Asynchronous global -> shared copies of 4 or 16 bytes (no registers held while in flight);
// cp_async_wait_all() waits for the calling thread's own copies.
__device__ __forceinline__ void cp_async_4(void* dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_16(void* dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch: the kernels of a decode step are launched back to back with
// the programmatic-serialization attribute.  Each one does the set-up that may run early, waits
// for its predecessor to have completed (and its writes to be visible), and only then lets its
// successor start getting scheduled.
// Every kernel of the chain executes its wait BEFORE it lets its successor start, so when a kernel
// starts running, the kernel before its predecessor -- and by induction everything earlier in
// the stream -- has completed: what a kernel does ahead of its own wait may read anything that
// was written two or more launches back (the attention kernels plan their first work items there,
// from the launch plan, the step descriptors and the page tables; a step's first attention launch,
// right behind the kernel that writes those, waits first).
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with the programmatic-serialization attribute (plain stream order if the predecessor
// in the stream is not a kernel).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// 8x8 transpose of 16-bit elements held one row-pair per lane (row lane/4, columns 2*(lane%4)..)
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
// D(16x8, fp32) += A(16x16, bf16, row) * B(16x8, bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// Ask the L2 for a line.  Also of what an earlier kernel may still be writing: the L2 is where its writes and the reads
// after the wait for it meet.
__device__ __forceinline__ void l2_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// two fp32 -> packed bf16x2 (round to nearest even); `lo` lands in the low half
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ uint32_t pack_bf16x2_rz(float lo, float hi) {   // the same, rounded towards zero
  uint32_t d;
  asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

__device__ __forceinline__ void bf16x8_to_f32(const uint4& r, float* f) {
  f[0] = __uint_as_float(r.x << 16);
  f[1] = __uint_as_float(r.x & 0xffff0000u);
  f[2] = __uint_as_float(r.y << 16);
  f[3] = __uint_as_float(r.y & 0xffff0000u);
  f[4] = __uint_as_float(r.z << 16);
  f[5] = __uint_as_float(r.z & 0xffff0000u);
  f[6] = __uint_as_float(r.w << 16);
  f[7] = __uint_as_float(r.w & 0xffff0000u);
}

__device__ __forceinline__ uint16_t f32_to_bf16_rne(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7fffffffu) > 0x7f800000u) return static_cast<uint16_t>((u >> 16) | 0x40);   // NaN
  u += 0x7fffu + ((u >> 16) & 1u);
  return static_cast<uint16_t>(u >> 16);
}

// Record an error: the device word (largest code wins) and its mirror in mapped host memory.
__device__ __forceinline__ void report_error(int32_t* err, int32_t* err_host, int code) {
  atomicMax(err, code);
  if (err_host != nullptr) {
    *reinterpret_cast<volatile int32_t*>(err_host) = code;
    __threadfence_system();
  }
}

__device__ __forceinline__ size_t table_row(const Params& P, int layer, int stream, int seq_id) {
  return ((static_cast<size_t>(layer) * 4 + stream) * P.max_seqs + seq_id) * P.max_pages;
}

// 2^x, single MUFU instruction (2^-inf = 0; results below 2^-126 are 0)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Two fp32 operations in one instruction: the pairs are adjacent elements.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ float2 bf16x2_to_f32(uint32_t r) { return make_float2(__uint_as_float(r << 16), __uint_as_float(r & 0xffff0000u)); }
__device__ __forceinline__ void bf16x8_to_f32x2(const uint4& r, float2* f) {
  f[0] = bf16x2_to_f32(r.x), f[1] = bf16x2_to_f32(r.y), f[2] = bf16x2_to_f32(r.z), f[3] = bf16x2_to_f32(r.w);
}

// ------------------------------------------------------------------------------------------
// per-warp tile ring
// ------------------------------------------------------------------------------------------
//
// A warp owns RING tile slots in shared memory and one mbarrier per slot.  Lane 0 issues the
// copies of the K tile and the V tiles of each page of the warp's current item (and of the
// next one, so the ring never drains at an item boundary; an item that takes its scores from
// the logit cache has no K tiles); all lanes wait on a slot's
// barrier before reading it.  Every wait is bounded: when it runs out the worker records the
// error, stops fetching, lets the copies in flight land (again bounded) and leaves.

// Item descriptor and page ids of one item, as the ring needs them.
struct ItemPages {
  Item item;
  int32_t kv_head;     // item.head / group
  int32_t pad[3];
  uint4 new_k[16];     // folded append: the new token's k row of the item's K layer and the v row of its
  uint4 new_v[16];     // first consumer that takes the new token (fetched with the queries)
  int32_t pages[1 + kMaxCons][kMaxChunkPages];   // [0]: K pages, [1 + x]: V pages of consumer x
};

struct WorkerState {
  int n_my;            // items this worker owns
  int cons_k;          // item being consumed
  int iss_k;           // item being fetched (cons_k or cons_k + 1)
  int iss_pages;       // pages of it not yet requested (0: it has not been looked at, or is done)
  int iss_which, iss_first, iss_last;   // stream of the next tile (0: K, 1 + x: V of consumer x), of a page's first and last tile
  uint32_t iss_addr;   // where the next tile's page id is (shared memory)
  int iss_kv_head;
  int iss_slot, cons_slot;
  uint32_t cons_phase;
  int in_flight;
  bool dead;           // a bounded wait ran out: stop fetching, drain, leave
  bool drop_next;      // test hook: the next tile's copy is left out
  uint64_t policy;     // L2 policy of the tile copies
};

__device__ __forceinline__ void worker_init(WorkerState& st, int n_my) {
  st.n_my = n_my;
  st.cons_k = st.iss_k = 0;
  st.iss_pages = st.iss_which = st.iss_first = st.iss_last = 0;
  st.iss_addr = 0;
  st.iss_kv_head = 0;
  st.iss_slot = st.cons_slot = 0;
  st.cons_phase = 0;
  st.in_flight = 0;
  st.dead = false;
  st.drop_next = false;
  st.policy = l2_evict_first_policy();
}

// Issue the copy of the next tile.  D: head dim; RING: slots; TMAP: copy through the tensor
// map (swizzled tile: two 64-element column halves per row when D == 128) instead of one
// linear 16*D*2-byte bulk copy.  `ctx(k)` returns the ItemPages of the worker's k-th item.
// What an item's tiles have in common is looked up once per item: a worker issues a copy for every
// tile it consumes, between the arithmetic of two tiles, so each instruction here is on its path
// (with the look-ups per tile, a proxy fence and a policy made for each copy, a copy cost 700
// cycles and a page of a K and a V tile 3 100, in a CTA with every worker busy; now 550 and 2 500).  No proxy fence is needed for a slot that was only
// read; where a worker writes into a tile (new rows, cleared rows) it fences itself.
template <int D, int RING, bool TMAP, typename CtxFn>
__device__ __forceinline__ bool issue_one(WorkerState& st, CtxFn ctx, uint32_t ring, uint64_t* full, const Params& P,
                                          int lane) {
  constexpr uint32_t kTile = kPage * D * 2;
  if (st.iss_pages == 0) {   // the next item
    if (st.dead || st.iss_k >= st.n_my || st.iss_k > st.cons_k + 1) return false;
    const ItemPages& c = ctx(st.iss_k);
    st.iss_pages = c.item.n_pages;
    st.iss_first = (c.item.flags & kFlagReadLogits) ? 1 : 0;   // (scores from the logit cache: no K tile)
    st.iss_last = c.item.n_cons;
    st.iss_which = st.iss_first;
    st.iss_kv_head = c.kv_head;
    st.iss_addr = smem_u32(&c.pages[st.iss_first][0]);
  }
  int pid;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(pid) : "r"(st.iss_addr) : "memory");
  if (static_cast<uint32_t>(pid) >= static_cast<uint64_t>(P.n_pool_pages)) {   // never read outside the pool
    if (lane == 0) report_error(P.err, P.err_host, kErrBadPage);
    pid = 0;
  }
  if (st.drop_next) {
    // test hook: count the tile as in flight without requesting it; its wait will run out
    st.drop_next = false;
  } else if (lane == 0) {
    uint64_t* bar = full + st.iss_slot;
    const uint32_t dst = ring + st.iss_slot * kTile;
    mbar_expect_tx(bar, kTile);
    if (TMAP) {
      tensor_g2s_3d(dst, &P.tmap, 0, (pid * P.hkv + st.iss_kv_head) * kPage, 0, bar, st.policy);
    } else {
      const uint16_t* src = P.pool + (static_cast<size_t>(pid) * P.hkv + st.iss_kv_head) * (kPage * D);
      bulk_g2s(dst, src, kTile, bar, st.policy);
    }
  }
  st.iss_slot = (st.iss_slot + 1 == RING) ? 0 : st.iss_slot + 1;
  st.in_flight++;
  constexpr uint32_t kStream = kMaxChunkPages * 4;   // bytes from one stream's page ids to the next one's
  if (st.iss_which == st.iss_last) {   // next page
    st.iss_addr -= (st.iss_last - st.iss_first) * kStream - 4;
    st.iss_which = st.iss_first;
    if (--st.iss_pages == 0) st.iss_k++;
  } else {
    st.iss_addr += kStream;
    st.iss_which++;
  }
  return true;
}

template <int D, int RING, bool TMAP, typename CtxFn>
__device__ __forceinline__ void fill_ring(WorkerState& st, CtxFn ctx, uint32_t ring, uint64_t* full, const Params& P,
                                          int lane) {
  while (st.in_flight < RING) {
    if (!issue_one<D, RING, TMAP>(st, ctx, ring, full, P, lane)) break;
  }
}

// Wait until the oldest tile in flight has landed; returns its shared-memory address.
template <int D>
__device__ __forceinline__ uint32_t wait_tile(WorkerState& st, uint32_t ring, uint64_t* full, const Params& P,
                                              int lane) {
  constexpr uint32_t kTile = kPage * D * 2;
  uint64_t* bar = full + st.cons_slot;
  if (!mbar_try_wait(bar, st.cons_phase)) {
    uint32_t done = 0;
    const uint32_t limit = P.debug_drop_tile ? kDebugSpinLimit : kSpinLimit;
    for (uint32_t spin = 0; !done && spin < limit; ++spin) done = mbar_try_wait(bar, st.cons_phase);
    if (!done) {
      if (lane == 0) report_error(P.err, P.err_host, kErrTimeout);
      st.dead = true;
    }
  }
  return ring + st.cons_slot * kTile;
}

template <int RING>
__device__ __forceinline__ void release_tile(WorkerState& st) {
  __syncwarp();
  st.in_flight--;
  if (++st.cons_slot == RING) {
    st.cons_slot = 0;
    st.cons_phase ^= 1u;
  }
}

// After a failed wait: copies still in flight write into this CTA's shared memory; give them
// a bounded chance to land before the warp leaves.
template <int RING>
__device__ __forceinline__ void drain_ring(WorkerState& st, uint64_t* full, uint32_t limit = kSpinLimit) {
  while (st.in_flight > 0) {
    uint64_t* bar = &full[st.cons_slot];
    uint32_t done = 0;
    for (uint32_t spin = 0; !done && spin < limit; ++spin) done = mbar_try_wait(bar, st.cons_phase);
    st.in_flight--;
    if (++st.cons_slot == RING) {
      st.cons_slot = 0;
      st.cons_phase ^= 1u;
    }
  }
}

// A warp keeps the contexts of three items: the one it consumes, the next one (whose tiles the ring
// already fetches) and the one after, which is being filled by asynchronous copies meanwhile.
constexpr int kCtxSlots = 3;

// Start filling a context slot that holds an item with the page ids of its K stream and V streams
// (asynchronous copies; cp_async_wait_all() + __syncwarp() completes them).
__device__ __forceinline__ void begin_item_pages(ItemPages& c, const Params& P, int lane) {
  const Item& it = c.item;
  if (lane < it.n_pages) {
    cp_async_4(&c.pages[0][lane], P.table + table_row(P, it.k_layer, it.stream, it.seq_id) + it.first_page + lane);
    for (int x = 0; x < it.n_cons; ++x)
      cp_async_4(&c.pages[1 + x][lane],
                 P.table + table_row(P, it.v_layer[x], 2 + it.stream, it.seq_id) + it.first_page + lane);
  }
}

// Fetch an item's descriptor from the item list into a context slot.  (Items live in shared memory only: a
// variable whose arrays are indexed at run time is local memory, and what twelve warps have of that does not stay
// in the L1 cache beside the tiles.)
__device__ __forceinline__ void load_item(ItemPages& c, const Params& P, int item_idx, int lane) {
  __syncwarp();   // the slot's previous item is no longer read
  if (lane < 2) reinterpret_cast<uint4*>(&c.item)[lane] = __ldg(reinterpret_cast<const uint4*>(P.items + item_idx) + lane);
  __syncwarp();
  if (lane == 0) c.kv_head = c.item.head / P.group;
}

// Items of a launch are handed out in list order (heaviest first, so the work left at the end
// comes in small pieces).  A claim is an atomic increment by lane 0.  It is issued when an item ends and
// looked at when the next one begins; issued an item ahead, its result is one more register across the
// page loops, which have none to spare (one-launch steps, us per layer: 12 sequences of 1 300 keys 32.8 -> 31.3 with the
// claim at the end, 4 of 4 200 36.0 -> 35.1, 30 of 260 13.7 -> 13.4).
__device__ __forceinline__ int claim_issue(const Params& P, int lane) {
  int idx = 0;
  if (lane == 0) idx = atomicAdd(P.work_counter + P.launch_index, 1);
  return idx;
}
// Where the scaled scores of (stream, sequence, head) start in the logit cache; key j of the stream
// is element j.
__device__ __forceinline__ float* logit_row(const Params& P, int stream, int seq_id, int head) {
  return P.logits + ((static_cast<size_t>(stream) * P.max_seqs + seq_id) * P.hq + head) *
                        (static_cast<size_t>(P.max_pages) * kPage);
}

// Turns the value returned by claim_issue into an item index, or -1 when the list is used up.
__device__ __forceinline__ int claim_take(const Params& P, int issued) {
  const int idx = __shfl_sync(0xffffffffu, issued, 0);
  return idx < P.item_end - P.item_begin ? P.item_begin + idx : -1;
}

// ------------------------------------------------------------------------------------------
// static partition of a launch
// ------------------------------------------------------------------------------------------
//
// The work of a launch is laid out in tiles: listed sequences in order, inside a sequence the rows
// (one per query head, or per query group with GQA), inside a row the launch's plan positions,
// inside a position the row's pages, each page worth w tiles (one K tile unless the scores come
// from the logit cache, one V tile per consumer) after a fixed part_row_cost (what starting and
// finishing an item costs a worker).  The space of T tiles is cut into ranges of part_q tiles; a
// page belongs to the range its first tile falls into.  Physical worker i takes ranges i*part_k ..
// i*part_k + part_k - 1, which are adjacent, so it walks forward from one starting point; the
// workers of a CTA are adjacent too, so a CTA owns one stretch of tiles and with it, apart from the
// rows at the two ends of the stretch, everything that the output rows in it need (finish_cta).
// The pages of a row and position that one range owns are one piece: an Item whose partial result
// goes to slot (range - range owning the first of those pages) of the row's stream.  The host plans
// part_q so that a range is at least as long as any page (every range between a row's first and
// last owns a page of it: no slot is left unwritten), a piece has at most kMaxChunkPages pages and
// a row at most slots_per_stream pieces per stream; T < 2^31.

struct __align__(16) RangeCursor {
  int32_t r0;        // tile offset of the first page of the current row and position
  int32_t vw_end;    // first tile beyond the current range
  int32_t vw, vw_stop;
  int32_t pos, si, u;
  int32_t row_pages, w;     // pages of the current row and position; tiles per page of its job
  int32_t page;             // next page to hand out
  int32_t owner0;           // range that owns the first page
  int32_t len_text, len_vis, seq_id;   // of the current sequence
  int32_t pad[2];
  Job job;
};
static_assert(sizeof(RangeCursor) == 80, "RangeCursor layout");

// What the partition of one launch is made of (the attention kernels take it from their
// parameters, the kernel that plans every launch of a step ahead from its launch list).
struct PartView {
  const PlanJob* plan;
  const StepSeq* seqs;
  int32_t* err;
  int32_t* err_host;
  int32_t pos_begin, pos_end, n_seqs;
  int32_t q, k, vw, row_cost;          // tiles per range, ranges per worker, ranges, fixed tiles per row and position
  int32_t wv, wt;                      // tiles per page summed over the launch's visual / text positions
  int32_t rows, heads_per_item, group, slots_per_stream;   // rows per sequence; query heads per row
};

__device__ __forceinline__ PartView part_view(const Params& P) {
  PartView V;
  V.plan = P.plan, V.seqs = P.seqs, V.err = P.err, V.err_host = P.err_host;
  V.pos_begin = P.pos_begin, V.pos_end = P.pos_end, V.n_seqs = P.n_seqs;
  V.q = P.part_q, V.k = P.part_k, V.vw = P.part_vw, V.row_cost = P.part_row_cost;
  V.wv = P.part_wv, V.wt = P.part_wt;
  V.rows = P.heads_per_item_dim, V.heads_per_item = P.heads_per_item, V.group = P.group;
  V.slots_per_stream = P.slots_per_stream;
  return V;
}
__device__ __forceinline__ PartView part_view(const Params& P, const LaunchDesc& L) {
  PartView V = part_view(P);
  V.pos_begin = L.pos_begin, V.pos_end = L.pos_end;
  V.q = L.part_q, V.k = L.part_k, V.vw = L.part_vw, V.row_cost = L.part_row_cost;
  V.wv = L.part_wv, V.wt = L.part_wt;
  return V;
}

__device__ __forceinline__ int job_tiles_per_page(const Job& j) {
  return ((j.flags & kFlagReadLogits) ? 0 : 1) + j.n_cons;
}
__device__ __forceinline__ int pages_of(int tokens) { return (tokens + kPage - 1) / kPage; }

// Tile offset at which the rows of listed sequence si start; tiles of one of its rows.
__device__ __forceinline__ int32_t seq_base(const PartView& V, int32_t pre_v, int32_t pre_t, int si) {
  return V.rows * (V.wv * pre_v + V.wt * pre_t + V.row_cost * (V.pos_end - V.pos_begin) * si);
}
__device__ __forceinline__ int32_t row_tiles(const PartView& V, int32_t len_vis, int32_t len_text) {
  return V.wv * pages_of(len_vis) + V.wt * pages_of(len_text) + V.row_cost * (V.pos_end - V.pos_begin);
}

// The listed sequence and the row that tile t falls into; returns the row's first tile.
__device__ __forceinline__ int32_t find_row(const PartView& V, int32_t t, int& si, int& u, StepSeq& sq) {
  int lo = 0, hi = V.n_seqs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (seq_base(V, V.seqs[mid].pre_v, V.seqs[mid].pre_t, mid) <= t) lo = mid;
    else hi = mid - 1;
  }
  si = lo;
  sq = V.seqs[lo];
  const int32_t base = seq_base(V, sq.pre_v, sq.pre_t, lo), per_row = row_tiles(V, sq.len_vis, sq.len_text);
  u = per_row > 0 ? min(V.rows - 1, (t - base) / per_row) : 0;
  return base + u * per_row;
}

// Load the job of plan position c.pos into the cursor.
__device__ __forceinline__ void cursor_load_job(RangeCursor& c, const PartView& V) {
  const uint4 raw = __ldg(reinterpret_cast<const uint4*>(V.plan + c.pos));
  *reinterpret_cast<uint4*>(&c.job) = raw;
  c.w = job_tiles_per_page(c.job);
  c.row_pages = pages_of(c.job.stream ? c.len_vis : c.len_text);
}

// Place the cursor of worker `wid` at its first range; false if the worker has no work.  Reads the
// launch plan and the step's sequence descriptors only.
__device__ __forceinline__ bool cursor_init(RangeCursor& c, const PartView& V, int wid) {
  c.vw = wid * V.k;
  c.vw_stop = min(c.vw + V.k, V.vw);
  if (c.vw >= c.vw_stop) return false;
  const int32_t t0 = c.vw * V.q;
  c.vw_end = t0 + V.q;
  StepSeq sq;
  const int32_t row0 = find_row(V, t0, c.si, c.u, sq);
  c.len_text = sq.len_text, c.len_vis = sq.len_vis, c.seq_id = sq.seq_id;
  // the first position of the row whose pages do not all start before t0, or the last one
  c.r0 = row0 + V.row_cost;
  c.pos = V.pos_begin;
  cursor_load_job(c, V);
  while (c.pos + 1 < V.pos_end && c.r0 + c.w * c.row_pages <= t0) {
    c.r0 += c.w * c.row_pages + V.row_cost;
    ++c.pos;
    cursor_load_job(c, V);
  }
  c.page = t0 > c.r0 ? (t0 - c.r0 + c.w - 1) / c.w : 0;   // first page that starts at or after t0
  c.owner0 = c.r0 / V.q;
  c.pad[0] = c.pad[1] = 0;
  return true;
}

// Next piece of the worker's ranges, or false when they are used up.  Warp-uniform.
__device__ __forceinline__ bool cursor_next(RangeCursor& c, const PartView& V, Item& it) {
  for (;;) {
    if (c.vw >= c.vw_stop) return false;
    if (c.page >= c.row_pages) {   // next position, row, sequence
      c.r0 += c.w * c.row_pages + V.row_cost;
      c.page = 0;
      if (++c.pos == V.pos_end) {
        c.pos = V.pos_begin;
        if (++c.u == V.rows) {
          c.u = 0;
          if (++c.si == V.n_seqs) {
            c.vw = c.vw_stop;
            return false;
          }
          const StepSeq sq = V.seqs[c.si];
          c.len_text = sq.len_text, c.len_vis = sq.len_vis, c.seq_id = sq.seq_id;
        }
      }
      cursor_load_job(c, V);
      c.owner0 = c.r0 / V.q;
      continue;
    }
    const int32_t d = c.vw_end - c.r0;
    const int lim = d <= 0 ? 0 : min(c.row_pages, (d + c.w - 1) / c.w);
    if (c.page < lim) {
      const int hpi = V.heads_per_item;
      const int n_sub = (V.group + hpi - 1) / hpi;
      const int kv_head = c.u / n_sub, sub = c.u - kv_head * n_sub;
      const int slot = c.vw - c.owner0;
      it.k_layer = c.job.k_layer;
      it.stream = c.job.stream;
      it.n_cons = c.job.n_cons;
      it.flags = c.job.flags;
#pragma unroll
      for (int x = 0; x < kMaxCons; ++x) {
        it.v_layer[x] = c.job.v_layer[x];
        it.q_layer[x] = c.job.q_layer[x];
      }
      it.seq_id = static_cast<uint16_t>(c.seq_id);
      it.seq_idx = static_cast<uint16_t>(c.si);
      it.head = static_cast<uint16_t>(kv_head * V.group + sub * hpi);
      it.slot = static_cast<uint16_t>((c.job.stream ? 0 : V.slots_per_stream) + slot);
      it.first_page = static_cast<uint16_t>(c.page);
      it.n_pages = static_cast<uint16_t>(lim - c.page);
      const bool last = lim == c.row_pages;
      if (last) it.flags |= kFlagStreamEnd;
      it.n_valid_last = static_cast<uint16_t>(last ? (c.job.stream ? c.len_vis : c.len_text) - (c.row_pages - 1) * kPage : kPage);
      it.n_heads = static_cast<uint8_t>(min(hpi, V.group - sub * hpi));
      it.skip_new = c.job.skip_new;
      it.pad0 = it.pad1 = 0;
      // the piece that holds the first page tells the merge how many pieces there are
      it.n_pieces = c.page == 0 ? static_cast<uint16_t>((c.r0 + c.w * (c.row_pages - 1)) / V.q - c.owner0 + 1) : 0;
      if (lim - c.page > kMaxChunkPages || slot < 0 || slot >= V.slots_per_stream) {   // outside the plan's limits
        report_error(V.err, V.err_host, kErrPlan);
        c.vw = c.vw_stop;
        return false;
      }
      c.page = lim;
      return true;
    }
    // the current range owns nothing (more) of this row and position
    ++c.vw;
    c.vw_end += V.q;
  }
}

// One step of a worker's cursor, kept in shared memory between items: the next item into a context slot.
// Warp-uniform.
__device__ __forceinline__ bool cursor_step(RangeCursor* cursor, const Params& P, ItemPages& slot, int lane) {
  __syncwarp();
  RangeCursor c = *cursor;
  Item it;
  const bool ok = cursor_next(c, part_view(P), it);
  __syncwarp();
  if (lane == 0) {
    *cursor = c;
    if (ok) {
      slot.item = it;
      slot.kv_head = it.head / P.group;
    }
  }
  __syncwarp();
  return ok;
}

// Folded append: is page `pg` of the item the page that receives the step's new token?
__device__ __forceinline__ bool holds_new_token(const Params& P, const Item& it, int pg) {
  return P.fold_append && it.stream == 0 && (it.flags & kFlagStreamEnd) && pg == it.n_pages - 1;
}

// Folded append: start fetching the new token's rows of an item that ends its layer's text stream
// (this layer's inputs: after the wait for the previous kernel, with the queries).
__device__ __forceinline__ int first_taker(const Item& it) {   // first consumer that does not leave out the new token
  for (int x = 0; x < it.n_cons; ++x)
    if (!((it.skip_new >> x) & 1)) return x;
  return -1;
}
__device__ __forceinline__ void begin_new_rows(ItemPages& c, const Params& P, int lane, int d) {
  const Item& it = c.item;
  if (!(P.fold_append && it.stream == 0 && (it.flags & kFlagStreamEnd))) return;
  const int n_vec = d / 8, kv_head = it.head / P.group;
  if (lane < n_vec)
    cp_async_16(&c.new_k[lane], reinterpret_cast<const uint4*>(
                                    P.k + ((static_cast<size_t>(it.k_layer) * P.n_seqs + it.seq_idx) * P.hkv + kv_head) * d) + lane);
  const int x = first_taker(it);
  if (x >= 0 && lane >= 16 && lane - 16 < n_vec)
    cp_async_16(&c.new_v[lane - 16],
                reinterpret_cast<const uint4*>(
                    P.v + ((static_cast<size_t>(it.v_layer[x]) * P.n_seqs + it.seq_idx) * P.hkv + kv_head) * d) + (lane - 16));
}

// Start of a worker from the descriptor planned for it when the step began: the first item goes
// into the first context slot together with the page ids of its first two pages, the second item
// into the second slot, the cursor into the worker's cursor slot.  False if the worker has no
// work.  `stage`: 48 bytes of shared memory.  The first warp also fetches the CTA's descriptor,
// where the launch merges its rows itself.
__device__ __forceinline__ bool load_worker_desc(const Params& P, int wid, ItemPages& c0, ItemPages& c1, RangeCursor* cursor,
                                                 int32_t* stage, CtaDesc* cta, int lane) {
  const uint4* d = reinterpret_cast<const uint4*>(P.wdesc + static_cast<size_t>(P.launch_index) * kPlanWorkers + wid);
  if (lane < 12) {
    uint4* dst = lane < 2 ? reinterpret_cast<uint4*>(&c0.item) + lane
                 : lane < 4 ? reinterpret_cast<uint4*>(&c1.item) + (lane - 2)
                 : lane < 7 ? reinterpret_cast<uint4*>(stage) + (lane - 4)
                            : reinterpret_cast<uint4*>(cursor) + (lane - 7);
    cp_async_16(dst, d + lane);
  } else if (lane < 17 && threadIdx.x < 32 && P.fused_merge) {
    cp_async_16(reinterpret_cast<uint4*>(cta) + (lane - 12),
                reinterpret_cast<const uint4*>(P.cdesc + static_cast<size_t>(P.launch_index) * kPlanCtas + blockIdx.x) + (lane - 12));
  }
  cp_async_wait_all();
  __syncwarp();
  if (c0.item.n_pages == 0) return false;
  if (lane < 2 * (1 + kMaxCons)) c0.pages[lane >> 1][lane & 1] = stage[lane];
  if (lane == 0) c0.kv_head = c0.item.head / P.group, c1.kv_head = c1.item.head / P.group;
  __syncwarp();
  return true;
}

// Which worker of a statically partitioned launch a warp is, or -1: the workers of a CTA are
// adjacent (the same rows, page-table lines and queries, and the rows a CTA can merge by itself).
__device__ __forceinline__ int worker_index(const Params& P, int warp) {
  return warp < P.part_wpc ? static_cast<int>(blockIdx.x) * P.part_wpc + warp : -1;
}

// Under the static partition, the piece that holds a row's first page records how many pieces
// the row has: one entry per consumer layer and query head, visual and text streams side by side.
__device__ __forceinline__ void record_row_slots(const Params& P, const Item& it, int lane) {
  if (it.n_pieces == 0 || P.planned_pieces) return;   // (planned: row_pieces has them)
  const int x = lane >> 3, h = lane & 7;
  if (x < it.n_cons && h < it.n_heads) {
    const size_t row = (static_cast<size_t>(it.v_layer[x]) * P.max_seqs + it.seq_idx) * P.hq + it.head + h;
    P.row_slots[2 * row + (it.stream ? 0 : 1)] = it.n_pieces;
  }
}

// ------------------------------------------------------------------------------------------
// log-sum-exp merge of output rows
// ------------------------------------------------------------------------------------------
//
// An output row's partials are nv rows of the visual stream in slots 0 .. nv - 1 and nt rows of the
// text stream in slots text0 .. text0 + nt - 1.  They may have been written by other SMs moments
// ago: they are read past the L1 cache.

template <int D>
struct RowSum {   // one warp's sum over partials; lane i holds elements i * D/32 ...
  float m, l, acc[D / 32];
};

template <int VPL>
__device__ __forceinline__ void load_elems(float (&v)[VPL], const float* src) {
  if constexpr (VPL == 4) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(src));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
  } else {
    const float2 a = __ldcg(reinterpret_cast<const float2*>(src));
    v[0] = a.x, v[1] = a.y;
  }
}

// Sum of partials first, first + step, ... of the n = nv + nt of one output row.  Lane s holds the
// (max, sum) pair of the s-th of them; the accumulator rows do not depend on the pairs, so the
// first of them are requested together with the pairs.
template <int D>
__device__ __forceinline__ void sum_partials(const Params& P, size_t base, int head, int nv, int nt, int text0, int first,
                                             int step, int lane, RowSum<D>& r) {
  constexpr int VPL = D / 32;
  constexpr int kBatch = D == 128 ? 12 : 16;
  const int n = nv + nt;
  const float* acc0 = P.part_acc + (base * P.hq + head) * D + lane * VPL;
  const float2* ml0 = P.part_ml + base * P.hq + head;
  const uint32_t acc_stride = static_cast<uint32_t>(P.hq) * D;
  auto slot_of = [&](int s) { return static_cast<uint32_t>(s < nv ? s : text0 + (s - nv)); };
  r.m = -INFINITY, r.l = 0.f;
#pragma unroll
  for (int e = 0; e < VPL; ++e) r.acc[e] = 0.f;
  for (int c0 = first; c0 < n; c0 += 32 * step) {
    const int cnt = min(32, (n - c0 + step - 1) / step);
    float2 ml = make_float2(-INFINITY, 0.f);
    if (lane < cnt) ml = __ldcg(ml0 + static_cast<size_t>(slot_of(c0 + lane * step)) * P.hq);
    float v[kBatch][VPL];
    auto request = [&](int s0) {
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (s0 + u < cnt) load_elems<VPL>(v[u], acc0 + static_cast<size_t>(slot_of(c0 + (s0 + u) * step)) * acc_stride);
    };
    request(0);
    // A sweep that left out its only key has an empty partial (sum 0, weight 0).  A sum that is not a number
    // has weight 0 too, but makes the row's sum, and with it the row, not a number.
    float m_new = ml.y > 0.f ? ml.x : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, o));
    m_new = fmaxf(m_new, r.m);
    const float ref = m_new == -INFINITY ? 0.f : m_new;   // (nothing that counts so far)
    const float corr = exp2f(r.m - ref);
    const float w = ml.y > 0.f ? exp2f(ml.x - ref) : 0.f;
    float ls = ml.y * w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
    r.m = m_new;
    r.l = r.l * corr + ls;
#pragma unroll
    for (int e = 0; e < VPL; ++e) r.acc[e] *= corr;
    for (int s0 = 0; s0 < cnt; s0 += kBatch) {
      if (s0 > 0) request(s0);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const float wu = __shfl_sync(0xffffffffu, w, (s0 + u) & 31);
        if (s0 + u < cnt && wu > 0.f) {
#pragma unroll
          for (int e = 0; e < VPL; ++e) r.acc[e] = fmaf(v[u][e], wu, r.acc[e]);
        }
      }
    }
  }
}

// The finished output row: normalised, bf16, with the optional log-sum-exp.
template <int D>
__device__ __forceinline__ void store_row(const Params& P, int layer, int si, int head, const RowSum<D>& r, int lane) {
  constexpr int VPL = D / 32;
  const float inv = 1.f / r.l;
  const size_t orow = ((static_cast<size_t>(layer) * P.n_seqs + si) * P.hq + head);
  uint16_t* dst = P.out + orow * D + lane * VPL;
  uint32_t o[VPL / 2];
#pragma unroll
  for (int e = 0; e < VPL; e += 2)
    o[e / 2] = f32_to_bf16_rne(r.acc[e] * inv) | (static_cast<uint32_t>(f32_to_bf16_rne(r.acc[e + 1] * inv)) << 16);
  if constexpr (VPL == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(o[0], o[1]);
  else *reinterpret_cast<uint32_t*>(dst) = o[0];
  if (P.lse != nullptr && lane == 0) P.lse[orow] = (r.m + log2f(r.l)) * 0.6931471805599453f;
}

// Merge of one output row by a launch of its own (merge_kernel), including the wait for the launch that leaves
// the last partials.  With claimed items the numbers of partials follow from the stream lengths; launches of
// one layer under the static partition have them planned; otherwise the sweeps recorded them.
// P.extra_key_leader >= 0 adds the step's new token as one more key (rows of a GLA follower under the in-order
// schedule; Eq. 6). ROWS: the step's rows had thread blocks of their own, what there is is one partial row from
// the leader's launch (an instantiation of its own: with both in one, two turns of 8 steps of a 64-wide GLA
// stack took 1 272 us, now 1 223, and a step of two layers with claimed items 14.6 us, now 14.45).
template <int D, bool ROWS>
__device__ __forceinline__ void merge_row(const Params& P, int layer, int si, int head, int lane) {
  constexpr int VPL = D / 32;
  const size_t base = (static_cast<size_t>(layer) * P.max_seqs + si) * P.max_slots;
  const int kvh = head / P.group, extra_leader = P.extra_key_leader;
  const StepSeq sq = P.seqs[si];
  int nv = sq.ncv, nt = sq.n_slots - sq.ncv, text0 = sq.ncv;
  if (ROWS) {
    nv = 1, nt = 0;
  } else if (P.planned_pieces) {
    const int hpi = P.heads_per_item, n_sub = (P.group + hpi - 1) / hpi, rows = P.heads_per_item_dim;
    const int u = kvh * n_sub + (head - kvh * P.group) / hpi;
    const uint32_t both = __ldcg(P.row_pieces + (static_cast<size_t>(P.launch_index) * P.max_seqs + si) * rows + u);
    nv = both & 0xffffu, nt = both >> 16, text0 = P.slots_per_stream;
  }
  const int pos = sq.len_text - 1;
  int pid = 0, pid_v = -1;
  if (extra_leader >= 0) {
    pid = P.table[table_row(P, extra_leader, 0, sq.seq_id) + pos / kPage];
    if (P.fold_append && head % P.group == 0) pid_v = P.table[table_row(P, layer, 2, sq.seq_id) + pos / kPage];
    if (static_cast<uint32_t>(pid) >= static_cast<uint64_t>(P.n_pool_pages)) {   // never read outside the pool
      if (lane == 0) report_error(P.err, P.err_host, kErrBadPage);
      pid = 0;
    }
  }
  // the layer's new v row is the caller's tensor and seldom in the L2 yet (12 layers of 64-wide heads in GLA blocks of four, two
  // turns of 8 steps: 1 282 -> 1 268 us)
  if (extra_leader >= 0 && lane < VPL / 2)
    l2_prefetch(P.v + ((static_cast<size_t>(layer) * P.n_seqs + si) * P.hkv + kvh) * D + lane * 64);
  pdl_wait();
  pdl_launch_dependents();
  if (!ROWS && P.part_static && !P.planned_pieces) {
    const size_t row = (static_cast<size_t>(layer) * P.max_seqs + si) * P.hq + head;
    const uint32_t both = __ldcg(reinterpret_cast<const uint32_t*>(P.row_slots + 2 * row));
    nv = sq.len_vis > 0 ? static_cast<int>(both & 0xffffu) : 0;
    nt = static_cast<int>(both >> 16);
    text0 = P.slots_per_stream;
  }
  float s_new = -INFINITY, vn[VPL];
  if (extra_leader >= 0) {
    const uint16_t* qrow = P.qcache + ((static_cast<size_t>(extra_leader) * P.max_seqs + sq.seq_id) * P.hq + head) * D;
    // the leader's new k: the last row of its text K stream (appended before this kernel ran)
    const uint16_t* krow = P.pool + ((static_cast<size_t>(pid) * P.hkv + kvh) * kPage + pos % kPage) * D;
    const uint16_t* v_new = P.v + ((static_cast<size_t>(layer) * P.n_seqs + si) * P.hkv + kvh) * D + lane * VPL;
    uint32_t q2[VPL / 2], k2[VPL / 2], v2[VPL / 2];
#pragma unroll
    for (int e = 0; e < VPL / 2; ++e) {
      q2[e] = __ldcg(reinterpret_cast<const uint32_t*>(qrow + lane * VPL) + e);
      k2[e] = __ldcg(reinterpret_cast<const uint32_t*>(krow + lane * VPL) + e);
      v2[e] = __ldcg(reinterpret_cast<const uint32_t*>(v_new) + e);
    }
    float dot = 0.f;
#pragma unroll
    for (int e = 0; e < VPL / 2; ++e) {
      dot = fmaf(__uint_as_float(q2[e] << 16), __uint_as_float(k2[e] << 16), dot);
      dot = fmaf(__uint_as_float(q2[e] & 0xffff0000u), __uint_as_float(k2[e] & 0xffff0000u), dot);
      vn[2 * e] = __uint_as_float(v2[e] << 16);
      vn[2 * e + 1] = __uint_as_float(v2[e] & 0xffff0000u);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    s_new = dot * P.scale_log2;
    if (P.fold_append && head % P.group == 0) {
      // this layer's new v row has no sweep to store it: the merge warp of the KV head's first query head does
      if (static_cast<uint32_t>(pid_v) < static_cast<uint64_t>(P.n_pool_pages)) {
        uint32_t* dst_v = reinterpret_cast<uint32_t*>(
            P.pool + ((static_cast<size_t>(pid_v) * P.hkv + kvh) * kPage + pos % kPage) * D + lane * VPL);
#pragma unroll
        for (int e = 0; e < VPL / 2; ++e) dst_v[e] = v2[e];
      } else if (lane == 0) {
        report_error(P.err, P.err_host, kErrBadPage);
      }
    }
  }
  RowSum<D> r;
  sum_partials<D>(P, base, head, nv, nt, text0, 0, 1, lane, r);
  if (extra_leader >= 0) {
    const float m_new = fmaxf(r.m, s_new);
    const float corr = exp2f(r.m - m_new), w = exp2f(s_new - m_new);
    r.m = m_new;
    r.l = r.l * corr + w;
#pragma unroll
    for (int e = 0; e < VPL; ++e) r.acc[e] = fmaf(w, vn[e], r.acc[e] * corr);
  }
  store_row<D>(P, layer, si, head, r, lane);
}

// ------------------------------------------------------------------------------------------
// merge by the attention launch itself (static partition, launches of one layer, no query groups)
// ------------------------------------------------------------------------------------------
//
// A CTA's workers own one stretch of the launch's tiles, ordered by output row.  When they are done,
// the rows that lie inside the stretch are complete: the CTA merges them.  The first and the
// last row of the stretch may be shared with other CTAs: such a row has a page counter, and the CTA
// whose pages complete the count merges it.  Everything but the partials themselves is known
// from the plan (which rows, how many pages and pieces), so what is left when the last worker
// stops is a barrier, one atomic per end (1 us), one round of reads and the store (2 us).  With the
// rows, pages and pieces worked out here instead it took 4.6 us, longer than a merge launch.

template <int D>
struct FinishSmem {
  float acc[kWarps][D];
  float2 ml[kWarps];
  int32_t ready[2];
  int32_t dead;
};

// Adds to a row's page counter: releases the partials that the CTA's workers stored (they are ordered
// before by the CTA's barrier), and the CTA that completes the count acquires everybody's.
__device__ __forceinline__ int count_pages(int32_t* counter, int n) {
  int old;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(old) : "l"(counter), "r"(n) : "memory");
  return old;
}

template <int D>
__device__ __forceinline__ void finish_cta(const Params& P, FinishSmem<D>& F, const CtaDesc& cta, bool dead, int warp, int lane) {
  constexpr int VPL = D / 32;
  if (!P.fused_merge) return;
  if (dead && lane == 0) F.dead = 1;
  __syncthreads();   // every worker's partial rows are stored
  if (F.dead) return;
  const int layer = P.layer_begin, rows = P.heads_per_item_dim;   // (one row per query head)
  if (warp < 2) {   // the rows at the ends: are they complete?
    const EndRow& e = cta.end[warp];
    int ready = e.here == e.total;
    if (e.here == 0) {
      ready = 0;
    } else if (!ready) {
      if (lane == 0) {
        ready = count_pages(P.row_done + e.counter, e.here) + e.here == e.total;
        if (ready) P.row_done[e.counter] = 0;   // for the next step
      }
    }
    if (lane == 0) F.ready[warp] = ready;
  }
  const int n_inner = max(0, cta.row_last - cta.row_first - 1);
  // first the rows between the ends, one warp per output row; then the ends that this CTA completed,
  // half of the warps each: which CTA completes a row, and whether it completes one or two, depends
  // on the run, so neither may decide the order in which the row's partials are added
  constexpr int kShare = kWarps / 2;
  static_assert(2 * kShare == kWarps, "two end rows share the warps");
  const int end = warp / kShare;
  RowSum<D> r;
  int o = kWarps - 1 - warp, n_out = n_inner, si = 0, head = 0;
#pragma unroll 1
  for (int phase = 0;; ++phase) {
#pragma unroll 1
    for (; o < n_out; o += kWarps) {
      int nv, nt;
      if (phase == 0) {
        const int row = cta.row_first + 1 + o;
        si = row / rows, head = row - si * rows;
        const uint32_t both = __ldcg(P.row_pieces + static_cast<size_t>(P.launch_index) * P.max_seqs * rows + row);
        nv = both & 0xffffu, nt = both >> 16;
      } else {
        const EndRow& e = cta.end[o];
        si = e.si, head = e.head, nv = e.nv, nt = e.nt;
      }
      sum_partials<D>(P, (static_cast<size_t>(layer) * P.max_seqs + si) * P.max_slots, head, nv, nt, P.slots_per_stream,
                      phase ? warp % kShare : 0, phase ? kShare : 1, lane, r);
      if (phase == 1) break;
      store_row<D>(P, layer, si, head, r, lane);
    }
    if (phase == 1) break;
    __syncthreads();
    if (!F.ready[0] && !F.ready[1]) return;
    o = end;
    n_out = F.ready[end] ? end + 1 : 0;   // (at most one round)
  }
  if (n_out > 0) {
#pragma unroll
    for (int e = 0; e < VPL; ++e) F.acc[warp][lane * VPL + e] = r.acc[e];
    if (lane == 0) F.ml[warp] = make_float2(r.m, r.l);
  }
  __syncthreads();
  if (n_out == 0) return;
  // every thread of the row's warps weighs their sums for some of the elements
  const int w0 = end * kShare;
  float w[kShare], m = -INFINITY, l = 0.f;
#pragma unroll
  for (int x = 0; x < kShare; ++x)
    if (F.ml[w0 + x].y > 0.f) m = fmaxf(m, F.ml[w0 + x].x);
#pragma unroll
  for (int x = 0; x < kShare; ++x) {
    const float2 ml = F.ml[w0 + x];
    w[x] = ml.y > 0.f ? exp2f(ml.x - m) : 0.f;   // (no partial, or empty ones: nothing)
    l = fmaf(ml.y, w[x], l);                     // (a sum that is not a number stays one)
  }
  const float inv = 1.f / l;
  const size_t orow = (static_cast<size_t>(layer) * P.n_seqs + si) * P.hq + head;
  for (int d = 2 * ((warp - w0) * 32 + lane); d < D; d += 64 * kShare) {
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int x = 0; x < kShare; ++x) {
      if (w[x] > 0.f) {
        a0 = fmaf(F.acc[w0 + x][d], w[x], a0);
        a1 = fmaf(F.acc[w0 + x][d + 1], w[x], a1);
      }
    }
    *reinterpret_cast<uint32_t*>(P.out + orow * D + d) =
        f32_to_bf16_rne(a0 * inv) | (static_cast<uint32_t>(f32_to_bf16_rne(a1 * inv)) << 16);
  }
  if (P.lse != nullptr && lane == 0 && warp == w0) P.lse[orow] = (m + log2f(l)) * 0.6931471805599453f;
}

}  // namespace
}  // namespace qc
