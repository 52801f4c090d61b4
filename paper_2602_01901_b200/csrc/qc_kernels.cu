// CUDA kernels of the Lazy Attention decode path (sm_100a).
//
//   setup_kernel    expands the step's (plan position, sequence) pairs into split-KV work items,
//                   applies page-table patches, resets the work counters and -- on steps without
//                   patches -- also does the append
//   append_kernel   writes the new token's k / v rows into the text streams and every
//                   ordinary layer's q into the Q Cache (a launch of its own on steps with patches
//                   and per launch group of the host-buffer entry point)
//   plan_kernel     for a step whose launches are cut into static tile ranges: where every worker of
//                   every launch starts (first item, its first page ids, the cursor for the rest)
//   attend_kernel   persistent split-KV partial attention, one query head per work item (MHA):
//                   each warp is an independent worker that takes items -- claimed from a counter,
//                   or the pieces of its static range of the launch's tiles -- streams K/V page
//                   tiles through its own shared-memory ring with bulk asynchronous copies and
//                   keeps an online softmax in registers; a leader's sweep can weight several
//                   layers' V rows with one set of scores, store its scaled scores in the logit
//                   cache, or leave out the step's new token for its followers
//                   (the grouped-query variant on tensor cores is in qc_attend_tc.cu)
//   merge_kernel    log-sum-exp merge of the partials, bf16 output
//   prefill_store_kernel  stores prompt K/V rows into their pages
//
// Attention arithmetic: scores are kept in the log2 domain (q is pre-multiplied by
// scale * log2 e), accumulation is fp32, inputs and outputs are bf16.

#include "qc_device.cuh"

namespace qc {
namespace {

// ------------------------------------------------------------------------------------------
// setup: page-table patches + item expansion
// ------------------------------------------------------------------------------------------

// new token's k, v rows of one (sequence, layer) and the Q Cache refresh
__device__ __forceinline__ void append_rows(const Params& P, const StepSeq& sq, int si, int layer) {
  const int pos = sq.len_text - 1;          // ordinal of the new token in the text stream
  const int pg = pos / kPage, slot = pos % kPage;
  const uint8_t lf = P.layer_flags[layer];
  const int vec_per_row = P.d / 8;          // uint4 per head row
  const int n_kv_vec = P.hkv * vec_per_row;
  const size_t in_kv = (static_cast<size_t>(layer) * P.n_seqs + si) * P.hkv * P.d;

  const int pid_v = P.table[table_row(P, layer, 2, sq.seq_id) + pg];
  const int pid_k = (lf & kLayerOwnsTextK) ? P.table[table_row(P, layer, 0, sq.seq_id) + pg] : -1;
  for (int e = threadIdx.x; e < n_kv_vec; e += blockDim.x) {
    const int head = e / vec_per_row, j = e - head * vec_per_row;
    const size_t src = in_kv + static_cast<size_t>(head) * P.d + j * 8;
    const size_t dst_v = ((static_cast<size_t>(pid_v) * P.hkv + head) * kPage + slot) * P.d + j * 8;
    *reinterpret_cast<uint4*>(P.pool + dst_v) = *reinterpret_cast<const uint4*>(P.v + src);
    if (pid_k >= 0) {
      const size_t dst_k = ((static_cast<size_t>(pid_k) * P.hkv + head) * kPage + slot) * P.d + j * 8;
      *reinterpret_cast<uint4*>(P.pool + dst_k) = *reinterpret_cast<const uint4*>(P.k + src);
    }
  }
  if (lf & kLayerWritesQCache) {
    const int n_q_vec = P.hq * vec_per_row;
    const size_t src0 = (static_cast<size_t>(layer) * P.n_seqs + si) * P.hq * P.d;
    const size_t dst0 = (static_cast<size_t>(layer) * P.max_seqs + sq.seq_id) * P.hq * P.d;
    for (int e = threadIdx.x; e < n_q_vec; e += blockDim.x)
      reinterpret_cast<uint4*>(P.qcache + dst0)[e] = reinterpret_cast<const uint4*>(P.q + src0)[e];
  }
}

// Block roles, in grid order: n_pos * n_seqs blocks expand one (plan position, sequence) each
// into work items; housekeeping blocks apply page-table patches, reset the work counters and
// store the inline sequence descriptors for the later kernels; with fused_append, n_seqs *
// n_layers blocks do the append.  (The append reads page ids from the table, so it is only
// fused on steps without patches.)
__global__ void setup_kernel(const __grid_constant__ Params P, const __grid_constant__ StepInline inl) {
  // With claimed items the attention kernel touches nothing before its own wait, so it may be
  // scheduled while this kernel runs; under the static partition it plans its first work ahead of
  // its wait from what this kernel writes, and must not start early.
  if (!P.part_static) pdl_launch_dependents();
  pdl_wait();
  const StepSeq* seqs = P.inline_seqs ? inl.seqs : P.seqs;
  const int n_expand = P.n_pos * P.n_seqs;
  const int n_house = (max(max(P.n_patches, P.n_layers), P.n_seqs * 8) + blockDim.x - 1) / blockDim.x;
  int b = blockIdx.x;
  if (b >= n_expand + n_house) {   // append blocks
    b -= n_expand + n_house;
    const int si = b % P.n_seqs, layer = b / P.n_seqs;
    append_rows(P, seqs[si], si, layer);
    return;
  }
  if (b >= n_expand) {   // housekeeping blocks
    const int i = (b - n_expand) * blockDim.x + threadIdx.x;
    if (i < P.n_patches) P.table[P.patches[i].index] = P.patches[i].page;
    if (i < P.n_layers) P.work_counter[i] = 0;
    if (P.inline_seqs && i < P.n_seqs * 8)
      reinterpret_cast<int32_t*>(P.seqs)[i] = reinterpret_cast<const int32_t*>(inl.seqs)[i];
    return;
  }
  const int pos = b / P.n_seqs, si = b - pos * P.n_seqs;
  const StepSeq sq = seqs[si];
  const PlanJob pj = P.plan[pos];
  const Job jb = pj.job;
  const int len = jb.stream ? sq.len_vis : sq.len_text;
  const int n_chunks = jb.stream ? sq.ncv : sq.n_slots - sq.ncv;
  const int item_base = pj.vis_before * P.tot_v + pj.text_before * P.tot_t + (jb.stream ? sq.pre_v : sq.pre_t);
  const int slot_base = jb.stream ? 0 : sq.ncv;
  const int per_chunk = P.heads_per_item_dim;   // items per chunk
  const int hpi = P.heads_per_item;
  const int n_sub = (P.group + hpi - 1) / hpi;  // items per KV head
  const int total_pages = (len + kPage - 1) / kPage;
  const int n = n_chunks * per_chunk;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int chunk = t / per_chunk;
    const int u = t - chunk * per_chunk;
    const int kv_head = u / n_sub, sub = u - kv_head * n_sub;
    Item it;
    it.k_layer = jb.k_layer;
    it.stream = jb.stream;
    it.n_cons = jb.n_cons;
    it.flags = jb.flags;
#pragma unroll
    for (int x = 0; x < kMaxCons; ++x) {
      it.v_layer[x] = jb.v_layer[x];
      it.q_layer[x] = jb.q_layer[x];
    }
    it.seq_id = static_cast<uint16_t>(sq.seq_id);
    it.seq_idx = static_cast<uint16_t>(si);
    it.head = static_cast<uint16_t>(kv_head * P.group + sub * hpi);
    it.slot = static_cast<uint16_t>(slot_base + chunk);
    const int first = chunk * P.chunk_pages;
    const int np = min(P.chunk_pages, total_pages - first);
    it.first_page = static_cast<uint16_t>(first);
    it.n_pages = static_cast<uint16_t>(np);
    const bool last = (first + np == total_pages);
    if (last) it.flags |= kFlagStreamEnd;
    it.n_valid_last = static_cast<uint16_t>(last ? len - (total_pages - 1) * kPage : kPage);
    it.n_heads = static_cast<uint8_t>(min(hpi, P.group - sub * hpi));
    it.skip_new = jb.skip_new;
    it.pad0 = it.pad1 = 0;
    it.n_pieces = 0;
    P.items[item_base + t] = it;
  }
}

// ------------------------------------------------------------------------------------------
// append: new token's k, v rows and the Q Cache refresh (separate launch on steps with patches)
// ------------------------------------------------------------------------------------------

__global__ void append_kernel(const __grid_constant__ Params P) {
  pdl_wait();
  // what the next kernel does ahead of its own wait reads nothing this kernel writes (an attention
  // worker's early tiles leave out the page that can hold the new token)
  pdl_launch_dependents();
  append_rows(P, P.seqs[blockIdx.x], blockIdx.x, P.layer_begin + blockIdx.y);   // layers of one launch group
}

// ------------------------------------------------------------------------------------------
// plan: where every worker of every statically partitioned launch of the step starts
// ------------------------------------------------------------------------------------------

// Three kinds of threads, by block: one per worker (where it starts), one per CTA (the rows at the
// ends of its stretch) and one per row (its numbers of partials), for every launch of the step.
// All of it is integer arithmetic on the sequence descriptors, which a block keeps in shared memory
// (a search in them would otherwise be five dependent reads for a batch of 32).
constexpr int kPlanBlock = 128;
constexpr int kPlanSeqs = 128;    // descriptors kept in shared memory; longer lists are read from global memory
__global__ void __launch_bounds__(kPlanBlock) plan_kernel(const __grid_constant__ Params P, const __grid_constant__ LaunchList list,
                                                          int cta_blocks) {
  __shared__ StepSeq seqs[kPlanSeqs];
  pdl_wait();   // the page tables and the sequence descriptors are final
  const int g = blockIdx.y;
  const LaunchDesc& L = list.launch[g];
  PartView V = part_view(P, L);
  if (P.n_seqs <= kPlanSeqs) {
    for (int i = threadIdx.x; i < 2 * P.n_seqs; i += kPlanBlock)
      reinterpret_cast<uint4*>(seqs)[i] = reinterpret_cast<const uint4*>(P.seqs)[i];
    __syncthreads();
    V.seqs = seqs;
  }
  // numbers of partial rows that launch G leaves for row (si, u) of `layer`, of the streams it sweeps
  auto count_pieces = [&](const PartView& G, const StepSeq& sq, int si, int u, int layer, int& nv, int& nt) {
    int32_t r0 = seq_base(G, sq.pre_v, sq.pre_t, si) + u * row_tiles(G, sq.len_vis, sq.len_text);
    for (int pos = G.pos_begin; pos < G.pos_end; ++pos) {
      const uint4 raw = __ldg(reinterpret_cast<const uint4*>(G.plan + pos));
      const Job& job = *reinterpret_cast<const Job*>(&raw);
      const int w = job_tiles_per_page(job), pages = pages_of(job.stream ? sq.len_vis : sq.len_text);
      r0 += G.row_cost;
      const int n = pages > 0 ? (r0 + w * (pages - 1)) / G.q - r0 / G.q + 1 : 0;
      for (int x = 0; x < job.n_cons; ++x)
        if (job.v_layer[x] == layer) (job.stream ? nv : nt) = n;
      r0 += w * pages;
    }
  };
  auto row_counts = [&](const StepSeq& sq, int si, int u, int& nv, int& nt) {
    nv = nt = 0;
    int unused;
    count_pieces(V, sq, si, u, L.layer, nv, nt);
    if (L.vis_launch != g) count_pieces(part_view(P, list.launch[L.vis_launch]), sq, si, u, L.layer, nv, unused);
    if (L.text_launch != g) count_pieces(part_view(P, list.launch[L.text_launch]), sq, si, u, L.layer, unused, nt);
  };

  constexpr int kWorkerBlocks = kPlanWorkers / kPlanBlock;
  if (blockIdx.x >= kWorkerBlocks) {
    if (L.layer < 0) return;
    int id = (blockIdx.x - kWorkerBlocks) * kPlanBlock + threadIdx.x;
    if (blockIdx.x >= kWorkerBlocks + cta_blocks) {   // ---- rows
      id -= cta_blocks * kPlanBlock;
      if (id >= P.n_seqs * V.rows) return;
      const int si = id / V.rows, u = id - si * V.rows;
      int nv, nt;
      row_counts(V.seqs[si], si, u, nv, nt);
      P.row_pieces[static_cast<size_t>(g) * P.max_seqs * V.rows + id] = static_cast<uint32_t>(nv) | (static_cast<uint32_t>(nt) << 16);
      return;
    }
    // ---- CTAs
    if (!L.fused_merge || id * L.part_wpc >= L.part_workers) return;
    const int32_t per_cta = L.part_wpc * V.k;
    const int32_t a = id * per_cta * V.q, b = min((id + 1) * per_cta, V.vw) * V.q;   // the CTA's tiles
    CtaDesc d;
    d.pad[0] = d.pad[1] = 0;
    for (int e = 0; e < 2; ++e) {
      EndRow& r = d.end[e];
      int si, u;
      StepSeq sq;
      int32_t r0 = find_row(V, e == 0 ? a : b - 1, si, u, sq);
      (e == 0 ? d.row_first : d.row_last) = si * V.rows + u;
      r.here = r.total = 0;
      for (int pos = V.pos_begin; pos < V.pos_end; ++pos) {
        const uint4 raw = __ldg(reinterpret_cast<const uint4*>(V.plan + pos));
        const Job& job = *reinterpret_cast<const Job*>(&raw);
        const int w = job_tiles_per_page(job), pages = pages_of(job.stream ? sq.len_vis : sq.len_text);
        r0 += V.row_cost;
        auto before = [&](int32_t t) { return t <= r0 ? 0 : min(pages, (t - r0 + w - 1) / w); };   // pages that start before tile t
        r.here += before(b) - before(a);
        r.total += pages;
        r0 += w * pages;
      }
      r.si = si;
      r.head = u;   // (no query groups: a row per query head)
      r.pad = 0;
      r.counter = (L.layer * P.max_seqs + si) * P.hq + u;
      row_counts(sq, si, u, r.nv, r.nt);
    }
    if (d.row_last == d.row_first) d.end[1].here = 0;
    uint4* out = reinterpret_cast<uint4*>(const_cast<CtaDesc*>(P.cdesc) + static_cast<size_t>(g) * kPlanCtas + id);
#pragma unroll
    for (int i = 0; i < 5; ++i) out[i] = reinterpret_cast<const uint4*>(&d)[i];
    return;
  }

  // ---- workers
  const int wid = blockIdx.x * kPlanBlock + threadIdx.x;
  WorkerDesc* out = const_cast<WorkerDesc*>(P.wdesc) + static_cast<size_t>(g) * kPlanWorkers + wid;
  WorkerDesc d;
  d.item[0].n_pages = d.item[1].n_pages = 0;
  RangeCursor c;
  if (wid < L.part_workers && cursor_init(c, V, wid) && cursor_next(c, V, d.item[0])) {
    const Item& it = d.item[0];
    for (int j = 0; j < 2; ++j) {
      const int pg = it.first_page + min(j, it.n_pages - 1);
      d.pids[0][j] = P.table[table_row(P, it.k_layer, it.stream, it.seq_id) + pg];
      for (int x = 0; x < kMaxCons; ++x)
        d.pids[1 + x][j] = x < it.n_cons ? P.table[table_row(P, it.v_layer[x], 2 + it.stream, it.seq_id) + pg] : 0;
    }
    d.pad[0] = d.pad[1] = 0;
    if (!cursor_next(c, V, d.item[1])) d.item[1].n_pages = 0;
    *reinterpret_cast<RangeCursor*>(d.cursor) = c;
  } else {
    d.item[0].n_pages = 0;
  }
  const uint4* src = reinterpret_cast<const uint4*>(&d);
  uint4* dst = reinterpret_cast<uint4*>(out);
  if (d.item[0].n_pages == 0) {   // no work: an all-zero item says so
    dst[0] = make_uint4(0, 0, 0, 0);
    dst[1] = make_uint4(0, 0, 0, 0);
    return;
  }
#pragma unroll
  for (int i = 0; i < 12; ++i) dst[i] = src[i];
}

// ------------------------------------------------------------------------------------------
// prompt rows into pages
// ------------------------------------------------------------------------------------------

// Stores prompt tokens' K/V rows into their pages.  A unit is what one page receives of one run of
// tokens (StoreSeg: up to 16 consecutive tokens of one stream) for one layer, tensor and group of heads: rows
// strided in the caller's tensor, contiguous per head in the page.  A tensor-map copy brings 16 rows into
// shared memory -- 16 tokens of one head, or fewer tokens of more heads where the run is short -- and a bulk
// copy per head writes the valid ones out, so no data passes through registers; a lane of the block's one warp
// owns one buffer and walks its own units.
// The next kernel in the stream may start while this one runs: the prompt's attention reads the
// caller's tensors and pages stored earlier, nothing of what is stored here (it waits for this
// kernel before it ends).  One block per SM (28 KB of shared memory) fits beside two blocks of the
// tcgen05 kernel, and the stores happen while the tensor cores work.
// Per call, rows passing through registers in a launch ahead of the attention -> this: 675 tokens, 32
// layers 451 -> 343 us; 4 352 tokens 5.94 -> 5.47 ms; alone, 32 prompts of 1 120 tokens with 4 heads 1.62 ->
// 0.63 ms, 8 of 3 008 with 32 heads 3.79 -> 3.31 ms (6.8 TB/s).
// Tokens that alternate between text and visual (a run is one token), 32 layers x 32 heads, storing alone / with the
// attention: with 16 rows of one head fetched for every run 0.32 / 1.50 ms at 675 tokens, 1.58 / 7.17 at 3 008; by the
// length of the run 0.17 / 0.57 and 0.55 / 5.31 (through registers 0.17 / 0.65 and 0.56 / 5.74).
constexpr int kStoreLanes = 7;
template <int D>
__global__ void __launch_bounds__(32) prefill_store_kernel(const __grid_constant__ Params P, const __grid_constant__ StoreMaps maps,
                                                           const __grid_constant__ StoreList list) {
  constexpr uint32_t kTile = kPage * D * 2;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[kStoreLanes];
  pdl_launch_dependents();
  const int lane = threadIdx.x;
  if (lane >= kStoreLanes) return;
  mbar_init(&full[lane], 1);
  fence_mbar_init();
  const uint32_t buf = smem_u32(smem) + lane * kTile;
  // units per (layer, tensor): runs of one kind after those of another, groups of heads fastest
  uint32_t before[kStoreKinds + 1];
  before[0] = 0;
#pragma unroll
  for (int i = 0; i < kStoreKinds; ++i)
    before[i + 1] = before[i] + static_cast<uint32_t>(list.first[i + 1] - list.first[i]) * ((P.hkv + (1 << i) - 1) >> i);
  const uint32_t per_tensor = before[kStoreKinds], n_units = per_tensor * P.n_layers * 2, stride = gridDim.x * kStoreLanes;
  struct Unit {
    int32_t head, heads, row, pid, slot, bytes, kind;
    bool value;
  };
  // the lane's next unit at or after u that is stored at all
  auto find = [&](uint32_t& u, Unit& x) -> bool {
    for (; u < n_units; u += stride) {
      const uint32_t b = u / per_tensor, r = u - b * per_tensor, layer = b >> 1;
      int kind = 0;
      uint32_t base = 0;
#pragma unroll
      for (int i = 1; i < kStoreKinds; ++i)
        if (r >= before[i]) kind = i, base = before[i];
      const uint32_t groups = (P.hkv + (1 << kind) - 1) >> kind, run = (r - base) / groups;
      const StoreSeg sg = list.segs[list.first[kind] + run];
      const int stream = sg.ord < 0, ord = sg.ord & 0x7fffffff;
      x.value = b & 1;
      const uint8_t lf = P.layer_flags[layer];
      // K of a lazy layer: visual rows are never kept; text rows only where the mode keeps them
      if (!x.value && !((lf & kLayerWritesQCache) || (stream == 0 && (lf & kLayerOwnsTextK)))) continue;
      x.kind = kind;
      x.head = static_cast<int>(r - base - run * groups) << kind;
      x.heads = min(1 << kind, P.hkv - x.head);
      x.row = layer * list.n_tokens + sg.tok;
      x.pid = P.table[table_row(P, layer, (x.value ? 2 : 0) + stream, sg.seq) + ord / kPage];
      x.slot = ord % kPage;
      x.bytes = sg.n * (D * 2);
      if (static_cast<uint32_t>(x.pid) < static_cast<uint64_t>(P.n_pool_pages)) return true;   // never write outside the pool
      report_error(P.err, P.err_host, kErrBadPage);
    }
    return false;
  };
  uint32_t u = blockIdx.x * kStoreLanes + lane, phase = 0;
  Unit x;
  bool any = find(u, x);
  while (any) {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the buffer's last rows have been read
    mbar_expect_tx(&full[lane], kTile);
    tensor_g2s_3d(buf, x.value ? &maps.v[x.kind] : &maps.k[x.kind], 0, x.row, x.head, &full[lane]);
    const Unit now = x;
    u += stride;
    any = find(u, x);   // (its reads overlap the copy)
    uint32_t done = 0;
    for (uint32_t spin = 0; !done && spin < kSpinLimit; ++spin) done = mbar_try_wait(&full[lane], phase);
    if (!done) {
      report_error(P.err, P.err_host, kErrTimeout);
      // the copy still writes into this block's shared memory: a bounded chance to land
      for (uint32_t spin = 0; !done && spin < kSpinLimit; ++spin) done = mbar_try_wait(&full[lane], phase);
      break;
    }
    phase ^= 1u;
    uint16_t* dst = P.pool + ((static_cast<size_t>(now.pid) * P.hkv + now.head) * kPage + now.slot) * D;
    for (int h = 0; h < now.heads; ++h, dst += kPage * D)
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(buf + h * (kTile >> now.kind)), "r"(now.bytes)
                   : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------------------------------------
// attend: persistent split-KV partial attention, one independent worker per warp
// ------------------------------------------------------------------------------------------

constexpr int kRing = 2;                  // tiles in flight per warp

template <int D>
struct WarpCtx {
  ItemPages ip;
  uint4 qraw[kMaxCons][D / 8];
};

// Start fetching the raw queries of the item in a context slot (asynchronous copies).
template <int D>
__device__ __forceinline__ void begin_queries(WarpCtx<D>& c, const Params& P, int lane) {
  const Item& it = c.ip.item;
  const int nq = (it.flags & kFlagShared) ? 1 : it.n_cons;
  if (lane < D / 8) {
    for (int x = 0; x < nq; ++x) {
      const bool cached = (it.flags >> (kFlagCachedShift + x)) & 1;
      const uint16_t* src =
          cached ? P.qcache + ((static_cast<size_t>(it.q_layer[x]) * P.max_seqs + it.seq_id) * P.hq + it.head) * D
                 : P.q + ((static_cast<size_t>(it.q_layer[x]) * P.n_seqs + it.seq_idx) * P.hq + it.head) * D;
      cp_async_16(&c.qraw[x][lane], reinterpret_cast<const uint4*>(src) + lane);
    }
  }
}

// One item: NQ queries score the K tiles, NV value streams are accumulated.
// NQ == 1: every consumer shares the weights; NQ == NV: consumer x has its own query.
// MODE 1 (one query, one consumer) also stores the scaled scores in the logit cache; MODE 2 takes
// them from there instead of reading K tiles (the ring then carries V tiles only).
// SKIP (shared weights only): the consumers named in the item's skip_new mask leave out the
// stream's last key -- the step's new token, whose value row of a follower does not exist yet when
// its leader's launch runs (Eq. 6: V = [cached V, new v]); they get their own sum of weights.
// FOLD: the item may end its layer's text stream under the folded append (the new token's rows come
// from the step's inputs).  Launches without the folded append use the instantiation without it,
// whose page loop then carries none of this (with it in every instantiation the one-launch step was
// 3.5 % slower); under the folded append every single-consumer item of a launch takes this one
// (sending only the items that end a stream here made the workers alternate between two copies of
// the loop: 1.20 against 1.09 ms per step at config 2).
template <int D, int NQ, int NV, int MODE = 0, bool SKIP = false, bool FOLD = false>
__device__ __forceinline__ void process_item(WorkerState& st, const WarpCtx<D>* ctx, uint32_t ring, uint64_t* full,
                                             const Params& P, int lane) {
  auto ctx_of = [ctx](int k) -> const ItemPages& { return ctx[k % kCtxSlots].ip; };
  constexpr int EP2 = D / 16;   // element pairs of a row held by one lane
  constexpr int LPR = D / 64;   // 16-byte loads per lane per row
  const WarpCtx<D>& c = ctx[st.cons_k % kCtxSlots];
  const int kg = lane >> 3;     // which of 4 keys of a pass
  const int c8 = lane & 7;      // which 16-byte chunk of the row (and of its second half)
  const uint32_t lane_off = kg * (D * 2) + c8 * 16;   // this lane's first chunk of a pass's rows

  // The arithmetic on elements runs on pairs (fma.rn.f32x2): half the instructions, same fp32 results.
  float2 qf[NQ][EP2];
#pragma unroll
  for (int x = 0; x < NQ; ++x) {
#pragma unroll
    for (int j = 0; j < LPR; ++j) {
      const uint4 raw = c.qraw[x][c8 + 8 * j];
      bf16x8_to_f32x2(raw, &qf[x][4 * j]);
    }
#pragma unroll
    for (int e = 0; e < EP2; ++e) qf[x][e] = mul2(qf[x][e], make_float2(P.scale_log2, P.scale_log2));
  }

  float m[NQ], l[NQ];
  float2 acc[NV][EP2];
#pragma unroll
  for (int x = 0; x < NQ; ++x) {
    m[x] = -INFINITY;
    l[x] = 0.f;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int e = 0; e < EP2; ++e) acc[v][e] = make_float2(0.f, 0.f);

  const int n_pages = c.ip.item.n_pages;
  const int n_valid_last = c.ip.item.n_valid_last;
  // SKIP: the new token is key n_valid_last - 1 of the item's last page when that page ends the stream
  const bool skip_here = SKIP && (c.ip.item.flags & kFlagStreamEnd);
  const uint32_t skip_mask = SKIP ? c.ip.item.skip_new : 0u;
  float l_skip = 0.f;       // sum of weights without the new token
  float* lg = nullptr;      // this item's first key in the logit cache
  float lg_next[4] = {0.f, 0.f, 0.f, 0.f};
  if (MODE != 0) {
    lg = logit_row(P, c.ip.item.stream, c.ip.item.seq_id, c.ip.item.head) + c.ip.item.first_page * kPage;
    if (MODE == 2) {
#pragma unroll
      for (int i = 0; i < 4; ++i) lg_next[i] = lg[4 * i + kg];
    }
  }

  constexpr bool kMayFold = FOLD || SKIP;
  const int new_pg = (kMayFold && holds_new_token(P, c.ip.item, n_pages - 1)) ? n_pages - 1 : -1;   // folded append: page of the new token
  float p[NQ][4];
  for (int pg = 0; pg < n_pages && !st.dead; ++pg) {
    const int nvalid = (pg == n_pages - 1) ? n_valid_last : kPage;
    // softmax step of the page's 16 scores
    auto weigh = [&]() {
#pragma unroll
      for (int x = 0; x < NQ; ++x) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float s = p[x][i];
          if (MODE != 2) {
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 4);
          }
          if (MODE == 1 && c8 == 0 && 4 * i + kg < nvalid) lg[pg * kPage + 4 * i + kg] = s;
          p[x][i] = (4 * i + kg < nvalid) ? s : -INFINITY;
        }
        float tmax = fmaxf(fmaxf(p[x][0], p[x][1]), fmaxf(p[x][2], p[x][3]));
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 8));
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 16));
        const float m_new = fmaxf(m[x], tmax);
        const float corr = ex2_approx(m[x] - m_new);
        float psum = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          p[x][i] = ex2_approx(p[x][i] - m_new);
          psum += p[x][i];
        }
        l[x] = l[x] * corr + psum;
        if (SKIP) {
          float psum_skip = psum;
          if (skip_here && pg == n_pages - 1) {
            const int r_new = nvalid - 1;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (4 * i + kg == r_new) psum_skip -= p[x][i];
          }
          l_skip = l_skip * corr + psum_skip;
        }
        m[x] = m_new;
        if (corr != 1.f) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            if (NQ == 1 || v == x) {
#pragma unroll
              for (int e = 0; e < EP2; ++e) acc[v][e] = mul2(acc[v][e], make_float2(corr, corr));
            }
          }
        }
      }
    };
    auto score = [&](uint32_t tile) {   // K tile: scores of 16 keys
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float2 kf[EP2];
#pragma unroll
        for (int j = 0; j < LPR; ++j) bf16x8_to_f32x2(lds128(tile + lane_off + i * (4 * D * 2) + j * 128), &kf[4 * j]);
#pragma unroll
        for (int x = 0; x < NQ; ++x) {
          float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
#pragma unroll
          for (int e = 0; e < EP2; e += 2) {
            a0 = fma2(kf[e], qf[x][e], a0);
            a1 = fma2(kf[e + 1], qf[x][e + 1], a1);
          }
          p[x][i] = (a0.x + a1.x) + (a0.y + a1.y);
        }
      }
    };
    auto add = [&](uint32_t tile, int v) {   // V tile: weighted sum for consumer v (a constant after unrolling)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float2 vf[EP2];
#pragma unroll
        for (int j = 0; j < LPR; ++j) bf16x8_to_f32x2(lds128(tile + lane_off + i * (4 * D * 2) + j * 128), &vf[4 * j]);
        const float pv = p[NQ == 1 ? 0 : v][i];
#pragma unroll
        for (int e = 0; e < EP2; ++e) acc[v][e] = fma2(vf[e], make_float2(pv, pv), acc[v][e]);
      }
    };
    auto clear_tail = [&](uint32_t tile, int n) {
      // rows past the end hold whatever the pool held (a zero weight does not cancel a NaN): cleared
      for (int r = n * (D / 8) + lane; r < kPage * (D / 8); r += 32) sts128(tile + r * 16, make_uint4(0u, 0u, 0u, 0u));
      fence_proxy_async();   // these generic-proxy writes precede the slot's next asynchronous refill
      __syncwarp();
    };
    if constexpr (NQ > 1) {
      uint32_t tile = wait_tile<D>(st, ring, full, P, lane);
      if (st.dead) break;
      score(tile);
      release_tile<kRing>(st);
      fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
      weigh();
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        tile = wait_tile<D>(st, ring, full, P, lane);
        if (st.dead) break;
        if (nvalid < kPage) clear_tail(tile, nvalid);
        add(tile, v);
        release_tile<kRing>(st);
        fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
      }
      continue;
    }
    if (MODE == 2) {
      // ---- scores of 16 keys from the logit cache; the next page's are requested now
#pragma unroll
      for (int i = 0; i < 4; ++i) p[0][i] = lg_next[i];
      if (pg + 1 < n_pages) {
#pragma unroll
        for (int i = 0; i < 4; ++i) lg_next[i] = lg[(pg + 1) * kPage + 4 * i + kg];
      }
    }
    // The page's tiles, K (t = 0) and then one V tile per consumer.  Workers that go from a row's
    // visual to its text stream go from one copy of this loop to another, and an SM's twelve are all
    // somewhere else, so with short rows the size of the code is what a launch waits for: a page that
    // is not full has no loop of its own (30 sequences of 260 tokens, 16 heads, 20.0 -> 19.4 us a layer).  Left
    // rolled up the loop is smaller still, but its branches cost more: 17.9 against 17.6 us there, batch 16 31.1
    // / 30.3, one-launch steps of 2 short sequences with 64-wide heads 2.21 / 2.05.
#pragma unroll
    for (int t = MODE == 2 ? 1 : 0; t <= NV; ++t) {
      if (t == 1) weigh();
      const uint32_t tile = wait_tile<D>(st, ring, full, P, lane);
      if (st.dead) break;
      const int skips = (SKIP && t > 0 && skip_here && pg == n_pages - 1) ? static_cast<int>((skip_mask >> (t - 1)) & 1u) : 0;
      if (kMayFold && pg == new_pg && !skips) {
        // the new token's row comes from the step's input: into the tile, and into the pool for later steps
        const Item& it = c.ip.item;
        if (lane < D / 8) {
          const uint4 val = t == 0 ? c.ip.new_k[lane]
                            : t - 1 == first_taker(it)
                                ? c.ip.new_v[lane]
                                : reinterpret_cast<const uint4*>(
                                      P.v + ((static_cast<size_t>(it.v_layer[t - 1]) * P.n_seqs + it.seq_idx) * P.hkv + c.ip.kv_head) * D)[lane];
          sts128(tile + (nvalid - 1) * (D * 2) + lane * 16, val);
          const int pid = c.ip.pages[t][pg];
          if (static_cast<uint32_t>(pid) < static_cast<uint64_t>(P.n_pool_pages))
            reinterpret_cast<uint4*>(P.pool + ((static_cast<size_t>(pid) * P.hkv + c.ip.kv_head) * kPage + (nvalid - 1)) * D)[lane] = val;
          // an ordinary layer's query goes to the Q Cache
          if (t == 0 && it.q_layer[0] == it.k_layer && !((it.flags >> kFlagCachedShift) & 1) &&
              (P.layer_flags[it.k_layer] & kLayerWritesQCache))
            reinterpret_cast<uint4*>(P.qcache + ((static_cast<size_t>(it.k_layer) * P.max_seqs + it.seq_id) * P.hq + it.head) * D)[lane] =
                c.qraw[0][lane];
        }
        fence_proxy_async();   // these generic-proxy writes precede the slot's next asynchronous refill
        __syncwarp();
      }
      if (t == 0) {
        score(tile);
      } else {
        if (nvalid - skips < kPage) clear_tail(tile, nvalid - skips);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (t == v + 1) add(tile, v);
      }
      release_tile<kRing>(st);
      fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
    }
  }
  if (st.dead) return;

  // ---- partial results: sum over the 4 key groups, then lanes 0..7 store
#pragma unroll
  for (int x = 0; x < NQ; ++x) {
    l[x] += __shfl_xor_sync(0xffffffffu, l[x], 8);
    l[x] += __shfl_xor_sync(0xffffffffu, l[x], 16);
  }
  if (SKIP) {
    l_skip += __shfl_xor_sync(0xffffffffu, l_skip, 8);
    l_skip += __shfl_xor_sync(0xffffffffu, l_skip, 16);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
#pragma unroll
    for (int e = 0; e < EP2; ++e) {
      acc[v][e].x += __shfl_xor_sync(0xffffffffu, acc[v][e].x, 8);
      acc[v][e].y += __shfl_xor_sync(0xffffffffu, acc[v][e].y, 8);
      acc[v][e].x += __shfl_xor_sync(0xffffffffu, acc[v][e].x, 16);
      acc[v][e].y += __shfl_xor_sync(0xffffffffu, acc[v][e].y, 16);
    }
  }
  if (kg == 0) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const size_t row =
          ((static_cast<size_t>(c.ip.item.v_layer[v]) * P.max_seqs + c.ip.item.seq_idx) * P.max_slots + c.ip.item.slot) *
              P.hq + c.ip.item.head;
      float* dst = P.part_acc + row * D;
#pragma unroll
      for (int j = 0; j < LPR; ++j) {
        float4* d4 = reinterpret_cast<float4*>(dst + 64 * j + 8 * c8);
        d4[0] = make_float4(acc[v][4 * j + 0].x, acc[v][4 * j + 0].y, acc[v][4 * j + 1].x, acc[v][4 * j + 1].y);
        d4[1] = make_float4(acc[v][4 * j + 2].x, acc[v][4 * j + 2].y, acc[v][4 * j + 3].x, acc[v][4 * j + 3].y);
      }
      const bool skipping = SKIP && ((skip_mask >> v) & 1u);
      if (c8 == 0) P.part_ml[row] = make_float2(m[NQ == 1 ? 0 : v], skipping ? l_skip : l[NQ == 1 ? 0 : v]);
    }
  }
}

// A worker's life: take items (claimed from the list, or the pieces of its static ranges), keep
// the tile ring full across item boundaries, process each item.  While item k is processed the
// ring already fetches tiles of item k + 1 and the context of item k + 2 (descriptor, page ids,
// queries) arrives by asynchronous copies.
// False if a wait ran out.
// OWN: launches with sweeps that score with a query per consumer.  Those sweeps hold up to four queries and
// four accumulators; in a kernel of their own they do not cost the others registers (with both in one, items in local
// memory and all of the L1 given to tiles -> now, us per layer: batch 1 10.5 -> 9.7, batch 16 32.7 -> 31.6, 30 short
// sequences 19.3 -> 17.9; own-query sweeps of four, 12 sequences of 800 keys, 28.4 -> 25.0).
template <int D, bool STATIC, bool OWN>
__device__ __forceinline__ bool attend_worker(const Params& P, WarpCtx<D>* ctx, uint32_t ring, uint64_t* full,
                                              RangeCursor* cursor, int32_t* stage, CtaDesc* cta, int wid, int lane) {
  auto ctx_of = [ctx](int k) -> const ItemPages& { return ctx[k % kCtxSlots].ip; };
  WorkerState st;
  worker_init(st, 0);
  st.drop_next = P.debug_drop_tile != 0;   // (test hook)
  int issued = 0;
  auto take = [&](ItemPages& slot) -> bool {   // the next item into a context slot
    if (STATIC) return cursor_step(cursor, P, slot, lane);
    const int idx = claim_take(P, issued);
    if (idx < 0) return false;
    load_item(slot, P, idx, lane);
    return true;
  };
  // ---- ahead of the wait for the previous kernel: the first two items and their page ids (from the
  // launch plan, the step descriptors and the page tables, all written before that kernel
  // started), and the first tiles unless they could hold a new token that an earlier launch of the
  // step stores (with the folded append the worker patches the new token's row itself).  After it,
  // only the layer's inputs.
  bool more;
  if (STATIC) {
    if (P.follows_setup) pdl_wait();   // (a step's first launch: the plan or the descriptors are the previous kernel's)
    bool any = wid >= 0 && wid < P.part_workers;
    if (P.wdesc != nullptr) {
      // planned ahead: one read gives the first two items, the first page ids and the cursor
      any = any && load_worker_desc(P, wid, ctx[0].ip, ctx[1].ip, cursor, stage, cta, lane);
    } else {
      RangeCursor c;
      any = any && cursor_init(c, part_view(P), wid);
      if (lane == 0) *cursor = c;
      __syncwarp();
      any = any && take(ctx[0].ip);
      if (any) {
        begin_item_pages(ctx[0].ip, P, lane);
        cp_async_wait_all();
        __syncwarp();
      }
    }
    if (!any) {
      pdl_wait();   // (a warp without work may still merge)
      return true;
    }
    st.n_my = 1;
    const Item& first = ctx[0].ip.item;
    const bool early_tiles = P.fold_append || !(first.stream == 0 && (first.flags & kFlagStreamEnd) && first.n_pages <= kRing);
    if (early_tiles) fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
    if (P.wdesc != nullptr) {
      if (first.n_pages > 2) begin_item_pages(ctx[0].ip, P, lane);   // the whole page list, while the tiles fly
      more = ctx[1].ip.item.n_pages > 0;
    } else {
      more = take(ctx[1].ip);
    }
    if (more) begin_item_pages(ctx[1].ip, P, lane);
    pdl_wait();
    pdl_launch_dependents();
  } else {
    pdl_wait();   // the item list and the work counter are the previous kernel's
    pdl_launch_dependents();
    issued = claim_issue(P, lane);
    if (!take(ctx[0].ip)) return true;
    begin_item_pages(ctx[0].ip, P, lane);
    cp_async_wait_all();
    __syncwarp();
    st.n_my = 1;
    fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
    issued = claim_issue(P, lane);
  }
  begin_queries<D>(ctx[0], P, lane);
  begin_new_rows(ctx[0].ip, P, lane, D);
  if (!STATIC) {
    more = take(ctx[1].ip);
    if (more) begin_item_pages(ctx[1].ip, P, lane);
  }
  cp_async_commit_group();
  if (more) {
    begin_queries<D>(ctx[1], P, lane);
    begin_new_rows(ctx[1].ip, P, lane, D);
  }
  cp_async_commit_group();   // the second item's inputs are waited for when the first item is done
  if (STATIC) cp_async_wait_group<1>();
  else cp_async_wait_all();
  __syncwarp();
  if (more) st.n_my = 2;
  fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
  bool pending = false;   // a context is being filled for item st.n_my
  if (!STATIC && more) issued = claim_issue(P, lane);

  for (int k = 0; k < st.n_my && !st.dead; ++k) {
    const Item& cur = ctx[k % kCtxSlots].ip.item;
    const int nc = cur.n_cons;
    if (more) {
      // the third slot is free (it held the item before this one): start filling it with the item after next
      WarpCtx<D>& next = ctx[(k + 2) % kCtxSlots];
      more = take(next.ip);
      if (more) {
        begin_item_pages(next.ip, P, lane);
        begin_queries<D>(next, P, lane);
        begin_new_rows(next.ip, P, lane, D);
        pending = true;
      }
    }
    if constexpr (OWN) {
      if (nc == 1) process_item<D, 1, 1>(st, ctx, ring, full, P, lane);
      else if (nc == 2) process_item<D, 2, 2>(st, ctx, ring, full, P, lane);
      else if (nc == 3) process_item<D, 3, 3>(st, ctx, ring, full, P, lane);
      else process_item<D, 4, 4>(st, ctx, ring, full, P, lane);
    } else if (nc == 1 && (cur.flags & kFlagReadLogits)) process_item<D, 1, 1, 2>(st, ctx, ring, full, P, lane);
    else if (nc == 1 && (cur.flags & kFlagWriteLogits)) process_item<D, 1, 1, 1>(st, ctx, ring, full, P, lane);
    else if (P.any_skip) {   // (one copy of the loop per launch here too: GLA blocks of short rows 16.4 -> 14.8 us a layer)
      if (nc == 1) process_item<D, 1, 1, 0, true>(st, ctx, ring, full, P, lane);
      else if (nc == 2) process_item<D, 1, 2, 0, true>(st, ctx, ring, full, P, lane);
      else if (nc == 3) process_item<D, 1, 3, 0, true>(st, ctx, ring, full, P, lane);
      else process_item<D, 1, 4, 0, true>(st, ctx, ring, full, P, lane);
    }
    else if (nc == 1 && P.fold_append) process_item<D, 1, 1, 0, false, true>(st, ctx, ring, full, P, lane);   // (one code path per launch)
    else if (nc == 1) process_item<D, 1, 1>(st, ctx, ring, full, P, lane);
    else if (nc == 2) process_item<D, 1, 2>(st, ctx, ring, full, P, lane);
    else if (nc == 3) process_item<D, 1, 3>(st, ctx, ring, full, P, lane);
    else process_item<D, 1, 4>(st, ctx, ring, full, P, lane);
    if (st.dead) break;
    if (!STATIC && more) issued = claim_issue(P, lane);   // (not held across the page loops, which need the registers)
    if (STATIC) record_row_slots(P, cur, lane);
    if (k + 1 < st.n_my) {   // the contexts of items k + 1 and k + 2 have had this item's time to arrive
      cp_async_wait_all();
      __syncwarp();
      if (pending) st.n_my = k + 3;
      pending = false;
    }
    st.cons_k = k + 1;
    fill_ring<D, kRing, false>(st, ctx_of, ring, full, P, lane);
  }
  if (st.dead) {
    cp_async_wait_all();
    drain_ring<kRing>(st, full, P.debug_drop_tile ? kDebugSpinLimit : kSpinLimit);
  }
  return !st.dead;
}

template <int D, bool STATIC, bool OWN>
__global__ void __launch_bounds__(kThreads, kAttendCtasPerSm) attend_kernel(const __grid_constant__ Params P) {
  constexpr uint32_t kTile = kPage * D * 2;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full_all[kWarps][kRing];
  __shared__ __align__(16) RangeCursor cursors[kWarps];
  __shared__ __align__(16) int32_t stages[kWarps][12];
  __shared__ __align__(16) FinishSmem<D> finish;
  __shared__ CtaDesc cta;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ring = smem_u32(smem) + static_cast<uint32_t>(warp) * kRing * kTile;
  WarpCtx<D>* ctx = reinterpret_cast<WarpCtx<D>*>(smem + static_cast<size_t>(kWarps) * kRing * kTile) + warp * kCtxSlots;
  uint64_t* full = full_all[warp];

  if (lane == 0) {
    for (int s = 0; s < kRing; ++s) mbar_init(&full[s], 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) finish.dead = 0;
  __syncthreads();

  const bool ok = attend_worker<D, STATIC, OWN>(P, ctx, ring, full, &cursors[warp], stages[warp], &cta, worker_index(P, warp), lane);
  if (STATIC) finish_cta<D>(P, finish, cta, !ok, warp, lane);
}

// ------------------------------------------------------------------------------------------
// merge: log-sum-exp combination of the partials of one (layer, sequence, head) per warp
// ------------------------------------------------------------------------------------------

// One warp per (layer, sequence, head).  What it reads besides the partials (the sequence's
// descriptor, the numbers of partials where they are planned, page ids) was written when the step
// began and is read ahead of the wait for the attention kernel, so that one round of reads is left.
template <int D, bool ROWS>
__global__ void merge_kernel(const __grid_constant__ Params P) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_layers = P.layer_end - P.layer_begin;
  const int idx = blockIdx.x * (blockDim.x >> 5) + warp;
  if (idx >= n_layers * P.n_seqs * P.hq) {
    pdl_wait();
    return;
  }
  merge_row<D, ROWS>(P, P.layer_begin + idx / (P.hq * P.n_seqs), (idx / P.hq) % P.n_seqs, idx % P.hq, lane);
}

template <int D>
constexpr int attend_smem_bytes() {
  return kWarps * kRing * kPage * D * 2 + kWarps * kCtxSlots * static_cast<int>(sizeof(WarpCtx<D>));
}

}  // namespace

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------

namespace {
// Shared memory for as many blocks as an SM holds of the kernel, and no more: the rest is L1 cache.
template <typename K>
cudaError_t configure_attend(K kernel, int smem) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes a;
  e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  const int need = kAttendCtasPerSm * (smem + static_cast<int>(a.sharedSizeBytes) + 1024), all = 228 * 1024;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, min(100, (100 * need + all - 1) / all));
}
}  // namespace

cudaError_t configure_kernels(int* attend_smem) {
  cudaError_t e = configure_attend(attend_kernel<128, false, false>, attend_smem_bytes<128>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<128, false, true>, attend_smem_bytes<128>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<128, true, false>, attend_smem_bytes<128>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<128, true, true>, attend_smem_bytes<128>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<64, false, false>, attend_smem_bytes<64>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<64, false, true>, attend_smem_bytes<64>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<64, true, false>, attend_smem_bytes<64>());
  if (e == cudaSuccess) e = configure_attend(attend_kernel<64, true, true>, attend_smem_bytes<64>());
  if (attend_smem) *attend_smem = attend_smem_bytes<128>();
  return e;
}

cudaError_t launch_setup(const Params& p, const StepInline* inl, cudaStream_t stream) {
  constexpr int kBlock = 256;
  const int n_house = (max(max(p.n_patches, p.n_layers), p.n_seqs * 8) + kBlock - 1) / kBlock;
  const int blocks = p.n_pos * p.n_seqs + n_house + (p.fused_append ? p.n_seqs * p.n_layers : 0);
  static const StepInline kNone{};
  return launch_pdl(setup_kernel, dim3(blocks), dim3(kBlock), 0, stream, p, inl ? *inl : kNone);
}

cudaError_t launch_plan(const Params& p, const LaunchList& list, int n_launches, cudaStream_t stream) {
  if (n_launches <= 0) return cudaSuccess;
  int ctas = 0;
  bool rows = false;
  for (int g = 0; g < n_launches; ++g) {
    const LaunchDesc& l = list.launch[g];
    if (l.fused_merge) ctas = max(ctas, (l.part_workers + l.part_wpc - 1) / l.part_wpc);
    rows = rows || l.layer >= 0;
  }
  const int cta_blocks = (ctas + kPlanBlock - 1) / kPlanBlock;
  const int row_blocks = rows ? (p.n_seqs * p.heads_per_item_dim + kPlanBlock - 1) / kPlanBlock : 0;
  return launch_pdl(plan_kernel, dim3(kPlanWorkers / kPlanBlock + cta_blocks + row_blocks, n_launches), dim3(kPlanBlock), 0, stream, p,
                    list, cta_blocks);
}

cudaError_t launch_append(const Params& p, cudaStream_t stream) {
  dim3 grid(p.n_seqs, p.layer_end - p.layer_begin);
  return launch_pdl(append_kernel, grid, dim3(128), 0, stream, p);
}

cudaError_t launch_attend(const Params& p, int n_sms, cudaStream_t stream) {
  const int n_items = p.item_end - p.item_begin;
  if (!p.part_static && n_items <= 0) return cudaSuccess;
  const int grid = p.part_static ? (p.part_workers + p.part_wpc - 1) / p.part_wpc
                                 : min(n_sms * kAttendCtasPerSm, (n_items + kWarps - 1) / kWarps);
  auto launch = [&](auto kernel, int smem) { return launch_pdl(kernel, dim3(grid), dim3(kThreads), smem, stream, p); };
  if (p.d == 128) {
    const int smem = attend_smem_bytes<128>();
    if (p.part_static) return p.any_own ? launch(attend_kernel<128, true, true>, smem) : launch(attend_kernel<128, true, false>, smem);
    return p.any_own ? launch(attend_kernel<128, false, true>, smem) : launch(attend_kernel<128, false, false>, smem);
  }
  const int smem = attend_smem_bytes<64>();
  if (p.part_static) return p.any_own ? launch(attend_kernel<64, true, true>, smem) : launch(attend_kernel<64, true, false>, smem);
  return p.any_own ? launch(attend_kernel<64, false, true>, smem) : launch(attend_kernel<64, false, false>, smem);
}

cudaError_t launch_merge(const Params& p, cudaStream_t stream) {
  const int n = (p.layer_end - p.layer_begin) * p.n_seqs * p.hq;
  if (n <= 0) return cudaSuccess;
  const int warps_per_block = 8;
  const int blocks = (n + warps_per_block - 1) / warps_per_block;
  const dim3 grid(blocks), block(warps_per_block * 32);
  if (p.d == 128)
    return p.row_cluster > 0 ? launch_pdl(merge_kernel<128, true>, grid, block, 0, stream, p)
                             : launch_pdl(merge_kernel<128, false>, grid, block, 0, stream, p);
  return p.row_cluster > 0 ? launch_pdl(merge_kernel<64, true>, grid, block, 0, stream, p)
                           : launch_pdl(merge_kernel<64, false>, grid, block, 0, stream, p);
}

cudaError_t launch_prefill_store(const Params& p, const StoreMaps& maps, const StoreList& list, int blocks, cudaStream_t stream) {
  if (list.first[kStoreKinds] <= 0) return cudaSuccess;
  const int smem = kStoreLanes * kPage * p.d * 2;
  if (p.d == 128) prefill_store_kernel<128><<<blocks, 32, smem, stream>>>(p, maps, list);
  else prefill_store_kernel<64><<<blocks, 32, smem, stream>>>(p, maps, list);
  return cudaGetLastError();
}

}  // namespace qc
