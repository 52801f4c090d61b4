// Attention of one layer (in-order schedule) where every output row has thread blocks of its own.
//
// A launch of one layer for a small batch moves a few MB, which HBM delivers in 2 us, and what it costs is its
// chain of dependent steps; a launch for a large batch is bound by HBM and loses at its end what that chain
// takes.  Cut into tile ranges (qc_kernels.cu, qc_attend_tc.cu) the chain is: a worker's page, its partial row
// through the L2, an atomic per shared row, the partials of 40 workers read back by one CTA (or a merge
// launch).  Here a row (a query head, or a query group) belongs to a cluster of up to eight CTAs, or to one
// CTA, whose warps take its pages in turn -- all visual pages, then all text pages -- and the warps' sums are
// added in shared memory: first in each CTA, then over the cluster through distributed shared memory.  The
// launch writes finished rows; the only sums that reach HBM are one per row and follower of a lazy block (the
// sums of the keys it shares with its leader).  No plan, no counters, no merge launch, and every row is added
// up in one order.
// us per layer, tile ranges -> this: one sequence of 675 tokens, 32 heads 9.5 -> 6.9; 16 of them 30.8 -> 26.9;
// 32 of 500 44.9 -> 40.5; 32 of 1 120 with 4 KV heads 20.2 -> 17.7.  After the wait for the previous kernel the
// first of these spends, of some 12 000 cycles, 850 on the query, 2 300 on the first K tile and its softmax,
// 1 900 on the V tiles, as much on a second page, and 2 500 from the last page to the row.
//
// Every launch of the in-order schedule scores with one query per row (its layer's own), so one running softmax
// serves the row's streams: consumer 0 is the layer itself, consumers 1 .. are the followers whose cached V the
// leader's launch also weights.  Under VLA_QC those take no text keys: their softmax reference stays where the
// visual pages left it.
//
// One query head per KV head: fp32 arithmetic on pairs.  Query groups: mma.m16n8k16 with keys as M and the
// group as N, as in qc_attend_tc.cu, but with the weights as the sum of two bf16 values, a product each on the
// same V fragment (error against 64 bits, 32 sequences of 1 120 tokens: 2.05e-3 in tile ranges, 2.11e-3 here
// with one bf16 value -- fewer, longer pieces have fewer weights that are exactly 1 -- and 1.66e-3, the
// rounding of the output, with two; 17.9 us a layer with one, 17.7 with two and a single tensor-map copy per
// tile).

#include "qc_device.cuh"

#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

namespace qc {
namespace {

// Warps per CTA (W): six, or fewer where rows are many; an SM holds twelve in all (64-wide heads sixteen).  Tiles in
// flight per warp (RING): four where the next launch's first tiles are to land during this one; two where the
// launch is bound by HBM, which scattered tiles use worse the more there are in flight (512 rows of 43 pages, 3 warps:
// 27.5 us a layer with four, 27.0 with two); three for blocks of one warp (two, three, four: 1 024 rows of 19 pages 26.4,
// 25.9, 25.7; 1 110 of 38 46.5, 45.5, 46.3; 1 440 of 38 57.9, 59.0, 59.7).

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {   // the same place in another CTA's shared memory
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 peer_load4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 peer_load2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ int32_t peer_load_s32(uint32_t addr) {
  int32_t v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// Byte offset of 16-byte chunk `chunk` of row `row` in a tile: linear (MH), or as the tensor map's
// 128-byte swizzle leaves it.
template <int D, bool MH>
__device__ __forceinline__ uint32_t tile_at(int row, int chunk) {
  if (MH) return row * (D * 2) + (chunk << 4);
  if (D == 128) return ((chunk >> 3) << 11) + (row << 7) + (((chunk & 7) ^ (row & 7)) << 4);
  return (row << 7) + ((chunk ^ (row & 7)) << 4);
}

template <bool MH>
constexpr int kRowHeads = MH ? 1 : 8;          // heads of a row, padded
template <int D, bool MH, int NV>
constexpr int kRowStride = D + (MH || NV == 4 ? 0 : 4);   // floats from one head's sums to the next one's (bank conflicts, where there is room)

// What the CTA keeps of the row besides the tiles.
template <int D, bool MH, int NV, int W, int RING>
struct __align__(16) RowSmem {
  float red[NV][kRowHeads<MH>][D];                  // the CTA's sums
  float2 red_ml[NV > 1 ? 2 : 1][kRowHeads<MH>];     // and their (reference, sum of weights): own, followers'
  float2 ml[NV > 1 ? 2 : 1][kRowHeads<MH>][W];
  float weight[NV > 1 ? 2 : 1][kRowHeads<MH>][W + 2];   // of the warps' sums in the CTA's
  uint4 new_k[D / 8], new_v[D / 8];                 // the new token's rows (for the one warp that sweeps it)
  int32_t pages[W][1 + NV][32];             // page ids of a warp's next pages: K, V of each consumer
  uint64_t full[W][RING];
  int32_t dead;
};

template <int D, bool MH, int NV, int W, int RING>
__global__ void __launch_bounds__(W * 32, 12 / W) attend_rows_kernel(const __grid_constant__ Params P, const __grid_constant__ RowJobs J) {
  constexpr uint32_t kTile = kPage * D * 2;
  constexpr int KS = D / 16;
  constexpr int NH = MH ? 1 : 2;       // heads whose softmax a lane follows (query groups: columns 2t, 2t + 1)
  constexpr int EP2 = D / 16;          // MH: element pairs of a row held by one lane
  constexpr int LPR = D / 64;          // MH: 16-byte loads per lane per row
  constexpr int NC = NV > 1 ? 2 : 1;   // running softmaxes: the layer's own, its followers'
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;   // swizzled tiles sit on 1024-byte boundaries
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  using Smem = RowSmem<D, MH, NV, W, RING>;
  Smem& S = *reinterpret_cast<Smem*>(base_ptr + W * RING * kTile);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = cluster_rank(), n_ctas = cluster_size();
  const uint32_t ring = base + static_cast<uint32_t>(warp) * RING * kTile;
  uint64_t* full = S.full[warp];
  if (lane == 0) {
    for (int s = 0; s < RING; ++s) mbar_init(&full[s], 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) S.dead = 0;

  // ---- ahead of the wait for the previous kernel: the row, its page ids and the first tiles.  The sequence
  // descriptors, the page tables and the cached pages were written two or more launches back, but for a step's
  // first launch, which comes right after the one that writes the first two (its wait is 1 us of the 227 of a
  // step of 32 layers).
  if (P.follows_setup) pdl_wait();
  const int row = blockIdx.x / n_ctas, rows = P.heads_per_item_dim;
  const int si = row / rows, u = row - si * rows;
  const uint4 sq = *reinterpret_cast<const uint4*>(P.seqs + si);
  const int seq_id = sq.x, len_text = sq.y, len_vis = sq.z;
  const int hpi = P.heads_per_item, n_sub = (P.group + hpi - 1) / hpi, kv_head = u / n_sub, sub = u - kv_head * n_sub;
  const int head = kv_head * P.group + sub * hpi, n_heads = min(hpi, P.group - sub * hpi);
  const int n_vis = J.has_vis ? pages_of(len_vis) : 0, n_text = J.has_text ? pages_of(len_text) : 0;
  const int total = n_vis + n_text, step = n_ctas * W, first = rank * W + warp;
  const int n_my = total > first ? (total - first + step - 1) / step : 0;               // pages first, first + step, ...
  const int j_text = n_vis > first ? (n_vis - first + step - 1) / step : 0;             // the first of them that is a text page
  const int vis_cons = J.vis.n_cons, text_cons = J.text.n_cons;
  bool dead = false;
  const uint64_t policy = l2_evict_first_policy();

  auto load_pages = [&](int j0) {   // ids of pages j0 .. j0 + 31 of this warp
    __syncwarp();
    const int j = j0 + lane;
    if (j < n_my) {
      const bool vis = j < j_text;
      const Job& job = vis ? J.vis : J.text;
      const int pg = first + j * step - (vis ? 0 : n_vis);
      for (int t = 0; t <= job.n_cons; ++t) {
        int pid = P.table[table_row(P, t == 0 ? job.k_layer : job.v_layer[t - 1], (t == 0 ? 0 : 2) + (vis ? 1 : 0), seq_id) + pg];
        if (static_cast<uint32_t>(pid) >= static_cast<uint64_t>(P.n_pool_pages)) {   // never read outside the pool
          report_error(P.err, P.err_host, kErrBadPage);
          pid = -1;
        }
        S.pages[warp][t][lane] = pid;
      }
    }
    __syncwarp();
  };
  int iss_j = 0, iss_t = 0, iss_slot = 0, in_flight = 0, cons_slot = 0;
  uint32_t cons_phase = 0;
  bool drop_next = P.debug_drop_tile != 0;   // (test hook)
  auto fill = [&]() {
    while (in_flight < RING && iss_j < n_my) {
      if (iss_t == 0 && iss_j > 0 && (iss_j & 31) == 0) load_pages(iss_j);
      if (drop_next) {
        drop_next = false;   // counted as in flight without being requested: its wait will run out
      } else if (lane == 0) {
        const int pid = max(0, S.pages[warp][iss_t][iss_j & 31]);
        mbar_expect_tx(&full[iss_slot], kTile);
        const uint32_t dst = ring + iss_slot * kTile;
        if (MH) {
          bulk_g2s(dst, P.pool + (static_cast<size_t>(pid) * P.hkv + kv_head) * (kPage * D), kTile, &full[iss_slot], policy);
        } else {
          tensor_g2s_3d(dst, &P.tmap, 0, (pid * P.hkv + kv_head) * kPage, 0, &full[iss_slot], policy);
        }
      }
      iss_slot = iss_slot + 1 == RING ? 0 : iss_slot + 1;
      ++in_flight;
      if (iss_t == (iss_j < j_text ? vis_cons : text_cons)) iss_t = 0, ++iss_j;
      else ++iss_t;
    }
  };
  auto wait_next = [&]() -> uint32_t {   // the oldest tile in flight
    if (!mbar_try_wait(&full[cons_slot], cons_phase)) {
      uint32_t done = 0;
      const uint32_t limit = P.debug_drop_tile ? kDebugSpinLimit : kSpinLimit;
      for (uint32_t spin = 0; !done && spin < limit; ++spin) done = mbar_try_wait(&full[cons_slot], cons_phase);
      if (!done) {
        if (lane == 0) report_error(P.err, P.err_host, kErrTimeout);
        dead = true;
      }
    }
    return ring + cons_slot * kTile;
  };
  auto release = [&]() {
    __syncwarp();
    --in_flight;
    if (++cons_slot == RING) cons_slot = 0, cons_phase ^= 1u;
    fill();
  };

  if (n_my > 0) {
    load_pages(0);
    fill();
  }
  const bool sweeps_new = n_my > 0 && n_text > 0 && (total - 1 - first) % step == 0;   // the text stream ends in this warp's last page
  const size_t in_row = static_cast<size_t>(P.layer_begin) * P.n_seqs + si;
  const uint16_t* q_in = P.q + (in_row * P.hq + head) * D;
  // The layer's inputs may not be read yet, but the L2 may be asked for them: it is where whoever writes them
  // meets the reads below.
  if (warp == 0 && lane < n_heads * (D / 64)) l2_prefetch(q_in + lane * 64);
  if (sweeps_new && lane < D / 64) {
    l2_prefetch(P.k + (in_row * P.hkv + kv_head) * D + lane * 64);
    l2_prefetch(P.v + (in_row * P.hkv + kv_head) * D + lane * 64);
  }
  __syncthreads();   // (S.dead, before anybody may set it)
  pdl_wait();
  pdl_launch_dependents();

  // ---- the layer's inputs
  if (sweeps_new) {
    if (lane < D / 8) {
      cp_async_16(&S.new_k[lane], reinterpret_cast<const uint4*>(P.k + (in_row * P.hkv + kv_head) * D) + lane);
      cp_async_16(&S.new_v[lane], reinterpret_cast<const uint4*>(P.v + (in_row * P.hkv + kv_head) * D) + lane);
    }
    if (P.layer_flags[P.layer_begin] & kLayerWritesQCache) {   // an ordinary layer's queries go to the Q Cache
      const uint4* src = reinterpret_cast<const uint4*>(q_in);
      uint4* dst = reinterpret_cast<uint4*>(P.qcache + ((static_cast<size_t>(P.layer_begin) * P.max_seqs + seq_id) * P.hq + head) * D);
      for (int e = lane; e < n_heads * (D / 8); e += 32) dst[e] = __ldcg(src + e);
    }
  }
  const int kg = lane >> 3, c8 = lane & 7;   // MH: which of 4 keys of a pass, which 16-byte chunk of the row
  const int g = lane >> 2, t4 = lane & 3;    // query groups: fragment coordinates
  float2 qf[MH ? EP2 : 1];
  uint32_t qb[MH ? 1 : KS][2];
  if constexpr (MH) {
#pragma unroll
    for (int j = 0; j < LPR; ++j) {
      const uint4 raw = __ldcg(reinterpret_cast<const uint4*>(q_in) + c8 + 8 * j);
      bf16x8_to_f32x2(raw, &qf[4 * j]);
    }
#pragma unroll
    for (int e = 0; e < EP2; ++e) qf[e] = mul2(qf[e], make_float2(P.scale_log2, P.scale_log2));
  } else {
    const uint32_t* qrow = reinterpret_cast<const uint32_t*>(q_in + static_cast<size_t>(g) * D) + t4;
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      qb[kk][0] = g < n_heads ? __ldcg(qrow + 8 * kk) : 0u;
      qb[kk][1] = g < n_heads ? __ldcg(qrow + 8 * kk + 4) : 0u;
    }
  }

  // Softmax references and this lane's parts of the sums of weights.  References start at the lowest finite
  // value: the weight of a score of minus infinity then is zero also in a warp whose first pages hold no other.
  float m[NC][NH], l[NC][NH];
  float2 acc[MH ? NV : 1][MH ? EP2 : 1];
  float o[MH ? 1 : NV][MH ? 1 : KS][4];
#pragma unroll
  for (int x = 0; x < NC; ++x)
#pragma unroll
    for (int h = 0; h < NH; ++h) m[x][h] = -FLT_MAX, l[x][h] = 0.f;
#pragma unroll
  for (int x = 0; x < NV; ++x) {
    if constexpr (MH) {
#pragma unroll
      for (int e = 0; e < EP2; ++e) acc[x][e] = make_float2(0.f, 0.f);
    } else {
#pragma unroll
      for (int i = 0; i < KS; ++i) o[x][i][0] = o[x][i][1] = o[x][i][2] = o[x][i][3] = 0.f;
    }
  }
  const int lrow = lane & 7, lmat = lane >> 3;   // ldmatrix lane roles
  const uint32_t k_off = tile_at<D, MH>(lrow + ((lmat & 1) << 3), lmat >> 1), v_off = tile_at<D, MH>(lrow + ((lmat >> 1) << 3), lmat & 1);
  // chunk 2 * i further along a lane's row (tiles are 1024-byte aligned: the swizzle is an exclusive or on the
  // address)
  auto step_addr = [](uint32_t addr, int i) -> uint32_t { return (addr ^ ((i & 3) << 5)) + ((i >> 2) << 11); };

  for (int j = 0; j < n_my; ++j) {
    const bool vis = j < j_text;
    const int n_cons = vis ? vis_cons : text_cons;
    const int pg = first + j * step - (vis ? 0 : n_vis);
    const bool ends = pg == (vis ? n_vis : n_text) - 1;
    const int nvalid = ends ? (vis ? len_vis : len_text) - pg * kPage : kPage;
    const bool takes_new = ends && !vis;   // the page with the step's new token
    const bool with_followers = NV > 1 && n_cons > 1;
    // ---- K tile
    uint32_t tile = wait_next();
    if (dead) break;
    auto patch = [&](const uint4* rows_new, int t) {   // the new token's row: into the tile, and into the pool
      if (lane < D / 8) {
        const uint4 val = rows_new[lane];
        sts128(tile + tile_at<D, MH>(nvalid - 1, lane), val);
        const int pid = S.pages[warp][t][j & 31];
        if (pid >= 0)
          reinterpret_cast<uint4*>(P.pool + ((static_cast<size_t>(pid) * P.hkv + kv_head) * kPage + (nvalid - 1)) * D)[lane] = val;
      }
      if (iss_j < n_my) fence_proxy_async();   // these generic-proxy writes precede the slot's next asynchronous refill
      __syncwarp();
    };
    if (takes_new) {
      cp_async_wait_all();
      __syncwarp();
      patch(S.new_k, 0);
    }
    float w[NH][2];    // MH: w[0][0], the weight of this lane's key; query groups: keys g, g + 8 of heads 2t, 2t + 1
    float pk[4];       // MH: weights of keys kg, 4 + kg, 8 + kg, 12 + kg
    bool raise = false;
    if constexpr (MH) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float2 kf[EP2];
#pragma unroll
        for (int b = 0; b < LPR; ++b) bf16x8_to_f32x2(lds128(tile + (4 * i + kg) * (D * 2) + c8 * 16 + b * 128), &kf[4 * b]);
        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < EP2; e += 2) {
          a0 = fma2(kf[e], qf[e], a0);
          a1 = fma2(kf[e + 1], qf[e + 1], a1);
        }
        pk[i] = (a0.x + a1.x) + (a0.y + a1.y);
      }
      release();
      // sums over the 8 lanes of a key: each lane is left with one of its 4 keys
      const bool up4 = lane & 4, up2 = lane & 2;
      const float r0 = (up4 ? pk[2] : pk[0]) + __shfl_xor_sync(0xffffffffu, up4 ? pk[0] : pk[2], 4);
      const float r1 = (up4 ? pk[3] : pk[1]) + __shfl_xor_sync(0xffffffffu, up4 ? pk[1] : pk[3], 4);
      float r = (up2 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, up2 ? r0 : r1, 2);
      r += __shfl_xor_sync(0xffffffffu, r, 1);
      const int key = (up4 ? 8 : 0) + (up2 ? 4 : 0) + kg;
      w[0][0] = key < nvalid ? r : -INFINITY;
      w[0][1] = -INFINITY;
      raise = w[0][0] > m[0][0] + 8.f;   // (fp32 weights: up to 2^8 does no harm)
    } else {
      float s[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) s[0][i] = s[1][i] = 0.f;
#pragma unroll
      for (int kk = 0; kk < KS; ++kk) {   // two chains: a product waits for the one before it
        uint32_t a[4];
        ldmatrix_x4(a, step_addr(tile + k_off, kk));
        mma_bf16_16816(s[kk & 1], a, qb[kk]);
      }
      release();
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        w[h][0] = g < nvalid ? (s[0][h] + s[1][h]) * P.scale_log2 : -INFINITY;
        w[h][1] = g + 8 < nvalid ? (s[0][2 + h] + s[1][2 + h]) * P.scale_log2 : -INFINITY;
        raise = raise || fmaxf(w[h][0], w[h][1]) > m[0][h];   // (the maximum itself: bf16 weights are exact at 1)
      }
    }
    if (__any_sync(0xffffffffu, raise)) {   // move the reference to the maximum
      float corr[NH];
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        float top = fmaxf(w[h][0], w[h][1]);
#pragma unroll
        for (int off = MH ? 2 : 4; off < 32; off <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
        top = fmaxf(top, m[0][h]);
        corr[h] = ex2_approx(m[0][h] - top);
        m[0][h] = top;
        l[0][h] *= corr[h];
        if (with_followers) l[NC - 1][h] *= corr[h];
      }
      if (j > 0) {
#pragma unroll
        for (int x = 0; x < NV; ++x) {
          if (x == 0 || with_followers) {
            if constexpr (MH) {
#pragma unroll
              for (int e = 0; e < EP2; ++e) acc[x][e] = mul2(acc[x][e], make_float2(corr[0], corr[0]));
            } else {
#pragma unroll
              for (int i = 0; i < KS; ++i) o[x][i][0] *= corr[0], o[x][i][1] *= corr[NH - 1], o[x][i][2] *= corr[0], o[x][i][3] *= corr[NH - 1];
            }
          }
        }
      }
    }
    uint32_t pb[2][2], pb_skip[2][2];   // query groups: the weights as B operands, in two parts
    // The first part is the next bf16 value below the weight and the second what is left, so a weight that is
    // not zero has two positive parts: an infinite value element stays infinite (times a zero or negative part
    // it would not).
    auto operands = [&](uint32_t (&b)[2][2]) {
      constexpr float kBelow = 1.f - 0x1p-24f;   // the largest float below 1
#pragma unroll
      for (int j2 = 0; j2 < 2; ++j2) {
        const uint32_t hi = pack_bf16x2_rz(w[0][j2] * kBelow, w[NH - 1][j2] * kBelow);
        b[0][j2] = movmatrix_trans(hi);
        b[1][j2] = movmatrix_trans(pack_bf16x2(w[0][j2] - __uint_as_float(hi << 16), w[NH - 1][j2] - __uint_as_float(hi & 0xffff0000u)));
      }
    };
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      w[h][0] = ex2_approx(w[h][0] - m[0][h]);
      w[h][1] = MH ? 0.f : ex2_approx(w[h][1] - m[0][h]);
      l[0][h] += w[h][0] + w[h][1];
    }
    if constexpr (MH) {
#pragma unroll
      for (int i = 0; i < 4; ++i) pk[i] = __shfl_sync(0xffffffffu, w[0][0], (lane & 24) + (i >> 1) * 4 + (i & 1) * 2);
    } else {
      operands(pb);
    }
    if (with_followers) {   // they leave out the new token: its value row of theirs does not exist yet
      const int r_new = takes_new ? nvalid - 1 : kPage;
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        if (MH) {
          if ((lane & 4 ? 8 : 0) + (lane & 2 ? 4 : 0) + kg == r_new) w[h][0] = 0.f;
        } else {
          if (g == r_new) w[h][0] = 0.f;
          if (g + 8 == r_new) w[h][1] = 0.f;
        }
        m[NC - 1][h] = m[0][h];
        if (NC > 1) l[NC - 1][h] += w[h][0] + w[h][1];
      }
      if constexpr (!MH) {
        if (takes_new) operands(pb_skip);
      }
    }
    // ---- V tiles
#pragma unroll
    for (int x = 0; x < NV; ++x) {
      if (x < n_cons) {
        tile = wait_next();
        if (dead) break;
        if (takes_new && x == 0) patch(S.new_v, 1);
        const int nv = nvalid - (takes_new && x > 0 ? 1 : 0);
        if (nv < kPage) {
          // rows past the end hold whatever the pool held (a zero weight does not cancel a NaN): cleared
          for (int e = nv * (D / 8) + lane; e < kPage * (D / 8); e += 32) sts128(tile + tile_at<D, MH>(e / (D / 8), e % (D / 8)), make_uint4(0u, 0u, 0u, 0u));
          if (iss_j < n_my) fence_proxy_async();
          __syncwarp();
        }
        if constexpr (MH) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float2 vf[EP2];
#pragma unroll
            for (int b = 0; b < LPR; ++b) bf16x8_to_f32x2(lds128(tile + (4 * i + kg) * (D * 2) + c8 * 16 + b * 128), &vf[4 * b]);
#pragma unroll
            for (int e = 0; e < EP2; ++e) acc[x][e] = fma2(vf[e], make_float2(pk[i], pk[i]), acc[x][e]);
          }
        } else {
#pragma unroll
          for (int i = 0; i < KS; ++i) {
            uint32_t a[4];
            ldmatrix_x4_trans(a, step_addr(tile + v_off, i));
            if (x > 0 && takes_new) {
              mma_bf16_16816(o[x][i], a, pb_skip[0]);
              mma_bf16_16816(o[x][i], a, pb_skip[1]);
            } else {
              mma_bf16_16816(o[x][i], a, pb[0]);
              mma_bf16_16816(o[x][i], a, pb[1]);
            }
          }
        }
        release();
      }
    }
    if (dead) break;
  }
  if (dead) {
    cp_async_wait_all();
    S.dead = 1;
    const uint32_t limit = P.debug_drop_tile ? kDebugSpinLimit : kSpinLimit;
    while (in_flight > 0) {   // copies still in flight write into this CTA's shared memory: a bounded chance to land
      uint32_t done = 0;
      for (uint32_t spin = 0; !done && spin < limit; ++spin) done = mbar_try_wait(&full[cons_slot], cons_phase);
      --in_flight;
      if (++cons_slot == RING) cons_slot = 0, cons_phase ^= 1u;
    }
  }

  // ---- the warp's sums, over its own tiles (all consumed): [consumer][part or head][D]; the parts are a
  // head's sums over a quarter of the keys each (MH)
  constexpr int kParts = MH ? 4 : kRowHeads<MH>;
  static_assert(NV * kParts * kRowStride<D, MH, NV> * 4 <= RING * static_cast<int>(kTile), "a warp's sums fit its tiles");
  float* stage = reinterpret_cast<float*>(base_ptr + static_cast<size_t>(warp) * RING * kTile);
  // (a warp that had no pages has stored nothing but zeros, with no weight)
  __syncwarp();
  {
#pragma unroll
    for (int x = 0; x < NV; ++x) {
      if constexpr (MH) {
#pragma unroll
        for (int b = 0; b < LPR; ++b) {
          float4* d4 = reinterpret_cast<float4*>(stage + (x * kParts + kg) * kRowStride<D, MH, NV> + 64 * b + 8 * c8);
          d4[0] = make_float4(acc[x][4 * b].x, acc[x][4 * b].y, acc[x][4 * b + 1].x, acc[x][4 * b + 1].y);
          d4[1] = make_float4(acc[x][4 * b + 2].x, acc[x][4 * b + 2].y, acc[x][4 * b + 3].x, acc[x][4 * b + 3].y);
        }
      } else {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          float* d = stage + (x * kParts + 2 * t4 + h) * kRowStride<D, MH, NV> + g;
#pragma unroll
          for (int i = 0; i < KS; ++i) d[16 * i] = o[x][i][h], d[16 * i + 8] = o[x][i][2 + h];
        }
      }
    }
  }
#pragma unroll
  for (int x = 0; x < NC; ++x)
#pragma unroll
    for (int h = 0; h < NH; ++h) {
#pragma unroll
      for (int off = MH ? 2 : 4; off < 32; off <<= 1) l[x][h] += __shfl_xor_sync(0xffffffffu, l[x][h], off);
      if (lane < (MH ? 1 : 4)) S.ml[x][NH * t4 * (MH ? 0 : 1) + h][warp] = make_float2(m[x][h], l[x][h]);
    }
  __syncthreads();
  // ---- the CTA's sums: the warps' weights, then a thread per VE adjacent elements of a (consumer, head).  A sum with no
  // weight counts for nothing, one that is not a number makes the row not a number.
  if (threadIdx.x < NC * kRowHeads<MH>) {
    const int cl = threadIdx.x / kRowHeads<MH>, h = threadIdx.x % kRowHeads<MH>;
    float2 ml[W];
    float top = -INFINITY, sum = 0.f;
#pragma unroll
    for (int v = 0; v < W; ++v) {
      ml[v] = S.ml[cl][h][v];
      top = ml[v].y > 0.f ? fmaxf(top, ml[v].x) : top;
    }
#pragma unroll
    for (int v = 0; v < W; ++v) {
      const float wt = ml[v].y > 0.f ? ex2_approx(ml[v].x - top) : 0.f;
      sum = fmaf(ml[v].y, wt, sum);
      S.weight[cl][h][v] = wt;
    }
    S.red_ml[cl][h] = make_float2(top, sum);
  }
  __syncthreads();
  constexpr int VE = MH ? 2 : 4;
  using Vec = typename std::conditional<MH, float2, float4>::type;
  constexpr int kPerHead = D / VE;
  const int n_units = NV * n_heads * kPerHead;
  auto unit_of = [&](int i, int& x, int& h, int& e) {
    const int pair = i / kPerHead;
    e = (i - pair * kPerHead) * VE;
    x = MH ? pair : pair / n_heads, h = MH ? 0 : pair - x * n_heads;
  };
  auto mad = [](Vec& r, float w, const Vec& v) {
    if (!(w > 0.f)) return;   // (no weight times an infinite element would not be a number)
    r.x = fmaf(v.x, w, r.x), r.y = fmaf(v.y, w, r.y);
    if constexpr (!MH) r.z = fmaf(v.z, w, r.z), r.w = fmaf(v.w, w, r.w);
  };
  for (int i = threadIdx.x; i < n_units; i += (W * 32)) {
    int x, h, e;
    unit_of(i, x, h, e);
    const float* src = reinterpret_cast<const float*>(base_ptr) + (x * kParts + (MH ? 0 : h)) * kRowStride<D, MH, NV> + e;
    const float* wt = S.weight[x > 0 ? NC - 1 : 0][h];
    Vec r{};
#pragma unroll
    for (int v = 0; v < W; ++v) {
      const float* at = src + static_cast<size_t>(v) * RING * (kTile / 4);
      Vec a = *reinterpret_cast<const Vec*>(at);
      if constexpr (MH) {
#pragma unroll
        for (int k4 = 1; k4 < 4; ++k4) {
          const Vec b = *reinterpret_cast<const Vec*>(at + k4 * kRowStride<D, MH, NV>);
          a.x += b.x, a.y += b.y;
        }
      }
      mad(r, wt[v], a);
    }
    *reinterpret_cast<Vec*>(&S.red[x][h][e]) = r;
  }
  // ---- the row: its elements are dealt out over the cluster
  const int unit0 = threadIdx.x * n_ctas + rank, unit_step = (W * 32) * n_ctas;
  // what the leader's launch left for this layer (one consumer), asked for ahead of the barrier
  float2 e_ml = make_float2(-INFINITY, 0.f);
  Vec e_acc{};
  auto slot_row = [&](int layer, int h) {   // slot 0
    return (static_cast<size_t>(layer) * P.max_seqs + si) * P.max_slots * P.hq + head + h;
  };
  auto load_earlier = [&](int i) {
    int x, h, e;
    unit_of(i, x, h, e);
    const size_t at = slot_row(P.layer_begin, h);
    e_ml = __ldcg(P.part_ml + at);
    e_acc = __ldcg(reinterpret_cast<const Vec*>(P.part_acc + at * D + e));
  };
  if (J.add_earlier && unit0 < n_units) load_earlier(unit0);
  cluster_sync();
  auto gather = [&](auto most) {   // n_ctas <= most
    constexpr int kMost = decltype(most)::value;
    for (int i = unit0; i < n_units; i += unit_step) {
      int x, h, e;
      unit_of(i, x, h, e);
      const int cl = x > 0 ? NC - 1 : 0;
      if (J.add_earlier && i != unit0) load_earlier(i);
      const uint32_t ml_at = smem_u32(&S.red_ml[cl][h]), acc_at = smem_u32(&S.red[x][h][e]), dead_at = smem_u32(&S.dead);
      float2 ml[kMost];
      Vec a[kMost];
      int lost = 0;
#pragma unroll
      for (int c = 0; c < kMost; ++c) {
        const uint32_t peer = min(c, n_ctas - 1);
        ml[c] = peer_load2(peer_addr(ml_at, peer));
        if constexpr (MH) a[c] = peer_load2(peer_addr(acc_at, peer));
        else a[c] = peer_load4(peer_addr(acc_at, peer));
        lost |= peer_load_s32(peer_addr(dead_at, peer));
        if (c >= n_ctas) ml[c].y = 0.f;
      }
      if (lost) continue;   // a CTA gave up: the row stays unwritten
      float top = e_ml.y > 0.f ? e_ml.x : -INFINITY;
#pragma unroll
      for (int c = 0; c < kMost; ++c) top = ml[c].y > 0.f ? fmaxf(top, ml[c].x) : top;
      const float we = e_ml.y > 0.f ? ex2_approx(e_ml.x - top) : 0.f;
      float sum = e_ml.y * we;
      Vec r{};
      mad(r, we, e_acc);
#pragma unroll
      for (int c = 0; c < kMost; ++c) {
        const float wt = ml[c].y > 0.f ? ex2_approx(ml[c].x - top) : 0.f;
        sum = fmaf(ml[c].y, wt, sum);
        mad(r, wt, a[c]);
      }
      if (x == 0) {
        const float inv = 1.f / sum;
        const size_t orow = in_row * P.hq + head + h;
        uint32_t* dst = reinterpret_cast<uint32_t*>(P.out + orow * D + e);
        const uint32_t o0 = f32_to_bf16_rne(r.x * inv) | (static_cast<uint32_t>(f32_to_bf16_rne(r.y * inv)) << 16);
        if constexpr (MH) *dst = o0;
        else *reinterpret_cast<uint2*>(dst) = make_uint2(o0, f32_to_bf16_rne(r.z * inv) | (static_cast<uint32_t>(f32_to_bf16_rne(r.w * inv)) << 16));
        if (P.lse != nullptr && e == 0) P.lse[orow] = (top + log2f(sum)) * 0.6931471805599453f;
      } else {
        const size_t at = slot_row(J.vis.v_layer[x], h);
        *reinterpret_cast<Vec*>(P.part_acc + at * D + e) = r;
        if (e == 0) P.part_ml[at] = make_float2(top, sum);
      }
    }
  };
  if (n_ctas == 1) gather(std::integral_constant<int, 1>{});
  else if (n_ctas == 2) gather(std::integral_constant<int, 2>{});
  else if (n_ctas <= 4) gather(std::integral_constant<int, 4>{});
  else gather(std::integral_constant<int, 8>{});
  if (n_ctas > 1) cluster_sync();   // nobody reads this CTA's shared memory any more
}

template <int D, bool MH, int NV, int W, int RING>
constexpr int rows_smem_bytes() {
  return 1024 + W * RING * kPage * D * 2 + static_cast<int>(sizeof(RowSmem<D, MH, NV, W, RING>));
}

// Calls fn(kernel, shared memory) for the kernel that a launch takes.
template <typename Fn>
cudaError_t with_rows_kernel(int d, bool mh, int nv, int warps, Fn fn) {
  using std::integral_constant;
  auto by_nv = [&](auto dd, auto m, auto w, auto r) -> cudaError_t {
    constexpr int D = decltype(dd)::value, W = decltype(w)::value, R = decltype(r)::value;
    constexpr bool MH = decltype(m)::value;
    switch (nv) {
      case 1: return fn(attend_rows_kernel<D, MH, 1, W, R>, rows_smem_bytes<D, MH, 1, W, R>());
      case 2: return fn(attend_rows_kernel<D, MH, 2, W, R>, rows_smem_bytes<D, MH, 2, W, R>());
      case 3: return fn(attend_rows_kernel<D, MH, 3, W, R>, rows_smem_bytes<D, MH, 3, W, R>());
      default: return fn(attend_rows_kernel<D, MH, 4, W, R>, rows_smem_bytes<D, MH, 4, W, R>());
    }
  };
  auto by_warps = [&](auto dd) -> cudaError_t {
    if (!mh) return by_nv(dd, std::false_type{}, integral_constant<int, 6>{}, integral_constant<int, 4>{});
    switch (warps) {
      case 1: return by_nv(dd, std::true_type{}, integral_constant<int, 1>{}, integral_constant<int, 3>{});
      case 2: return by_nv(dd, std::true_type{}, integral_constant<int, 2>{}, integral_constant<int, 2>{});
      case 3: return by_nv(dd, std::true_type{}, integral_constant<int, 3>{}, integral_constant<int, 2>{});
      case 4: return by_nv(dd, std::true_type{}, integral_constant<int, 4>{}, integral_constant<int, 2>{});
      default: return by_nv(dd, std::true_type{}, integral_constant<int, 6>{}, integral_constant<int, 4>{});
    }
  };
  return d == 128 ? by_warps(integral_constant<int, 128>{}) : by_warps(integral_constant<int, 64>{});
}

}  // namespace

// The kernels that a cache's launches can take (each of them is loaded by this, so the others are left alone),
// and what is resident of the one that fits least.
cudaError_t configure_rows_kernels(int d, int group, const std::vector<RowJobs>& layers, RowPlaces& places) {
  for (int& n : places.clusters) n = INT_MAX;
  for (int& n : places.per_sm) n = INT_MAX;
  for (int nv = 1; nv <= kMaxCons; ++nv) {
    bool used = false;
    for (const RowJobs& j : layers) used = used || (j.has_vis ? j.vis.n_cons : j.has_text ? j.text.n_cons : 0) == nv;
    for (int warps : {6, 4, 3, 2, 1}) {
      if (!used || (group > 1 && warps != 6)) continue;
      const cudaError_t e = with_rows_kernel(d, group == 1, nv, warps, [&](auto kernel, int smem) {
        cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r == cudaSuccess) r = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        int n = 0;
        if (r == cudaSuccess && warps < 6) {
          r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, warps * 32, smem);
          places.per_sm[warps] = std::min(places.per_sm[warps], n);
        }
        for (int i = 0; r == cudaSuccess && warps == 6 && i < 4; ++i) {
          cudaLaunchConfig_t cfg{};
          cfg.gridDim = dim3(1u << i);
          cfg.blockDim = dim3(warps * 32);
          cfg.dynamicSmemBytes = smem;
          cudaLaunchAttribute attr;
          attr.id = cudaLaunchAttributeClusterDimension;
          attr.val.clusterDim.x = 1u << i, attr.val.clusterDim.y = 1, attr.val.clusterDim.z = 1;
          cfg.attrs = &attr;
          cfg.numAttrs = 1;
          r = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
          places.clusters[i] = std::min(places.clusters[i], n);
        }
        return r;
      });
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_attend_rows(const Params& p, const RowJobs& jobs, int n_sms, cudaStream_t stream) {
  const int nv = jobs.has_vis ? jobs.vis.n_cons : jobs.text.n_cons;
  return with_rows_kernel(p.d, p.group == 1, nv, p.row_warps, [&](auto kernel, int smem) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(p.n_seqs * p.heads_per_item_dim * p.row_cluster));
    cfg.blockDim = dim3(p.row_warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = p.row_cluster, attr[1].val.clusterDim.y = 1, attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    // An SM holds eight clusters at most, clusters of one too: single CTAs beyond that are launched as what
    // they are (1 280 rows of 19 pages 45.0 -> 31.1 us a layer, 1 760 48.0 -> 39.2; up to eight per SM clusters
    // are the better, 1 024 26.1 against 26.4).
    cfg.numAttrs = p.row_cluster > 1 || cfg.gridDim.x <= 8u * static_cast<unsigned>(n_sms) ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, p, jobs);
  });
}

}  // namespace qc
