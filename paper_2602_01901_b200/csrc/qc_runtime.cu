// Host runtime behind the C ABI of include/qc.h: context, cache object, paged allocator,
// page tables, per-step planning and kernel launches.  No device memory is allocated here:
// everything lives in the pool and the workspace the caller hands to qc_alloc_cache.

#include "../../include/qc.h"
#include "qc_internal.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

using namespace qc;

namespace {

constexpr int kStageSlots = 8;       // pinned step-descriptor ring
constexpr int kMaxProfileSteps = 16384;
constexpr size_t kStoreSegs = 1 << 14;          // runs of tokens per launch of the kernel that stores prompt rows
constexpr size_t kPromptBytes = 786432;   // a prompt's kinds, tile codes and passes, on the device and in pinned memory
constexpr int kStoreBlocksBeside = 1, kStoreBlocksAlone = 7;   // blocks per SM of the kernel that stores prompt rows
// Page tables of a prompt call: a small mirror goes to the device whole, in one copy; otherwise the used ids of up
// to four listed sequences in a copy each, as far as they fit; otherwise the whole mirror as it is.
constexpr size_t kStageTableBytes = 1 << 20, kSmallTableBytes = 1 << 17;
constexpr int kStageTableSeqs = 4;
constexpr size_t kPromptStageBytes = kStoreSegs * sizeof(StoreSeg) + kPromptBytes + kStageTableBytes;
// Shared-score passes run one CTA per SM (three accumulators fill tensor memory); that pays once
// a CTA has enough key tiles: measured -16 % / -10 % call time at 2048 / 3008 tokens, +4 % / +9 %
// at 1120 / 675.
constexpr int kPrefillShareMinTokens = 1536;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct SeqState {
  bool active = false;
  int32_t len_text = 0, len_vis = 0;
  std::vector<int32_t> alloc_order;
};

// One attention launch: a run of consecutive lazy blocks.
struct LaunchGroup {
  int job_begin, job_end, layer_begin, layer_end;
  int extra_key_leader;   // >= 0: the merge of these layers adds the step's new token (in-order schedule, GLA followers)
  int wv, wt;             // tiles per page summed over the launch's visual / text jobs
  int w_min, w_max;       // smallest / largest tiles per page of a job of the launch
  int w_max_v, w_max_t;   // largest tiles per page among its visual / text jobs
};

// A step opened by qc_decode_begin: what its layer-by-layer launches need.
struct OpenStep {
  bool active = false;
  Params p{};
  LaunchList launches{};
  bool use_static = false;
  int64_t tot_v = 0, tot_t = 0, bytes = 0;
  int next_layer = 0;
};

struct Layout {   // byte offsets into the workspace
  size_t table, layer_flags, layer_kind, leader, jobs, plan, qcache, part_acc, part_ml, logits, items, step, err, counters, row_slots, row_done, wdesc, cdesc, row_pieces, stage_q,
      stage_k, stage_v, stage_out, stage_lse, tok, prompt, total;
  size_t step_seqs, step_patches, step_bytes;   // offsets inside the step block
};

}  // namespace

struct qc_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int n_sms = 0;
};

struct qc_cache {
  qc_ctx* ctx = nullptr;
  qc_config cfg{};
  std::vector<uint8_t> kind;
  std::vector<int> leader;
  std::vector<uint8_t> layer_flags;
  int D = 0, hq = 0, hkv = 0, group = 0;
  int heads_per_item = 1;  // query heads one work item covers (8 with GQA: one query group, or a slice of it)
  int items_per_chunk = 0; // work items per (chunk, sequence)
  CUtensorMap tmap{};      // the pool's (page, head) tiles, for the query-group decode kernels
  CUtensorMap tmap_rows{}; // the pool's rows, for the prompt kernel
  bool paged = true;
  int max_pages = 0;       // per stream
  int chunk_pages = 0, min_chunk_pages = 0, max_slots = 0;
  bool auto_split = false;         // choose chunk_pages per step from the amount of work
  int n_visual_jobs = 0, n_text_jobs = 0;
  int64_t visual_row_reads = 0, text_row_reads = 0;   // K/V rows read per visual / text token per step
  // launch plan: jobs in item-list order (launch group by launch group, heaviest first)
  std::vector<PlanJob> plan;                 // plan[p] for p < n_pos, uploaded to the workspace
  std::vector<int> plan_vis_before, plan_text_before;   // n_pos + 1 entries
  std::vector<LaunchGroup> groups;
  std::vector<std::pair<int, int>> group_pos;           // plan positions [begin, end) of each launch
  bool plan_dirty = true;
  int plan_per = 0;               // blocks per launch the plan was built for (0 = all in one)
  // host-buffer entry point: copies of one launch group overlap the kernels of the others
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  std::vector<cudaEvent_t> ev_in, ev_done;
  bool prefill_tcgen05 = true;    // head_dim 128: tcgen05 kernel; otherwise (or when switched off) mma.sync kernel
  bool pool_map_ok = false;       // both were encoded
  int prefill_pair_min_tokens = 0;   // prompts this long that start a sequence run two query tiles per CTA (0: never)
  int prefill_shared = 1;         // GLA prefill: layers of a block whose scores coincide share one score pass
                                  // (0 never, 1 for prompts of kPrefillShareMinTokens or more, 2 always)
  std::vector<PrefillPass> prefill_passes;   // singles first, then shared passes (GLA only; else empty)
  int prefill_n_single = 0, prefill_n_shared = 0;
  int64_t n_pool_pages = 0;
  int layers_per_launch = 0;
  float scale = 0.f;

  uint8_t* ws = nullptr;
  uint16_t* pool = nullptr;
  Layout lay{};
  size_t max_items = 0, max_segs = 0, max_patches = 0;

  std::vector<int32_t> table;          // host mirror
  std::vector<int32_t> free_stack;
  std::vector<SeqState> seqs;
  std::vector<Job> jobs;
  std::vector<std::pair<int, int>> block_jobs;   // per lazy block: [job_begin, job_end)
  std::vector<std::pair<int, int>> block_layers; // per lazy block: [layer_begin, layer_end)
  std::vector<Job> layer_jobs;                    // per-layer schedule (logit cache)
  std::vector<std::pair<int, int>> layer_job_range;   // per layer: [job_begin, job_end) in layer_jobs
  std::vector<Job> inorder_jobs;                  // in-order schedule (a leader's launch also sweeps its followers' cached V)
  std::vector<std::pair<int, int>> inorder_job_range;
  std::vector<int> inorder_extra_key;             // per layer: the leader whose new token the merge adds, or -1
  std::vector<RowJobs> row_jobs;                  // per layer, for launches that give every output row a cluster
  bool rows_fit = false;                          // every layer's sweeps have that form
  int text_launches = 0, no_launches = 0;         // layers whose launch sweeps the text alone, that have no sweep
  RowPlaces row_places;                           // thread blocks of such launches that are resident at once
  int row_warps = 0;                              // warps of a CTA where rows have one each: 0 chosen per step
  int row_cluster = -1;                           // CTAs per output row: -1 chosen per step, 0 never, n always n
  int slots_per_stream = 0;
  int static_partition = -1;      // -1: static ranges when a step is several launches; 0 never; 1 always
  bool fused_merge = true;        // small launches of one layer merge their output rows themselves (no merge launch)
  bool fold_append = true;        // in-order schedule: new rows are taken and stored by the layer's own launch
  bool plan_ahead = true;         // one kernel per step works out where every worker of every launch starts
  int static_row_cost = 4;        // tiles a row counts for besides its pages (a worker's cost of one more item)
  int static_min_tiles = 1;       // a static range is at least this long when the launch has the work for it
                                  // (and at least a page of the heaviest job).  Small launches want every
                                  // worker there is: batch 1, 1 024 launches: 6 12.7 ms, 3 11.5, 1 11.0
  int text_streams_per_seq = 0;        // pages a sequence needs when its text crosses a page

  // pinned staging ring for step descriptors
  uint8_t* pinned = nullptr;
  uint8_t* prompt_stage = nullptr;    // pinned: what a prompt call uploads (runs of tokens | prompt | page-table rows)
  cudaEvent_t prompt_staged = nullptr;
  int32_t* err_host = nullptr;        // mapped host word the kernels mirror the device error word into
  int32_t* err_host_dev = nullptr;    // its device address
  int debug_drop_tile = 0;
  cudaEvent_t stage_done[kStageSlots]{};
  bool stage_used[kStageSlots]{};
  int stage_next = 0;

  // profiling
  int profile = 0;                     // 1: events per step; 2: also around every attention launch
  std::vector<cudaEvent_t> ev_launch;  // profile 2: begin / end of every attention launch
  int ev_launches = 0;
  std::vector<cudaEvent_t> ev;         // 4 per step: step begin, attend begin, attend end, step end
  int ev_steps = 0;
  int64_t prof_bytes = 0, prof_items = 0;
  std::vector<cudaEvent_t> ev_prefill; // 2 per profiled qc_prefill_attend call
  int ev_prefill_calls = 0;
  double prof_prefill_flops = 0.0;

  int64_t decode_steps = 0, attend_launches = 0, kernel_launches = 0, kv_bytes_swept = 0;
  OpenStep open;
};

namespace {

inline bool owns(const qc_cache* c, int layer, int stream) {
  if (stream >= 2 || c->kind[layer] == QC_LAYER_FULL) return true;
  if (stream == QC_STREAM_K_TEXT) return c->cfg.lazy_mode != QC_MODE_GLA;
  return false;
}

inline size_t trow(const qc_cache* c, int layer, int stream, int seq) {
  return ((static_cast<size_t>(layer) * 4 + stream) * c->cfg.max_seqs + seq) * c->max_pages;
}

int validate_config(const qc_config* cfg) {
  if (!cfg || !cfg->layer_kind) return QC_ERR_INVALID_ARG;
  if (cfg->n_layers < 1 || cfg->n_layers > 127) return QC_ERR_INVALID_ARG;
  if (cfg->n_kv_heads < 1 || cfg->n_q_heads < 1 || cfg->n_q_heads % cfg->n_kv_heads) return QC_ERR_INVALID_ARG;
  if (cfg->n_q_heads > 65535) return QC_ERR_INVALID_ARG;
  if (cfg->head_dim != 64 && cfg->head_dim != 128) return QC_ERR_UNSUPPORTED;
  if (cfg->page_size != 16 && cfg->page_size != 0) return QC_ERR_UNSUPPORTED;
  if (cfg->max_seqs < 1 || cfg->max_seqs > 4096) return QC_ERR_INVALID_ARG;
  if (cfg->max_tokens_per_seq < 1 || cfg->max_tokens_per_seq > (1 << 20) - 16) return QC_ERR_INVALID_ARG;
  if (cfg->page_size == 16 && (cfg->n_pages < 1 || cfg->n_pages > 0x7fffffffLL)) return QC_ERR_INVALID_ARG;
  if (cfg->lazy_mode < 0 || cfg->lazy_mode > 2) return QC_ERR_INVALID_ARG;
  if (cfg->split_tokens != 0 &&
      (cfg->split_tokens % 16 || cfg->split_tokens < 16 || cfg->split_tokens > 16 * kMaxChunkPages))
    return QC_ERR_INVALID_ARG;
  if (!(cfg->softmax_scale >= 0.f) || !std::isfinite(cfg->softmax_scale)) return QC_ERR_INVALID_ARG;
  for (int l = 0; l < cfg->n_layers; ++l)
    if (cfg->layer_kind[l] != QC_LAYER_FULL && cfg->layer_kind[l] != QC_LAYER_LAZY) return QC_ERR_INVALID_ARG;
  if (cfg->layer_kind[0] != QC_LAYER_FULL) return QC_ERR_STATE;
  return QC_OK;
}

// Jobs of the whole stack, lazy block by lazy block.
void build_jobs(const qc_config* cfg, std::vector<Job>& jobs, std::vector<std::pair<int, int>>& block_jobs,
                std::vector<std::pair<int, int>>& block_layers) {
  const int N = cfg->n_layers;
  // own-query sweeps keep one set of query fragments per consumer in registers: the
  // query-group (tensor-core) kernel feeds two layers per sweep, the one-head kernel four
  const int max_own = cfg->n_q_heads > cfg->n_kv_heads ? 2 : kMaxCons;
  int l = 0;
  while (l < N) {
    const int c = l;
    int e = l + 1;
    while (e < N && cfg->layer_kind[e] == QC_LAYER_LAZY) ++e;   // followers c+1 .. e-1
    const int job0 = static_cast<int>(jobs.size());
    auto shared_jobs = [&](int stream, bool cached) {
      // the leader's query scores once; weights applied to the V of the leader and followers
      for (int first = c; first < e; first += kMaxCons) {
        Job j{};
        j.k_layer = static_cast<uint8_t>(c);
        j.stream = static_cast<uint8_t>(stream);
        j.n_cons = static_cast<uint8_t>(std::min(kMaxCons, e - first));
        j.flags = kFlagShared;
        for (int x = 0; x < j.n_cons; ++x) {
          j.v_layer[x] = static_cast<uint8_t>(first + x);
          j.q_layer[x] = static_cast<uint8_t>(c);
        }
        if (cached && e - c > 1) j.flags |= static_cast<uint8_t>(1u << kFlagCachedShift);
        jobs.push_back(j);
      }
    };
    auto own_query_jobs_on_leader_keys = [&](int stream) {   // Eq. 8: own q on the leader's visual K
      for (int first = c; first < e; first += max_own) {
        Job j{};
        j.k_layer = static_cast<uint8_t>(c);
        j.stream = static_cast<uint8_t>(stream);
        j.n_cons = static_cast<uint8_t>(std::min(max_own, e - first));
        j.flags = (j.n_cons == 1) ? kFlagShared : 0;
        for (int x = 0; x < j.n_cons; ++x) {
          j.v_layer[x] = static_cast<uint8_t>(first + x);
          j.q_layer[x] = static_cast<uint8_t>(first + x);
        }
        jobs.push_back(j);
      }
    };
    auto own_jobs = [&](int stream) {   // every layer of the block: own q, own K, own V
      for (int x = c; x < e; ++x) {
        Job j{};
        j.k_layer = static_cast<uint8_t>(x);
        j.stream = static_cast<uint8_t>(stream);
        j.n_cons = 1;
        j.flags = kFlagShared;
        j.v_layer[0] = static_cast<uint8_t>(x);
        j.q_layer[0] = static_cast<uint8_t>(x);
        jobs.push_back(j);
      }
    };
    switch (cfg->lazy_mode) {
      case QC_MODE_VLA_QC:
        shared_jobs(1, true);
        own_jobs(0);
        break;
      case QC_MODE_VLA_EQ8:
        own_query_jobs_on_leader_keys(1);
        own_jobs(0);
        break;
      default:   // GLA
        shared_jobs(1, true);
        shared_jobs(0, true);
        break;
    }
    block_jobs.emplace_back(job0, static_cast<int>(jobs.size()));
    block_layers.emplace_back(c, e);
    l = e;
  }
}

// Jobs of the per-layer schedule, layer by layer: every sweep feeds one layer.  A leader with
// followers stores the scaled scores that its followers share (VLA_QC: of the visual keys; GLA: of
// all keys) in the logit cache; such a follower sweeps its own V pages with those scores and reads
// no K at all.  VLA_EQ8 followers score the leader's visual keys with their own query.
void build_layer_jobs(const qc_config* cfg, std::vector<Job>& jobs, std::vector<std::pair<int, int>>& layer_jobs) {
  const int N = cfg->n_layers;
  int leader = 0;
  for (int l = 0; l < N; ++l) {
    const bool lazy = cfg->layer_kind[l] == QC_LAYER_LAZY;
    if (!lazy) leader = l;
    const bool has_followers = !lazy && l + 1 < N && cfg->layer_kind[l + 1] == QC_LAYER_LAZY;
    const int job0 = static_cast<int>(jobs.size());
    for (int stream = 1; stream >= 0; --stream) {
      const bool shared_scores =
          cfg->lazy_mode == QC_MODE_GLA || (cfg->lazy_mode == QC_MODE_VLA_QC && stream == 1);
      Job j{};
      j.stream = static_cast<uint8_t>(stream);
      j.n_cons = 1;
      j.flags = kFlagShared;
      j.v_layer[0] = static_cast<uint8_t>(l);
      j.q_layer[0] = static_cast<uint8_t>(l);
      j.k_layer = static_cast<uint8_t>(l);
      if (lazy) {
        if (shared_scores) {
          j.k_layer = static_cast<uint8_t>(leader);   // (lengths and chunking follow the leader's stream)
          j.q_layer[0] = static_cast<uint8_t>(leader);
          j.flags |= kFlagReadLogits;
        } else if (stream == 1) {
          j.k_layer = static_cast<uint8_t>(leader);   // Eq. 8: own query on the leader's visual keys
        }
      } else if (has_followers && shared_scores) {
        j.flags |= kFlagWriteLogits;
      }
      jobs.push_back(j);
    }
    layer_jobs.emplace_back(job0, static_cast<int>(jobs.size()));
  }
}

// Jobs of the in-order schedule, layer by layer: the launch of layer l uses nothing of the layers
// after l, as in a model where a layer's q/k/v only exist once the previous layer has run.  What a
// follower shares with its leader are the scores (GLA: Q and K are the leader's, Eq. 6; VLA_QC: the
// cached query on the leader's visual K), and the V rows they weight were cached before the step:
// the visual stream never holds the new token, the text stream holds it last.  So the leader's
// sweep also weights its followers' cached V rows, one K read and one set of weights for up to
// kMaxCons layers, and leaves their partial rows behind.  A VLA_QC follower's own launch is its
// text sweep (own q, own text K); a GLA follower has no sweep at all: its merge adds the new token
// as one more key.  VLA_EQ8 followers score the leader's visual keys with their own query (Eq. 8
// shares K only), in their own launch.
void build_inorder_jobs(const qc_config* cfg, std::vector<Job>& jobs, std::vector<std::pair<int, int>>& layer_jobs,
                        std::vector<int>& extra_key) {
  const int N = cfg->n_layers;
  extra_key.assign(N, -1);
  int l = 0;
  while (l < N) {
    const int c = l;
    int e = l + 1;
    while (e < N && cfg->layer_kind[e] == QC_LAYER_LAZY) ++e;
    auto own = [&](int layer, int k_layer, int stream) {
      Job j{};
      j.k_layer = static_cast<uint8_t>(k_layer);
      j.stream = static_cast<uint8_t>(stream);
      j.n_cons = 1;
      j.flags = kFlagShared;
      j.v_layer[0] = static_cast<uint8_t>(layer);
      j.q_layer[0] = static_cast<uint8_t>(layer);
      jobs.push_back(j);
    };
    auto shared = [&](int stream, bool skip_new) {   // the leader's query; consumers c .. e-1, kMaxCons per sweep
      for (int first = c; first < e; first += kMaxCons) {
        Job j{};
        j.k_layer = static_cast<uint8_t>(c);
        j.stream = static_cast<uint8_t>(stream);
        j.n_cons = static_cast<uint8_t>(std::min(kMaxCons, e - first));
        j.flags = kFlagShared;
        for (int x = 0; x < j.n_cons; ++x) {
          j.v_layer[x] = static_cast<uint8_t>(first + x);
          j.q_layer[x] = static_cast<uint8_t>(c);
          if (skip_new && first + x != c) j.skip_new |= static_cast<uint8_t>(1u << x);
        }
        jobs.push_back(j);
      }
    };
    // the leader's launch
    int job0 = static_cast<int>(jobs.size());
    if (cfg->lazy_mode == QC_MODE_VLA_EQ8 || e - c == 1) {
      own(c, c, 1);
      own(c, c, 0);
    } else if (cfg->lazy_mode == QC_MODE_VLA_QC) {
      shared(1, false);
      own(c, c, 0);
    } else {
      shared(1, false);
      shared(0, true);
    }
    layer_jobs.emplace_back(job0, static_cast<int>(jobs.size()));
    // the followers' launches
    for (int f = c + 1; f < e; ++f) {
      job0 = static_cast<int>(jobs.size());
      if (cfg->lazy_mode == QC_MODE_VLA_EQ8) {
        own(f, c, 1);
        own(f, f, 0);
      } else if (cfg->lazy_mode == QC_MODE_VLA_QC) {
        own(f, f, 0);   // the visual partials are there already
      } else {
        extra_key[f] = c;
      }
      layer_jobs.emplace_back(job0, static_cast<int>(jobs.size()));
    }
    l = e;
  }
}

// The in-order schedule's jobs as launches that give every output row a cluster take them.
void build_row_jobs(qc_cache* c) {
  c->row_jobs.assign(c->cfg.n_layers, RowJobs{});
  c->rows_fit = true;
  for (int l = 0; l < c->cfg.n_layers; ++l) {
    RowJobs& r = c->row_jobs[l];
    for (int j = c->inorder_job_range[l].first; j < c->inorder_job_range[l].second; ++j) {
      const Job& job = c->inorder_jobs[j];
      int32_t& has = job.stream ? r.has_vis : r.has_text;
      c->rows_fit = c->rows_fit && !has && job.v_layer[0] == l && job.q_layer[0] == l;   // (a block of more than kMaxCons layers: two sweeps)
      has = 1;
      (job.stream ? r.vis : r.text) = job;
    }
    r.add_earlier = r.has_text && !r.has_vis;
    c->text_launches += r.add_earlier;
    c->no_launches += !r.has_text && !r.has_vis;
  }
}

int default_row_cost(const qc_cache* c) { return c->group > 1 ? 12 : 4; }
int default_min_tiles(const qc_cache* c) { return c->group > 1 ? 4 : 1; }

struct Sizes {
  int D, hq, hkv, max_pages, chunk_pages, max_slots, slots_per_stream;
  int64_t n_pool_pages;
  size_t page_bytes, pool_bytes, max_items, max_segs, max_patches;
  Layout lay;
};

int compute_sizes(const qc_config* cfg, Sizes* s) {
  int st = validate_config(cfg);
  if (st != QC_OK) return st;
  s->D = cfg->head_dim;
  s->hq = cfg->n_q_heads;
  s->hkv = cfg->n_kv_heads;
  s->max_pages = (cfg->max_tokens_per_seq + kPage - 1) / kPage;
  const int split = cfg->split_tokens ? cfg->split_tokens : 64;   // auto: the smallest chunk the per-step choice may take
  s->chunk_pages = split / kPage;
  // partial-row slots per stream of an output row: one per chunk when items are claimed.  Under the
  // static partition a row of P pages at w tiles per page is cut into at most P w / q + 2 pieces by
  // ranges of q tiles, and q may not exceed 30 pages of the launch's lightest job (a piece holds at
  // most kMaxChunkPages page ids); tiles per page differ by at most 5x between the jobs of a launch
  // (1 .. 1 + kMaxCons), so max_pages / 3 + 2 slots always leave room for a q within both bounds
  s->slots_per_stream = std::max((s->max_pages + s->chunk_pages - 1) / s->chunk_pages, (s->max_pages + 2) / 3 + 2);
  // a cache for few sequences may cut a row finer, down to one page per worker
  const int group = s->hq / s->hkv, rows = cfg->max_seqs * (group > 1 ? s->hkv * ((group + 7) / 8) : s->hq);
  s->slots_per_stream = std::max(s->slots_per_stream, std::min(s->max_pages + 2, kPlanWorkers / rows + 2));
  s->max_slots = 2 * s->slots_per_stream;
  s->page_bytes = static_cast<size_t>(s->hkv) * kPage * s->D * 2;
  if (cfg->page_size == 0)
    s->n_pool_pages = static_cast<int64_t>(cfg->n_layers) * 4 * cfg->max_seqs * s->max_pages;
  else
    s->n_pool_pages = cfg->n_pages;
  if (s->n_pool_pages > 0x7fffffffLL) return QC_ERR_INVALID_ARG;
  s->pool_bytes = static_cast<size_t>(s->n_pool_pages) * s->page_bytes;

  std::vector<Job> jobs;
  std::vector<std::pair<int, int>> bj, bl;
  build_jobs(cfg, jobs, bj, bl);
  std::vector<Job> layer_jobs;
  std::vector<std::pair<int, int>> lj;
  build_layer_jobs(cfg, layer_jobs, lj);
  std::vector<Job> inorder_jobs;
  std::vector<int> extra;
  lj.clear();
  build_inorder_jobs(cfg, inorder_jobs, lj, extra);
  const size_t n_jobs = std::max(std::max(jobs.size(), layer_jobs.size()), inorder_jobs.size());   // any schedule fits
  const size_t chunks_per_stream = (s->max_pages + s->chunk_pages - 1) / s->chunk_pages;
  s->max_segs = n_jobs * cfg->max_seqs;
  s->max_items = s->max_segs * chunks_per_stream * s->hq;
  s->max_patches = static_cast<size_t>(cfg->n_layers) * 2 * cfg->max_seqs;

  Layout& L = s->lay;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  const size_t N = cfg->n_layers, S = cfg->max_seqs;
  L.table = take(N * 4 * S * s->max_pages * sizeof(int32_t));
  L.layer_flags = take(N);
  L.layer_kind = take(N);
  L.leader = take(N);
  L.jobs = take(n_jobs * sizeof(Job));
  L.plan = take(n_jobs * sizeof(PlanJob));
  L.qcache = take(N * S * s->hq * s->D * 2);
  L.part_acc = take(N * S * s->max_slots * s->hq * s->D * sizeof(float));
  L.part_ml = take(N * S * s->max_slots * s->hq * sizeof(float2));
  L.logits = take(2 * S * s->hq * static_cast<size_t>(s->max_pages) * kPage * sizeof(float));
  L.items = take(s->max_items * sizeof(Item));
  // step block: header-free arrays at fixed offsets
  L.step_seqs = 0;
  L.step_patches = align_up(L.step_seqs + S * sizeof(StepSeq), 16);
  L.step_bytes = align_up(L.step_patches + s->max_patches * sizeof(Patch), 256);
  L.step = take(L.step_bytes);
  L.err = take(256);
  L.counters = take(N * sizeof(int32_t));
  L.row_slots = take(N * S * s->hq * 2 * sizeof(uint16_t));
  L.row_done = take(N * S * s->hq * sizeof(int32_t));
  L.wdesc = take(std::min<size_t>(N, kMaxPlanLaunches) * kPlanWorkers * sizeof(WorkerDesc));
  L.cdesc = take(std::min<size_t>(N, kMaxPlanLaunches) * kPlanCtas * sizeof(CtaDesc));
  L.row_pieces = take(std::min<size_t>(N, kMaxPlanLaunches) * S * s->hq * sizeof(uint32_t));
  L.stage_q = take(N * S * s->hq * s->D * 2);
  L.stage_k = take(N * S * s->hkv * s->D * 2);
  L.stage_v = take(N * S * s->hkv * s->D * 2);
  L.stage_out = take(N * S * s->hq * s->D * 2);
  L.stage_lse = take(N * S * s->hq * sizeof(float));
  L.tok = take(std::max(kStoreSegs * sizeof(StoreSeg), 3 * S * sizeof(int32_t)));
  L.prompt = take(kPromptBytes);
  L.total = off;
  return QC_OK;
}

#define QC_CUDA(expr)                            \
  do {                                           \
    cudaError_t e__ = (expr);                    \
    if (e__ != cudaSuccess) return QC_ERR_CUDA;  \
  } while (0)

Params base_params(const qc_cache* c) {
  Params p{};
  p.pool = c->pool;
  p.table = reinterpret_cast<int32_t*>(c->ws + c->lay.table);
  p.qcache = reinterpret_cast<uint16_t*>(c->ws + c->lay.qcache);
  p.part_acc = reinterpret_cast<float*>(c->ws + c->lay.part_acc);
  p.part_ml = reinterpret_cast<float2*>(c->ws + c->lay.part_ml);
  p.logits = reinterpret_cast<float*>(c->ws + c->lay.logits);
  p.items = reinterpret_cast<Item*>(c->ws + c->lay.items);
  p.plan = reinterpret_cast<const PlanJob*>(c->ws + c->lay.plan);
  p.jobs = reinterpret_cast<const Job*>(c->ws + c->lay.jobs);
  p.seqs = reinterpret_cast<StepSeq*>(c->ws + c->lay.step + c->lay.step_seqs);
  p.patches = reinterpret_cast<const Patch*>(c->ws + c->lay.step + c->lay.step_patches);
  p.layer_flags = c->ws + c->lay.layer_flags;
  p.err = reinterpret_cast<int32_t*>(c->ws + c->lay.err);
  p.err_host = c->err_host_dev;
  p.debug_drop_tile = c->debug_drop_tile;
  p.work_counter = reinterpret_cast<int32_t*>(c->ws + c->lay.counters);
  p.row_slots = reinterpret_cast<uint16_t*>(c->ws + c->lay.row_slots);
  p.row_done = reinterpret_cast<int32_t*>(c->ws + c->lay.row_done);
  p.cdesc = reinterpret_cast<const CtaDesc*>(c->ws + c->lay.cdesc);
  p.row_pieces = reinterpret_cast<uint32_t*>(c->ws + c->lay.row_pieces);
  p.slots_per_stream = c->slots_per_stream;
  p.extra_key_leader = -1;
  p.n_pool_pages = c->n_pool_pages;
  p.n_layers = c->cfg.n_layers;
  p.hq = c->hq;
  p.hkv = c->hkv;
  p.d = c->D;
  p.group = c->group;
  p.max_seqs = c->cfg.max_seqs;
  p.max_pages = c->max_pages;
  p.max_slots = c->max_slots;
  p.chunk_pages = c->chunk_pages;
  p.heads_per_item_dim = c->items_per_chunk;
  p.heads_per_item = c->heads_per_item;
  p.tmap = c->tmap;
  p.scale_log2 = c->scale * 1.4426950408889634f;
  return p;
}

// Pop pages for `n_new` more pages of (layer, stream, seq); records them in the host mirror.
void grow_stream(qc_cache* c, int layer, int stream, int seq, int have, int n_new, std::vector<Patch>* patches) {
  for (int i = 0; i < n_new; ++i) {
    const int32_t pid = c->free_stack.back();
    c->free_stack.pop_back();
    const size_t idx = trow(c, layer, stream, seq) + have + i;
    c->table[idx] = pid;
    c->seqs[seq].alloc_order.push_back(pid);
    if (patches) patches->push_back(Patch{static_cast<int32_t>(idx), pid});
  }
}

inline int pages_for(int tokens) { return (tokens + kPage - 1) / kPage; }

// The pool as the bf16 tensors that tile copies read it through: a (page, head) tile is 16 consecutive rows of
// [n_pool_pages * hkv * 16 rows][D].  For the decode kernels the column halves are a dimension of their own, [D / 64]
// [rows][64], and one copy brings a tile as [D / 64][16][64]; the prompt kernel's map is two-dimensional, box 16 x 64.
// Both with the 128-byte swizzle.  The driver entry point is looked up at run time; nothing links against the driver library.
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn tensor_map_encoder() {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
      qres != cudaDriverEntryPointSuccess)
    return nullptr;
  return reinterpret_cast<EncodeFn>(fn);
}

// A prompt tensor [n_layers][T][heads][128] bf16 as a 3-D tensor {128, heads, n_layers * T}: a
// box is 64 tokens x one head x 64 elements (128 bytes) with the 128-byte swizzle.  Rows past
// the end of the tensor read as zero.
int make_prompt_tensor_map(CUtensorMap* out, const void* base, int n_layers, int T, int heads) {
  EncodeFn enc = tensor_map_encoder();
  if (!enc) return QC_ERR_CUDA;
  const cuuint64_t dims[3] = {128, static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(n_layers) * T};
  const cuuint64_t strides[2] = {128 * 2, static_cast<cuuint64_t>(heads) * 128 * 2};
  const cuuint32_t box[3] = {64, 1, 64};
  const cuuint32_t elem_strides[3] = {1, 1, 1};
  const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                         elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? QC_OK : QC_ERR_CUDA;
}

// A prompt's K or V rows [n_rows][heads][d] bf16 as a 3-D tensor {d, n_rows, heads}: a box of the given kind is 16 rows
// in all, those of one head side by side and in row order (what a page holds of a head).
int make_rows_tensor_map(CUtensorMap* out, const void* base, int64_t n_rows, int heads, int d, int kind) {
  EncodeFn enc = tensor_map_encoder();
  if (!enc) return QC_ERR_CUDA;
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(n_rows), static_cast<cuuint64_t>(heads)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(heads) * d * 2, static_cast<cuuint64_t>(d) * 2};
  const cuuint32_t box[3] = {static_cast<cuuint32_t>(d), static_cast<cuuint32_t>(kPage >> kind), 1u << kind};
  const cuuint32_t elem_strides[3] = {1, 1, 1};
  const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, elem_strides,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? QC_OK : QC_ERR_CUDA;
}

// The prefill output [n_layers][T][hq][128] bf16 as a 4-D tensor {128, hq, T, n_layers}: a box is
// 128 tokens x one head x 64 elements; rows of a box past token T are not written.
int make_output_tensor_map(CUtensorMap* out, void* base, int n_layers, int T, int heads) {
  EncodeFn enc = tensor_map_encoder();
  if (!enc) return QC_ERR_CUDA;
  const cuuint64_t dims[4] = {128, static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(T),
                              static_cast<cuuint64_t>(n_layers)};
  const cuuint64_t strides[3] = {128 * 2, static_cast<cuuint64_t>(heads) * 128 * 2,
                                 static_cast<cuuint64_t>(T) * heads * 128 * 2};
  const cuuint32_t box[4] = {64, 1, 128, 1};
  const cuuint32_t elem_strides[4] = {1, 1, 1, 1};
  const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, elem_strides,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? QC_OK : QC_ERR_CUDA;
}

int make_pool_tensor_maps(qc_cache* c) {
  EncodeFn enc = tensor_map_encoder();
  if (!enc) return QC_ERR_CUDA;
  const cuuint64_t rows = static_cast<cuuint64_t>(c->n_pool_pages) * c->hkv * kPage;
  if (rows > 0x7fffffffULL) return QC_ERR_INVALID_ARG;   // tile coordinates are 32-bit
  const cuuint64_t d = static_cast<cuuint64_t>(c->D);
  const cuuint64_t row_dims[2] = {d, rows}, row_strides[1] = {d * 2}, dims[3] = {64, rows, d / 64}, strides[2] = {d * 2, 64 * 2};
  const cuuint32_t row_box[2] = {64, kPage}, box[3] = {64, kPage, static_cast<cuuint32_t>(d / 64)}, elem_strides[3] = {1, 1, 1};
  if (enc(&c->tmap_rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, c->pool, row_dims, row_strides, row_box, elem_strides,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return QC_ERR_CUDA;
  const CUresult r = enc(&c->tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, c->pool, dims, strides, box, elem_strides,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? QC_OK : QC_ERR_CUDA;
}

// Launch groups and the item-list order of the jobs.  Within a launch the heaviest sweeps (most
// tiles per page, visual before text) come first: items are claimed in list order, so the work
// left for the end of the launch comes in small pieces.
int rebuild_plan(qc_cache* c, int per_launch) {
  c->groups.clear();
  c->group_pos.clear();
  c->plan.clear();
  c->plan_vis_before.assign(1, 0);
  c->plan_text_before.assign(1, 0);
  // per_launch -1: the per-layer schedule with the logit cache; -2: the in-order schedule (one
  // launch per layer, a leader's launch also sweeps its followers' cached V); otherwise launches of
  // `per_launch` lazy blocks (0 = all blocks in one launch)
  const bool per_layer = per_launch < 0;
  const std::vector<Job>& jobs = per_launch == -2 ? c->inorder_jobs : (per_launch == -1 ? c->layer_jobs : c->jobs);
  const std::vector<std::pair<int, int>>& layer_range = per_launch == -2 ? c->inorder_job_range : c->layer_job_range;
  const int nb = static_cast<int>(per_layer ? layer_range.size() : c->block_jobs.size());
  const int per = per_layer ? 1 : (per_launch == 0 ? nb : per_launch);
  c->n_visual_jobs = c->n_text_jobs = 0;
  c->visual_row_reads = c->text_row_reads = 0;
  auto tiles_per_page = [](const Job& j) { return ((j.flags & kFlagReadLogits) ? 0 : 1) + j.n_cons; };
  for (const Job& j : jobs) {
    (j.stream ? c->n_visual_jobs : c->n_text_jobs)++;
    (j.stream ? c->visual_row_reads : c->text_row_reads) += tiles_per_page(j);
  }
  std::vector<int> order;
  for (int b = 0; b < nb; b += per) {
    const int e = std::min(nb, b + per);
    LaunchGroup g = per_layer ? LaunchGroup{layer_range[b].first, layer_range[b].second, b, b + 1}
                              : LaunchGroup{c->block_jobs[b].first, c->block_jobs[e - 1].second,
                                            c->block_layers[b].first, c->block_layers[e - 1].second};
    g.extra_key_leader = per_launch == -2 ? c->inorder_extra_key[b] : -1;
    order.resize(g.job_end - g.job_begin);
    for (int j = g.job_begin; j < g.job_end; ++j) order[j - g.job_begin] = j;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
      const Job &jx = jobs[x], &jy = jobs[y];
      if (jx.n_cons != jy.n_cons) return jx.n_cons > jy.n_cons;
      return jx.stream > jy.stream;
    });
    const int begin = static_cast<int>(c->plan.size());
    g.wv = g.wt = g.w_max = g.w_max_v = g.w_max_t = 0;
    g.w_min = 1 << 20;
    for (int j : order) {
      const int vb = c->plan_vis_before.back(), tb = c->plan_text_before.back();
      c->plan.push_back(PlanJob{jobs[j], vb, tb, {0, 0}});
      c->plan_vis_before.push_back(vb + (jobs[j].stream ? 1 : 0));
      c->plan_text_before.push_back(tb + (jobs[j].stream ? 0 : 1));
      const int w = tiles_per_page(jobs[j]);
      (jobs[j].stream ? g.wv : g.wt) += w;
      int& w_max_s = jobs[j].stream ? g.w_max_v : g.w_max_t;
      w_max_s = std::max(w_max_s, w);
      g.w_min = std::min(g.w_min, w);
      g.w_max = std::max(g.w_max, w);
    }
    c->groups.push_back(g);
    c->group_pos.emplace_back(begin, static_cast<int>(c->plan.size()));
  }
  QC_CUDA(cudaMemcpyAsync(c->ws + c->lay.plan, c->plan.data(), c->plan.size() * sizeof(PlanJob),
                          cudaMemcpyHostToDevice, c->ctx->stream));
  QC_CUDA(cudaStreamSynchronize(c->ctx->stream));   // the host vector may be rebuilt later
  c->plan_dirty = false;
  c->plan_per = per_launch;
  return QC_OK;
}

int sync_and_check(qc_cache* c) {
  QC_CUDA(cudaStreamSynchronize(c->ctx->stream));
  return QC_OK;
}

}  // namespace

// ------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------

extern "C" {

const char* qc_status_string(int32_t s) {
  switch (s) {
    case QC_OK: return "ok";
    case QC_ERR_INVALID_ARG: return "invalid argument";
    case QC_ERR_UNSUPPORTED: return "unsupported configuration";
    case QC_ERR_OOM_PAGES: return "out of pages";
    case QC_ERR_STATE: return "invalid state";
    case QC_ERR_CUDA: return "CUDA error";
    case QC_ERR_TIMEOUT: return "device wait timed out";
    case QC_ERR_BAD_PAGE: return "page id outside the pool";
    case QC_ERR_PLAN: return "work range outside its planned limits";
    default: return "unknown status";
  }
}

int32_t qc_init(int32_t device, void* cuda_stream, qc_ctx** out) {
  if (!out || device < 0) return QC_ERR_INVALID_ARG;
  *out = nullptr;
  int n_dev = 0;
  QC_CUDA(cudaGetDeviceCount(&n_dev));
  if (device >= n_dev) return QC_ERR_INVALID_ARG;
  QC_CUDA(cudaSetDevice(device));
  cudaDeviceProp prop;
  QC_CUDA(cudaGetDeviceProperties(&prop, device));
  if (prop.major < 10) return QC_ERR_UNSUPPORTED;
  int smem = 0, smem_tc = 0;
  QC_CUDA(configure_kernels(&smem));
  QC_CUDA(configure_kernels_tc(&smem_tc));
  QC_CUDA(configure_prefill_kernels());
  if (static_cast<size_t>(std::max(smem, smem_tc)) > prop.sharedMemPerBlockOptin) return QC_ERR_UNSUPPORTED;
  qc_ctx* ctx = new (std::nothrow) qc_ctx();
  if (!ctx) return QC_ERR_INVALID_ARG;
  ctx->device = device;
  ctx->stream = static_cast<cudaStream_t>(cuda_stream);
  ctx->n_sms = prop.multiProcessorCount;
  *out = ctx;
  return QC_OK;
}

int32_t qc_cache_bytes_required(const qc_config* cfg, size_t* pool_bytes, size_t* workspace_bytes) {
  Sizes s;
  int st = compute_sizes(cfg, &s);
  if (st != QC_OK) return st;
  if (pool_bytes) *pool_bytes = s.pool_bytes;
  if (workspace_bytes) *workspace_bytes = s.lay.total;
  return QC_OK;
}

int32_t qc_alloc_cache(qc_ctx* ctx, const qc_config* cfg, void* pool_dev, size_t pool_bytes, void* workspace_dev,
                       size_t workspace_bytes, qc_cache** out) {
  if (!ctx || !out || !pool_dev || !workspace_dev) return QC_ERR_INVALID_ARG;
  *out = nullptr;
  Sizes s;
  int st = compute_sizes(cfg, &s);
  if (st != QC_OK) return st;
  if (pool_bytes < s.pool_bytes || workspace_bytes < s.lay.total) return QC_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(pool_dev) & 255) || (reinterpret_cast<uintptr_t>(workspace_dev) & 255))
    return QC_ERR_INVALID_ARG;
  QC_CUDA(cudaSetDevice(ctx->device));

  qc_cache* c = new (std::nothrow) qc_cache();
  if (!c) return QC_ERR_INVALID_ARG;
  c->ctx = ctx;
  c->cfg = *cfg;
  c->kind.assign(cfg->layer_kind, cfg->layer_kind + cfg->n_layers);
  c->cfg.layer_kind = c->kind.data();
  c->D = s.D;
  c->hq = s.hq;
  c->hkv = s.hkv;
  c->group = s.hq / s.hkv;
  c->heads_per_item = c->group > 1 ? 8 : 1;
  // what one more item costs a worker, in tiles: a query-group item fetches its query fragments when it
  // starts and leaves up to eight partial rows (measured on launches of one layer: 4 resp. 12 best)
  c->static_row_cost = default_row_cost(c);
  c->static_min_tiles = default_min_tiles(c);
  c->items_per_chunk = c->group > 1 ? s.hkv * ((c->group + 7) / 8) : s.hq;
  c->paged = cfg->page_size == 16;
  c->max_pages = s.max_pages;
  c->chunk_pages = c->min_chunk_pages = s.chunk_pages;
  c->auto_split = cfg->split_tokens == 0;
  c->max_slots = s.max_slots;
  c->slots_per_stream = s.slots_per_stream;
  c->n_pool_pages = s.n_pool_pages;
  c->scale = cfg->softmax_scale > 0.f ? cfg->softmax_scale : 1.0f / std::sqrt(static_cast<float>(s.D));
  c->ws = static_cast<uint8_t*>(workspace_dev);
  c->pool = static_cast<uint16_t*>(pool_dev);
  c->lay = s.lay;
  c->max_items = s.max_items;
  c->max_segs = s.max_segs;
  c->max_patches = s.max_patches;
  c->leader.resize(cfg->n_layers);
  c->layer_flags.resize(cfg->n_layers);
  int last = 0;
  c->text_streams_per_seq = 0;
  for (int l = 0; l < cfg->n_layers; ++l) {
    if (c->kind[l] == QC_LAYER_FULL) last = l;
    c->leader[l] = last;
    uint8_t f = 0;
    if (owns(c, l, QC_STREAM_K_TEXT)) f |= kLayerOwnsTextK;
    if (c->kind[l] == QC_LAYER_FULL) f |= kLayerWritesQCache;
    c->layer_flags[l] = f;
    c->text_streams_per_seq += 1 + (owns(c, l, QC_STREAM_K_TEXT) ? 1 : 0);
  }
  build_jobs(&c->cfg, c->jobs, c->block_jobs, c->block_layers);
  build_layer_jobs(&c->cfg, c->layer_jobs, c->layer_job_range);
  build_inorder_jobs(&c->cfg, c->inorder_jobs, c->inorder_job_range, c->inorder_extra_key);
  build_row_jobs(c);
  if (c->cfg.lazy_mode == QC_MODE_GLA) {
    // Eq. 5: every layer of a lazy block attends with the block's first layer's Q and K, so runs
    // of up to three of its layers share one score pass of the prefill kernel
    std::vector<PrefillPass> shared;
    for (const auto& bl : c->block_layers) {
      for (int first = bl.first; first < bl.second; first += kPrefillSharedLayers) {
        PrefillPass ps{};
        ps.n = std::min(kPrefillSharedLayers, bl.second - first);
        for (int x = 0; x < ps.n; ++x) ps.v[x] = first + x;
        (ps.n > 1 ? shared : c->prefill_passes).push_back(ps);
      }
    }
    c->prefill_n_single = static_cast<int>(c->prefill_passes.size());
    c->prefill_n_shared = static_cast<int>(shared.size());
    c->prefill_passes.insert(c->prefill_passes.end(), shared.begin(), shared.end());
  }
  c->seqs.resize(cfg->max_seqs);
  c->table.assign(static_cast<size_t>(cfg->n_layers) * 4 * cfg->max_seqs * c->max_pages, -1);
  if (c->paged) {
    c->free_stack.resize(s.n_pool_pages);
    for (int64_t i = 0; i < s.n_pool_pages; ++i) c->free_stack[i] = static_cast<int32_t>(s.n_pool_pages - 1 - i);
  } else {
    // contiguous: stream (layer, stream, seq) owns pages [extent*max_pages, (extent+1)*max_pages)
    for (size_t i = 0; i < c->table.size(); ++i) c->table[i] = static_cast<int32_t>(i);
  }

  // the pool's tensor maps: needed by the query-group decode kernels; the prefill kernel uses its one for
  // cached tiles when it exists
  c->pool_map_ok = make_pool_tensor_maps(c) == QC_OK;
  if (c->group > 1 && !c->pool_map_ok) {
    delete c;
    return QC_ERR_CUDA;
  }

  cudaStream_t stream = ctx->stream;
  bool ok = !c->rows_fit || configure_rows_kernels(c->D, c->group, c->row_jobs, c->row_places) == cudaSuccess;
  ok = ok && cudaHostAlloc(reinterpret_cast<void**>(&c->pinned), kStageSlots * c->lay.step_bytes,
                          cudaHostAllocDefault) == cudaSuccess;
  for (int i = 0; ok && i < kStageSlots; ++i)
    ok = cudaEventCreateWithFlags(&c->stage_done[i], cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaHostAlloc(reinterpret_cast<void**>(&c->prompt_stage), kPromptStageBytes, cudaHostAllocDefault) == cudaSuccess &&
       cudaEventCreateWithFlags(&c->prompt_staged, cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaHostAlloc(reinterpret_cast<void**>(&c->err_host), 64, cudaHostAllocMapped) == cudaSuccess;
  if (ok) {
    *c->err_host = 0;
    ok = cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->err_host_dev), c->err_host, 0) == cudaSuccess;
  }
  ok = ok && cudaMemcpyAsync(c->ws + c->lay.table, c->table.data(), c->table.size() * sizeof(int32_t),
                             cudaMemcpyHostToDevice, stream) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(c->ws + c->lay.layer_flags, c->layer_flags.data(), c->layer_flags.size(),
                             cudaMemcpyHostToDevice, stream) == cudaSuccess;
  std::vector<uint8_t> leader8(c->leader.begin(), c->leader.end());
  ok = ok && cudaMemcpyAsync(c->ws + c->lay.layer_kind, c->kind.data(), c->kind.size(), cudaMemcpyHostToDevice,
                             stream) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(c->ws + c->lay.leader, leader8.data(), leader8.size(), cudaMemcpyHostToDevice,
                             stream) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(c->ws + c->lay.jobs, c->jobs.data(), c->jobs.size() * sizeof(Job),
                             cudaMemcpyHostToDevice, stream) == cudaSuccess;
  ok = ok && cudaMemsetAsync(c->ws + c->lay.err, 0, 256, stream) == cudaSuccess;
  ok = ok && cudaMemsetAsync(c->ws + c->lay.row_done, 0, c->lay.wdesc - c->lay.row_done, stream) == cudaSuccess;
  ok = ok && cudaMemsetAsync(c->ws + c->lay.qcache, 0, c->lay.part_acc - c->lay.qcache, stream) == cudaSuccess;
  ok = ok && cudaStreamSynchronize(stream) == cudaSuccess;
  if (!ok) {
    qc_free(nullptr, c);
    return QC_ERR_CUDA;
  }
  *out = c;
  return QC_OK;
}

int32_t qc_free(qc_ctx* ctx, qc_cache* cache) {
  if (cache) {
    if (cache->ctx) {
      cudaSetDevice(cache->ctx->device);
      cudaStreamSynchronize(cache->ctx->stream);
    }
    for (int i = 0; i < kStageSlots; ++i)
      if (cache->stage_done[i]) cudaEventDestroy(cache->stage_done[i]);
    for (cudaEvent_t e : cache->ev) cudaEventDestroy(e);
    for (cudaEvent_t e : cache->ev_launch) cudaEventDestroy(e);
    for (cudaEvent_t e : cache->ev_in) cudaEventDestroy(e);
    for (cudaEvent_t e : cache->ev_done) cudaEventDestroy(e);
    if (cache->copy_in) cudaStreamDestroy(cache->copy_in);
    if (cache->copy_out) cudaStreamDestroy(cache->copy_out);
    for (cudaEvent_t e : cache->ev_prefill) cudaEventDestroy(e);
    if (cache->pinned) cudaFreeHost(cache->pinned);
    if (cache->prompt_stage) cudaFreeHost(cache->prompt_stage);
    if (cache->prompt_staged) cudaEventDestroy(cache->prompt_staged);
    if (cache->err_host) cudaFreeHost(cache->err_host);
    delete cache;
  }
  if (ctx) delete ctx;
  return QC_OK;
}

}  // extern "C"

namespace {

// What qc_prefill_attend uploads for its kernel, along with the routing of the tokens.
struct PromptUpload {
  const uint8_t* codes;
  size_t n_codes;
  const std::vector<PrefillPass>* passes;   // null: none
  bool beside;   // the attention runs beside the stores (it does not with an event between them)
};
inline size_t codes_at(size_t n_tokens) { return align_up(n_tokens, 256); }
inline size_t passes_at(size_t n_tokens, size_t n_codes) { return codes_at(n_tokens) + align_up(n_codes, 256); }

// The body of qc_prefill_append.  Everything that is uploaded goes ahead of the kernel that stores
// the rows, through pinned memory, so that nothing stands between that kernel and the prompt's
// attention, which runs beside it.
int32_t store_prompt(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const int32_t* n_tokens, const uint8_t* kind,
                     const void* k_dev, const void* v_dev, const PromptUpload* up) {
  if (!c || n_seqs < 0 || (n_seqs > 0 && (!seq_ids || !n_tokens))) return QC_ERR_INVALID_ARG;
  if (c->open.active) return QC_ERR_STATE;   // a decode step is open
  if (n_seqs == 0) return QC_OK;
  if (!k_dev || !v_dev) return QC_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(k_dev) & 15) || (reinterpret_cast<uintptr_t>(v_dev) & 15)) return QC_ERR_INVALID_ARG;
  const int N = c->cfg.n_layers;
  // ---- validate and plan without touching the state
  int64_t total = 0, need = 0;
  std::vector<uint8_t> seen(c->cfg.max_seqs, 0);
  std::vector<int32_t> add_t(n_seqs), add_v(n_seqs);
  for (int i = 0; i < n_seqs; ++i) {
    const int s = seq_ids[i];
    if (s < 0 || s >= c->cfg.max_seqs || n_tokens[i] < 0) return QC_ERR_INVALID_ARG;
    if (seen[s]) return QC_ERR_STATE;
    seen[s] = 1;
    if (n_tokens[i] > 0 && !kind) return QC_ERR_INVALID_ARG;
    int nt = 0, nv = 0;
    for (int t = 0; t < n_tokens[i]; ++t) {
      const uint8_t kd = kind[total + t];
      if (kd == QC_KIND_TEXT) ++nt;
      else if (kd == QC_KIND_VISUAL) ++nv;
      else return QC_ERR_INVALID_ARG;
    }
    add_t[i] = nt;
    add_v[i] = nv;
    const SeqState& st = c->seqs[s];
    if (st.len_text + nt > c->cfg.max_tokens_per_seq || st.len_vis + nv > c->cfg.max_tokens_per_seq)
      return QC_ERR_INVALID_ARG;
    if (c->paged) {
      const int dt = pages_for(st.len_text + nt) - pages_for(st.len_text);
      const int dv = pages_for(st.len_vis + nv) - pages_for(st.len_vis);
      for (int l = 0; l < N; ++l)
        for (int stream = 0; stream < 4; ++stream)
          if (owns(c, l, stream)) need += (stream & 1) ? dv : dt;
    }
    total += n_tokens[i];
  }
  if (total > 0x7fffffffLL) return QC_ERR_INVALID_ARG;
  if (c->paged && need > static_cast<int64_t>(c->free_stack.size())) return QC_ERR_OOM_PAGES;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  cudaStream_t stream = c->ctx->stream;

  // ---- what can still fail without a change: the tensor maps of the caller's rows
  StoreMaps maps;
  if (total > 0) {
    if (static_cast<int64_t>(N) * total > 0x7fffffffLL) return QC_ERR_INVALID_ARG;   // rows are counted in 31 bits
    for (int i = 0; i < kStoreKinds; ++i)
      if (make_rows_tensor_map(&maps.k[i], k_dev, N * total, c->hkv, c->D, i) != QC_OK ||
          make_rows_tensor_map(&maps.v[i], v_dev, N * total, c->hkv, c->D, i) != QC_OK)
        return QC_ERR_CUDA;
  }
  QC_CUDA(cudaEventSynchronize(c->prompt_staged));   // the last call's copies from the staging area have run
  // ---- commit: pages (sequence -> layer -> stream order)
  std::vector<int32_t> at_t(n_seqs), at_v(n_seqs);   // where each sequence's new tokens start in its streams
  for (int i = 0; i < n_seqs; ++i) {
    const int s = seq_ids[i];
    SeqState& st = c->seqs[s];
    at_t[i] = st.len_text, at_v[i] = st.len_vis;
    if (c->paged) {
      const int have_t = pages_for(st.len_text), have_v = pages_for(st.len_vis);
      const int dt = pages_for(st.len_text + add_t[i]) - have_t;
      const int dv = pages_for(st.len_vis + add_v[i]) - have_v;
      for (int l = 0; l < N; ++l)
        for (int sm = 0; sm < 4; ++sm)
          if (owns(c, l, sm)) grow_stream(c, l, sm, s, (sm & 1) ? have_v : have_t, (sm & 1) ? dv : dt, nullptr);
    }
    st.len_text += add_t[i];
    st.len_vis += add_v[i];
    st.active = true;
  }
  StoreSeg* segs = reinterpret_cast<StoreSeg*>(c->prompt_stage);
  uint8_t* prompt = c->prompt_stage + kStoreSegs * sizeof(StoreSeg);
  int32_t* rows = reinterpret_cast<int32_t*>(prompt + kPromptBytes);
  if (c->paged) {
    const size_t row = c->max_pages * sizeof(int32_t), table_bytes = c->table.size() * sizeof(int32_t);
    int used = 1;   // page ids of the longest listed stream
    for (int i = 0; i < n_seqs; ++i)
      used = std::max(used, std::max(pages_for(c->seqs[seq_ids[i]].len_text), pages_for(c->seqs[seq_ids[i]].len_vis)));
    const size_t width = used * sizeof(int32_t), n_rows = static_cast<size_t>(N) * 4;
    if (table_bytes <= kSmallTableBytes) {
      std::memcpy(rows, c->table.data(), table_bytes);
      QC_CUDA(cudaMemcpyAsync(c->ws + c->lay.table, rows, table_bytes, cudaMemcpyHostToDevice, stream));
    } else if (n_seqs <= kStageTableSeqs && n_seqs * n_rows * width <= kStageTableBytes) {
      for (int i = 0; i < n_seqs; ++i, rows += n_rows * used) {
        for (size_t r = 0; r < n_rows; ++r)
          std::memcpy(rows + r * used, c->table.data() + trow(c, 0, static_cast<int>(r), seq_ids[i]), width);
        QC_CUDA(cudaMemcpy2DAsync(c->ws + c->lay.table + static_cast<size_t>(seq_ids[i]) * row, c->cfg.max_seqs * row, rows, width,
                                  width, n_rows, cudaMemcpyHostToDevice, stream));
      }
    } else {
      QC_CUDA(cudaMemcpyAsync(c->ws + c->lay.table, c->table.data(), table_bytes, cudaMemcpyHostToDevice, stream));
    }
  }
  if (up) {   // (one sequence; qc_prefill_attend has checked that it fits)
    const size_t n_kinds = static_cast<size_t>(total);
    std::memcpy(prompt, kind, n_kinds);
    std::memcpy(prompt + codes_at(n_kinds), up->codes, up->n_codes);
    size_t bytes = passes_at(n_kinds, up->n_codes);
    if (up->passes) {
      std::memcpy(prompt + bytes, up->passes->data(), up->passes->size() * sizeof(PrefillPass));
      bytes += up->passes->size() * sizeof(PrefillPass);
    }
    QC_CUDA(cudaMemcpyAsync(c->ws + c->lay.prompt, prompt, bytes, cudaMemcpyHostToDevice, stream));
  }
  QC_CUDA(cudaEventRecord(c->prompt_staged, stream));
  Params p = base_params(c);
  p.k = static_cast<const uint16_t*>(k_dev);
  p.v = static_cast<const uint16_t*>(v_dev);
  StoreSeg* segs_dev = reinterpret_cast<StoreSeg*>(c->ws + c->lay.tok);
  // runs of tokens, a batch at a time, by kind; beside the attention of the prompt the stores get one block
  // per SM, alone as many as fit
  std::vector<StoreSeg> runs[kStoreKinds];
  size_t n = 0;
  int64_t tok = 0;
  bool used = false;   // the staging area holds runs that are being copied
  auto flush = [&]() -> int32_t {
    if (used) QC_CUDA(cudaEventSynchronize(c->prompt_staged));
    StoreList list{segs_dev, {0}, static_cast<int32_t>(total)};
    for (int i = 0; i < kStoreKinds; ++i) {
      std::copy(runs[i].begin(), runs[i].end(), segs + list.first[i]);
      list.first[i + 1] = list.first[i] + static_cast<int32_t>(runs[i].size());
      runs[i].clear();
    }
    QC_CUDA(cudaMemcpyAsync(segs_dev, segs, n * sizeof(StoreSeg), cudaMemcpyHostToDevice, stream));
    QC_CUDA(cudaEventRecord(c->prompt_staged, stream));
    c->kernel_launches++;
    QC_CUDA(launch_prefill_store(p, maps, list, c->ctx->n_sms * (up && up->beside ? kStoreBlocksBeside : kStoreBlocksAlone), stream));
    n = 0;
    used = true;
    return QC_OK;
  };
  for (int i = 0; i < n_seqs; ++i) {
    for (int t = 0; t < n_tokens[i];) {
      const uint8_t kd = kind[tok + t];
      int& at = kd == QC_KIND_VISUAL ? at_v[i] : at_t[i];
      int len = 1;
      while (t + len < n_tokens[i] && kind[tok + t + len] == kd && (at + len) % kPage != 0) ++len;
      runs[store_kind(len)].push_back(StoreSeg{seq_ids[i], static_cast<int32_t>(static_cast<uint32_t>(at) | (kd == QC_KIND_VISUAL ? 0x80000000u : 0u)),
                                               static_cast<int32_t>(tok + t), len});
      at += len;
      t += len;
      if (++n == kStoreSegs) {
        const int32_t st = flush();
        if (st != QC_OK) return st;
      }
    }
    tok += n_tokens[i];
  }
  if (n > 0) {
    const int32_t st = flush();
    if (st != QC_OK) return st;
  }
  return QC_OK;
}

}  // namespace

extern "C" {

int32_t qc_prefill_append(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const int32_t* n_tokens,
                          const uint8_t* kind, const void* k_dev, const void* v_dev) {
  return store_prompt(c, n_seqs, seq_ids, n_tokens, kind, k_dev, v_dev, nullptr);
}

int32_t qc_prefill_attend(qc_cache* c, int32_t seq_id, int32_t n_tokens, const uint8_t* kind, const void* q_dev,
                          const void* k_dev, const void* v_dev, void* out_dev) {
  if (!c || n_tokens < 0 || seq_id < 0 || seq_id >= c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
  if (n_tokens == 0) return QC_OK;
  if (!kind || !q_dev || !k_dev || !v_dev || !out_dev) return QC_ERR_INVALID_ARG;
  const void* ptrs[4] = {q_dev, k_dev, v_dev, out_dev};
  for (const void* ptr : ptrs)
    if (reinterpret_cast<uintptr_t>(ptr) & 15) return QC_ERR_INVALID_ARG;
  // tokens the sequence holds already (an earlier prompt chunk, generated tokens) precede the new ones
  const int n0_text = c->seqs[seq_id].active ? c->seqs[seq_id].len_text : 0;
  const int n0_vis = c->seqs[seq_id].active ? c->seqs[seq_id].len_vis : 0;
  const int n_tiles = (n_tokens + 63) / 64;
  if (passes_at(n_tokens, n_tiles) + c->prefill_passes.size() * sizeof(PrefillPass) > kPromptBytes) return QC_ERR_INVALID_ARG;
  // what can fail without touching the cache comes first: the tensor maps over the caller's tensors
  PrefillMaps maps;
  const bool tc5 = c->prefill_tcgen05 && c->D == 128 && (c->pool_map_ok || n0_text + n0_vis == 0);
  if (tc5) {
    maps.pool = c->tmap_rows;
    if (make_prompt_tensor_map(&maps.q, q_dev, c->cfg.n_layers, n_tokens, c->hq) != QC_OK ||
        make_prompt_tensor_map(&maps.k, k_dev, c->cfg.n_layers, n_tokens, c->hkv) != QC_OK ||
        make_prompt_tensor_map(&maps.v, v_dev, c->cfg.n_layers, n_tokens, c->hkv) != QC_OK ||
        make_output_tensor_map(&maps.out, out_dev, c->cfg.n_layers, n_tokens, c->hq) != QC_OK)
      return QC_ERR_CUDA;
  }
  // per 64-token tile: all text, all visual or mixed (the tcgen05 kernel fetches unmixed tiles whole)
  std::vector<uint8_t> codes(n_tiles);
  for (int i = 0; i < n_tiles; ++i) {
    int nv = 0, n = std::min(64, n_tokens - 64 * i);
    for (int t = 0; t < n; ++t) nv += kind[64 * i + t] == QC_KIND_VISUAL;
    codes[i] = nv == 0 ? 0 : (nv == n ? 1 : 2);
  }
  const bool share = c->prefill_n_shared > 0 && n0_text + n0_vis == 0 &&
                     (c->prefill_shared == 2 || (c->prefill_shared == 1 && n_tokens >= kPrefillShareMinTokens));
  // store K/V: this validates the rest and leaves the cache unchanged on an error
  const bool timed = c->profile && c->ev_prefill_calls < kMaxProfileSteps;
  const PromptUpload up{codes.data(), codes.size(), share ? &c->prefill_passes : nullptr, !timed};
  const int st = store_prompt(c, 1, &seq_id, &n_tokens, kind, k_dev, v_dev, &up);
  if (st != QC_OK) return st;
  cudaStream_t stream = c->ctx->stream;
  const uint8_t* kind_dev = c->ws + c->lay.prompt;
  const uint8_t* codes_dev = kind_dev + codes_at(n_tokens);
  const PrefillPass* passes_dev = reinterpret_cast<const PrefillPass*>(kind_dev + passes_at(n_tokens, n_tiles));
  const Params p = base_params(c);
  cudaEvent_t* ev = nullptr;
  if (timed) {
    if (static_cast<int>(c->ev_prefill.size()) < 2 * (c->ev_prefill_calls + 1)) {
      for (int i = 0; i < 2; ++i) {
        cudaEvent_t e;
        QC_CUDA(cudaEventCreate(&e));
        c->ev_prefill.push_back(e);
      }
    }
    ev = &c->ev_prefill[2 * c->ev_prefill_calls];
    QC_CUDA(cudaEventRecord(ev[0], stream));
  }
  QC_CUDA(launch_prefill_attend(p, kind_dev, c->ws + c->lay.layer_kind, c->ws + c->lay.leader, c->leader.data(), q_dev, k_dev, v_dev,
                                out_dev, n_tokens, c->cfg.lazy_mode == QC_MODE_GLA ? 1 : 0, tc5 ? &maps : nullptr,
                                codes_dev, codes.data(), seq_id, n0_text, n0_vis, (tc5 && share) ? passes_dev : nullptr,
                                c->prefill_n_single, c->prefill_n_shared, c->prefill_pair_min_tokens, stream));
  const bool shared_run = tc5 && share;
  if (ev) {
    QC_CUDA(cudaEventRecord(ev[1], stream));
    c->ev_prefill_calls++;
    // executed arithmetic: 2 D flops per pair for the scores of every score pass, 2 D per pair for
    // the value product of every layer
    const double pairs = 0.5 * n_tokens * (n_tokens + 1.0) + static_cast<double>(n_tokens) * (n0_text + n0_vis);
    const int score_passes = shared_run ? c->prefill_n_single + c->prefill_n_shared : c->cfg.n_layers;
    c->prof_prefill_flops += 2.0 * c->D * pairs * c->hq * (score_passes + c->cfg.n_layers);
  }
  c->kernel_launches += (shared_run && c->prefill_n_single > 0) ? 2 : 1;
  return QC_OK;
}

int32_t qc_layer_similarity(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const void* q_dev, float* rows_dev,
                            int32_t max_len, float* similarity_host) {
  if (!c || n_seqs < 1 || n_seqs > c->cfg.max_seqs || !seq_ids || !q_dev || !rows_dev || !similarity_host)
    return QC_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q_dev) & 15) || (reinterpret_cast<uintptr_t>(rows_dev) & 15)) return QC_ERR_INVALID_ARG;
  if (max_len < 1 || max_len > 12288) return QC_ERR_UNSUPPORTED;   // one head's logits live in shared memory
  const int N = c->cfg.n_layers;
  for (int l = 0; l < N; ++l)
    if (c->kind[l] != QC_LAYER_FULL) return QC_ERR_STATE;          // the analysis runs on the unmodified stack
  std::vector<int32_t> host(3 * static_cast<size_t>(n_seqs));
  for (int i = 0; i < n_seqs; ++i) {
    const int s = seq_ids[i];
    if (s < 0 || s >= c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
    const SeqState& st = c->seqs[s];
    if (!st.active || st.len_text + st.len_vis == 0) return QC_ERR_STATE;
    if (st.len_text + st.len_vis > max_len) return QC_ERR_INVALID_ARG;
    host[i] = s;
    host[n_seqs + i] = st.len_text;
    host[2 * n_seqs + i] = st.len_vis;
  }
  QC_CUDA(cudaSetDevice(c->ctx->device));
  cudaStream_t stream = c->ctx->stream;
  int32_t* ids_dev = reinterpret_cast<int32_t*>(c->ws + c->lay.tok);
  float* js_dev = reinterpret_cast<float*>(c->ws + c->lay.stage_lse);   // (n_layers - 1) * n_seqs floats fit
  QC_CUDA(cudaMemcpyAsync(ids_dev, host.data(), host.size() * sizeof(int32_t), cudaMemcpyHostToDevice, stream));
  Params p = base_params(c);
  p.q = static_cast<const uint16_t*>(q_dev);
  p.n_seqs = n_seqs;
  QC_CUDA(launch_calibration(p, ids_dev, ids_dev + n_seqs, ids_dev + 2 * n_seqs, rows_dev, max_len, js_dev, stream));
  c->kernel_launches += N > 1 ? 2 : 1;
  std::vector<float> js(static_cast<size_t>(std::max(0, N - 1)) * n_seqs);
  if (!js.empty())
    QC_CUDA(cudaMemcpyAsync(js.data(), js_dev, js.size() * sizeof(float), cudaMemcpyDeviceToHost, stream));
  QC_CUDA(cudaStreamSynchronize(stream));
  for (int l = 0; l + 1 < N; ++l) {
    double acc = 0.0;
    for (int i = 0; i < n_seqs; ++i) acc += js[static_cast<size_t>(l) * n_seqs + i];
    similarity_host[l] = static_cast<float>(acc / n_seqs);
  }
  return QC_OK;
}

int32_t qc_lazy_blocks(const float* similarity, int32_t n_layers, float eps, int32_t max_block, uint8_t* layer_kind) {
  if (n_layers < 1 || !layer_kind || (n_layers > 1 && !similarity) || !(eps > 0.f) || eps > 1.f)
    return QC_ERR_INVALID_ARG;
  layer_kind[0] = QC_LAYER_FULL;
  int size = 1;
  for (int l = 1; l < n_layers; ++l) {
    if (similarity[l - 1] < eps && (max_block <= 0 || size < max_block)) {
      layer_kind[l] = QC_LAYER_LAZY;
      ++size;
    } else {
      layer_kind[l] = QC_LAYER_FULL;
      size = 1;
    }
  }
  return QC_OK;
}

}  // extern "C"

namespace {

// Events of the host-buffer entry point: launch group g waits for in[g] (its inputs have been
// copied) and records done[g] (its outputs may be copied back).
struct HostPipe {
  int per_launch;
  cudaEvent_t* in;
  cudaEvent_t* done;
};

// One attention launch of a step (group gi of the launch plan) with its merge; optionally the
// append of the group's layers first (host-buffer entry point, per-layer entry point).
int run_group(qc_cache* c, Params& p, size_t gi, const LaunchList& launches, bool use_static, int64_t tot_v,
              int64_t tot_t, bool append_first, cudaEvent_t wait_in, cudaEvent_t record_done, cudaEvent_t* ev,
              cudaStream_t stream) {
  const int pb = c->group_pos[gi].first, pe = c->group_pos[gi].second;
  p.item_begin = static_cast<int32_t>(c->plan_vis_before[pb] * tot_v + c->plan_text_before[pb] * tot_t);
  p.item_end = static_cast<int32_t>(c->plan_vis_before[pe] * tot_v + c->plan_text_before[pe] * tot_t);
  p.layer_begin = c->groups[gi].layer_begin;
  p.layer_end = c->groups[gi].layer_end;
  p.launch_index = static_cast<int32_t>(gi);
  p.pos_begin = pb;
  p.pos_end = pe;
  p.extra_key_leader = c->groups[gi].extra_key_leader;
  p.follows_setup = gi == 0 && !append_first;   // (an append waits for the set-up before it lets its successor start)
  bool has_work = p.item_end > p.item_begin;
  if (use_static) {   // (a step has at most n_layers <= 127 launches: every one has its entry)
    const LaunchDesc& one = launches.launch[gi];
    has_work = one.part_workers > 0;
    p.part_q = one.part_q;
    p.part_k = one.part_k;
    p.part_vw = one.part_vw;
    p.part_workers = one.part_workers;
    p.part_row_cost = one.part_row_cost;
    p.part_wpc = one.part_wpc;
    p.part_wv = one.part_wv;
    p.part_wt = one.part_wt;
  }
  const bool by_rows = p.row_cluster > 0;
  const RowJobs* row_jobs = by_rows ? &c->row_jobs[p.layer_begin] : nullptr;
  if (by_rows) has_work = row_jobs->has_vis || row_jobs->has_text;
  p.any_skip = p.any_own = 0;
  for (int pos = pb; pos < pe; ++pos) {
    const Job& job = c->plan[pos].job;
    p.any_skip |= job.skip_new ? 1 : 0;
    p.any_own |= job.n_cons > 1 && !(job.flags & kFlagShared) ? 1 : 0;
  }
  p.fused_merge = by_rows ? has_work : use_static ? launches.launch[gi].fused_merge : 0;
  p.planned_pieces = !by_rows && use_static && launches.launch[gi].layer >= 0 ? 1 : 0;
  if (wait_in) QC_CUDA(cudaStreamWaitEvent(stream, wait_in, 0));
  if (append_first) {
    QC_CUDA(launch_append(p, stream));   // this group's layers only
    c->kernel_launches++;
  }
  if (ev && gi == 0) QC_CUDA(cudaEventRecord(ev[1], stream));
  cudaEvent_t* evl = nullptr;
  if (ev && c->profile == 2 && has_work && c->ev_launches < 64 * kMaxProfileSteps) {
    if (static_cast<int>(c->ev_launch.size()) < 2 * (c->ev_launches + 1)) {
      for (int i = 0; i < 2; ++i) {
        cudaEvent_t e;
        QC_CUDA(cudaEventCreate(&e));
        c->ev_launch.push_back(e);
      }
    }
    evl = &c->ev_launch[2 * c->ev_launches++];
    QC_CUDA(cudaEventRecord(evl[0], stream));
  }
  // (a GLA follower of the in-order schedule has nothing to sweep: its merge does everything)
  if (has_work && by_rows) QC_CUDA(launch_attend_rows(p, *row_jobs, c->ctx->n_sms, stream));
  else if (has_work) QC_CUDA(c->group > 1 ? launch_attend_tc(p, c->ctx->n_sms, stream) : launch_attend(p, c->ctx->n_sms, stream));
  if (evl) QC_CUDA(cudaEventRecord(evl[1], stream));
  if (ev && gi + 1 == c->groups.size()) QC_CUDA(cudaEventRecord(ev[2], stream));
  if (!p.fused_merge) QC_CUDA(launch_merge(p, stream));
  if (record_done) QC_CUDA(cudaEventRecord(record_done, stream));
  c->attend_launches += has_work ? 1 : 0;
  c->kernel_launches += (has_work ? 1 : 0) + (p.fused_merge ? 0 : 1);
  return QC_OK;
}

// CTAs that an output row gets in the launches of a step of the in-order schedule, and their warps, or 0: its
// launches are cut into tile ranges.  All figures are us per layer in tile ranges / by rows; * is what the rule takes.
struct RowSplit {
  int cluster, warps;
};
RowSplit row_split_of(const qc_cache* c, int32_t n_seqs, const int32_t* seq_ids) {
  const RowSplit ranges{0, 0};
  if (!c->rows_fit || c->static_partition != -1 || !c->plan_ahead || !c->fused_merge || c->row_cluster == 0 ||
      c->static_row_cost != default_row_cost(c) || c->static_min_tiles != default_min_tiles(c))
    return ranges;
  if (c->group == 1 && c->row_warps > 0) return RowSplit{1, c->row_warps};
  if (c->row_cluster > 0) return RowSplit{c->row_cluster, kAttendWarps};
  const int rows = n_seqs * c->items_per_chunk, n_sms = c->ctx->n_sms;
  const bool gla = c->cfg.lazy_mode == QC_MODE_GLA;
  int64_t pages = 0, longest = 0, pages_t = 0, longest_t = 0;   // of a row in a launch; in one that sweeps the text alone
  for (int i = 0; i < n_seqs; ++i) {
    const SeqState& st = c->seqs[seq_ids[i]];
    const int64_t t = pages_for(st.len_text), n = pages_for(st.len_vis) + t;
    pages += n;
    pages_t += t;
    longest = std::max(longest, n);
    longest_t = std::max(longest_t, t);
  }
  // A launch takes as long as its longest row: batches whose longest row is over 1.6 times the average one stay with
  // the ranges.  Without query groups that also goes for all of a step's launches together, those included in which
  // followers sweep the text alone: sequences of equal totals, one with 3 000 tokens of text and seven with 16,
  // 56.4* / 65.1 (query groups lose more to ranges: 32 of 1 500 or 16 23.9 / 22.1*).
  const int64_t text_launches = c->text_launches, launches = c->cfg.n_layers - c->no_launches - text_launches;
  const int64_t worst = launches * longest + text_launches * longest_t, all = launches * pages + text_launches * pages_t;
  if (5 * longest * n_seqs > 8 * pages || (c->group == 1 && 5 * worst * n_seqs > 8 * all)) return ranges;
  auto places = [&](int n) { return c->row_places.clusters[n == 8 ? 3 : n / 2]; };
  RowSplit split = ranges;
  int64_t most = 0;   // pages that the longest row may have more than the average one
  if (rows <= places(1)) {
    int n = 8;
    if (places(1) > n_sms) {
      // Two six-warp CTAs fit an SM (296 of them; clusters of two, four and eight 148, 71 and 33 times).  As many CTAs
      // per row as leave one CTA per SM: the next launch then starts in the other half of each SM, and its first tiles
      // have landed when this one ends.  Twice that where a warp would still have more than six pages, if they are
      // resident at once.  1, 2, 4, 8 CTAs per row:
      //   32 rows of 43 pages 9.54 / 10.2, 7.53, 6.92*, 7.74; 32 of 188 13.8 / 30.2, 17.4, 12.4, 11.6*;
      //   34 of 500 24.2 / 68.3, 37.3, 23.8*, 31.4; 128 of 43 13.0 / 11.4, 10.4*, 16.1, 27.4;
      //   256 of 188 55.5 / 52.7*, 54.6, 62.2; 256 of 130, GLA, 34.4 / 32.7*, 32.8, 36.9;
      //   64-wide, GLA, 32 of 43 7.50 / 8.0, 5.9, 5.09*, 4.94; query groups, 32 of 50 11.7 / 12.3, 9.27, 8.34*, 9.98;
      //   4 of 71 12.2 / 16.3, 11.1, 8.64, 8.07*; 52 of 131 19.3 / 25.4, 17.2, 15.4*, 23.1;
      //   72 of 190 24.4 / 33.5, 21.8*, 31.0, 38.4; 128 of 71 20.2 / 18.7, 17.8*, 24.4
      while (n > 1 && n * rows > n_sms) n /= 2;
      if (n < 8 && rows <= places(2 * n) && longest > 36 * n) n *= 2;
      // Few rows, eight CTAs each, leave SMs idle, and ranges are the better the longer the rows are.  They pay for it
      // in merges of hundreds of partials per row, most where a merge launch per layer does them (query groups, GLA):
      //   VLA, 4 of 1 000 21.7 / 21.3*, of 1 880 24.7* / 35.2; 8 of 500 17.1 / 14.1*, of 1 000 19.9 / 21.7*,
      //   of 1 880 26.4* / 35.7; 64-wide, 16 of 500 14.1 / 13.4*, of 606 15.2* / 16.8; GLA blocks of four, 8 of 1 000
      //   24.4 / 18.0*, of 1 880 29.6 / 30.6*; query groups, VLA, 4 of 1 000 45.3 / 25.1*, of 2 000 48.8 / 42.9*,
      //   of 3 760 55.8* / 74.7
      const int few = (c->D == 64 ? 600 : 1000) * (gla == (c->group > 1) ? 1 : 2);
      if (8 * rows <= n_sms && longest > few) return ranges;
      // Long rows of 64-wide heads where some SMs have two CTAs and most have one:
      //   40 of 317 15.6* / 18.1, of 660 19.2* / 24.4; 48 of 500 20.3* / 21.0, of 250 14.4 / 13.7*; 56 of 500 22.1 / 21.3*;
      //   80 of 157 13.1* / 13.3, of 313 19.0* / 20.6; 96 of 198 19.5* / 21.6; 112 of 251 22.1 / 21.1*;
      //   query groups, GLA, 80 of 366 19.2* / 24.1
      const bool most_have_one = 10 * n * rows < 7 * places(1), nearly_all = 10 * n * rows < 6 * places(1);
      if (c->D == 64 && n * rows > n_sms && most_have_one && longest > (nearly_all && c->group == 1 ? 40 : 80) * n) return ranges;
    } else {
      // Query groups of 128-wide heads with two or three followers fit an SM once (148, 74, 33 and 15 clusters).  As
      // many CTAs per row as are resident, and ranges where a row's pages are too many for them.  1, 2, 4, 8 CTAs per
      // row, blocks of four:
      //   VLA_QC, 16 of 64 13.5 / 18.6, 12.7, 10.4*, 15.5; 64 of 64 16.1 / 19.1, 13.5*, 18.4; 64 of 190 22.5* / 44.6,
      //   26.4; 128 of 21 13.6 / 11.1*, 15.1; 128 of 64 19.4* / 19.6, 23.6;
      //   GLA, 16 of 64 10.4 / 17.6, 11.7, 8.3*, 12.3, of 500 24.0* / 106, 55.8, 30.1, 33.7; 72 of 64 13.5 / 18.0,
      //   12.7*, 20.9, of 190 21.9* / 43.1, 24.7; 80 of 64 13.8* / 18.1, 21.2
      while (rows > places(n)) n /= 2;
      static constexpr int kMostPages[2][4] = {{45, 135, 300, 900}, {0, 85, 270, 900}};
      if (longest > kMostPages[gla][n == 8 ? 3 : n / 2]) return ranges;
    }
    split = RowSplit{n, kAttendWarps};
    most = c->group > 1 ? 64 : n * c->D / 4;
  } else if (c->group == 1) {
    // More rows: one CTA per row, with the most warps that leave every row resident.  6, 4, 3, 2, 1 warps:
    //   384 of 64 32.7 / 36.0, 29.0*, 30.3, 35.8, 52.9; 512 of 43 30.8 / 30.9, 32.0, 26.9*, 29.4, 38.4;
    //   480 of 17 18.3 / 18.5, 17.2, 14.4*, 16.4, 20.5; 768 of 43 43.4 / 45.3, 42.8, 49.0, 38.5*, 43.7;
    //   1 024 of 32 44.9 / 49.3, 45.4, 43.3, 46.1, 40.5*;
    //   64-wide, of which an SM holds more, 480 of 63 25.2 / 25.7, 20.2*, 23.1, 27.5, 43.8; 640 of 63 32.2 / 37.4,
    //   37.0, 25.3*, 31.0, 47.6; 900 of 63 40.8 / 48.7, 40.1, 46.8, 34.0*, 48.2
    for (int warps : {1, 2, 3, 4})
      if (rows <= n_sms * (warps == 1 ? kWorkersPerSm : c->row_places.per_sm[warps])) split = RowSplit{1, warps};
    // Beyond the eight clusters that an SM holds, long rows: 1 280 of 32 42.2 / 39.3*, of 63 78.3 / 77.6*, of 80 131* / 141.
    if (rows > 8 * n_sms && longest > 64) return ranges;
    // Up to there one warp per row is for rows of one length: 1 024 of 0.4 to 1 times 38 41.7 / 45.0, 40.4, 40.7*, 40.5,
    // 43.3 (beyond it blocks of three run in a third wave: 1 280 of 4 to 6 20.6 / 27.7, 21.3, 19.2, 16.4, 15.7*).
    if (split.warps == 1 && rows <= 8 * n_sms && 20 * longest * n_seqs > 23 * pages) split.warps = 3;
    // 64-wide again, long rows that leave much of the chip's warps without work: 320 of 134 36.7* / 43.0.
    if (c->D == 64 && split.warps > 1 && 10 * rows < 7 * n_sms * c->row_places.per_sm[split.warps] && longest > 80) return ranges;
    // A few warps are a long way through text that half of the batch does not have: 600 rows of 115 or 4 pages 84.2* / 104,
    // 320 of 81 or 7, blocks of four, 36.5* / 44.2, 512 of 94 or 3, blocks of four, 60.3* / 66.9.
    if (text_launches > 0 && longest_t * n_seqs - pages_t > 25 * n_seqs) return ranges;
    most = c->D == 64 ? 25 : 50;
  }
  // Rows that are longer than the average one by more pages than a launch's start and end are worth: 32 for each
  // six-warp CTA of a row and 50 for rows of fewer warps (half of these for 64-wide heads), 64 for query groups.  By how many:
  //   256 of 188 31 45.5 / 44.8*; 240 of 251 38 68.4* / 70.3, 64 61.3* / 66.2; 480 of 251 35 86.3 / 82.6*, 58 78.1* / 78.6;
  //   384 of 188 42 61.3 / 58.8*; 64-wide, 240 of 251 46 33.2* / 34.9, 112 of 501 74 32.4* / 35.4; query groups, 240 of
  //   251 62 58.2 / 57.2*, 80 of 251 41 27.8 / 27.8*, 69 26.1* / 27.6; followers' text, 224 of 251 60 68.9* / 76.2, 64-wide
  //   query groups, 40 of 552 164 27.2* / 34.0
  if (worst * n_seqs - all > most * n_seqs * (launches + text_launches)) return ranges;
  return split;
}

int decode_step_core(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const void* q_dev, const void* k_dev,
                     const void* v_dev, void* out_dev, float* lse_out_dev, const HostPipe* pipe,
                     bool open_only = false) {
  if (!c || n_seqs < 0 || (n_seqs > 0 && !seq_ids)) return QC_ERR_INVALID_ARG;
  if (c->open.active) return QC_ERR_STATE;   // a step opened by qc_decode_begin has layers left
  if (n_seqs == 0) return open_only ? QC_ERR_INVALID_ARG : QC_OK;
  if (!open_only && (!q_dev || !k_dev || !v_dev || !out_dev)) return QC_ERR_INVALID_ARG;
  if (n_seqs > c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
  const void* ptrs[4] = {q_dev, k_dev, v_dev, out_dev};
  for (const void* ptr : ptrs)
    if (reinterpret_cast<uintptr_t>(ptr) & 15) return QC_ERR_INVALID_ARG;
  if (const int32_t dev_err = *static_cast<volatile int32_t*>(c->err_host)) return dev_err;   // an earlier kernel gave up
  const int N = c->cfg.n_layers;
  // ---- validate, count pages
  int64_t need = 0;
  {
    std::vector<uint8_t> seen(c->cfg.max_seqs, 0);
    for (int i = 0; i < n_seqs; ++i) {
      const int s = seq_ids[i];
      if (s < 0 || s >= c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
      if (!c->seqs[s].active || seen[s]) return QC_ERR_STATE;
      seen[s] = 1;
      if (c->seqs[s].len_text + 1 > c->cfg.max_tokens_per_seq) return QC_ERR_INVALID_ARG;
      if (c->paged && c->seqs[s].len_text % kPage == 0) need += c->text_streams_per_seq;
    }
  }
  if (c->paged && need > static_cast<int64_t>(c->free_stack.size())) return QC_ERR_OOM_PAGES;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  cudaStream_t stream = c->ctx->stream;

  const int want_per = open_only ? -2 : (pipe ? pipe->per_launch : c->layers_per_launch);
  if (c->plan_dirty || c->plan_per != want_per) {
    const int st = rebuild_plan(c, want_per);
    if (st != QC_OK) return st;
  }

  // ---- page planning (sequence -> layer -> K_T, V_T) and lengths
  std::vector<Patch> patches;
  for (int i = 0; i < n_seqs; ++i) {
    const int s = seq_ids[i];
    SeqState& st = c->seqs[s];
    if (c->paged && st.len_text % kPage == 0) {
      const int have = st.len_text / kPage;
      for (int l = 0; l < N; ++l) {
        if (owns(c, l, QC_STREAM_K_TEXT)) grow_stream(c, l, QC_STREAM_K_TEXT, s, have, 1, &patches);
        grow_stream(c, l, QC_STREAM_V_TEXT, s, have, 1, &patches);
      }
    }
    st.len_text += 1;
  }
  const int n_patches = static_cast<int>(patches.size());
  if (c->auto_split) {
    // Larger chunks mean fewer partial results to write and merge; smaller chunks mean more work items to balance
    // over the workers.  Take the largest chunk whose heaviest item is small against a worker's share of the launch: a
    // third of it, half where no stream is cut.  us per layer, with five items per worker asked for as before -> now:
    //   a step in one launch: 16 sequences of 677 tokens, 8 layers 30.1 -> 26.3; 24 of them 42.0 -> 37.8; 30 of 260,
    //   16 heads 14.0 -> 12.6; long steps as before;
    //   a launch per lazy block / per two / per four: 16 of 3 000 100.4 -> 98.2 / 92.1 -> 93.1 / 88.1 -> 88.3, in GLA
    //   blocks of four 75.4 -> 75.3 / 74.7 -> 75.3 / 72.2 -> 72.3; 8 of 4 100, VLA_EQ8, 65.8 / 63.9 / 60.7, no difference.
    // With query groups five items per worker (longer chunks were 4 to 17 % faster where a step has less, 13 sequences
    // of 2 100 tokens 11.0 -> 9.5, but have fewer weights that bf16 holds exactly: the error against 64 bits grows).
    // One and a half items per worker when it is one launch per layer (a short launch's partial rows and their merge
    // weigh more than the balance of its tail; 1, 2 and 3 were measured too).  With several launches per step, a long
    // stream cut small also means many partial rows per output row for every one of those launches' merges: beyond 24
    // rows the chunk is doubled as long as one and a half items per worker remain.
    const int64_t workers = static_cast<int64_t>(c->ctx->n_sms) * kWorkersPerSm * static_cast<int64_t>(c->groups.size());
    auto items_at = [&](int cp, int* max_slots) {
      int64_t cv = 0, ct = 0;
      int slots = 0;
      for (int i = 0; i < n_seqs; ++i) {
        const SeqState& st = c->seqs[seq_ids[i]];
        const int v = (pages_for(st.len_vis) + cp - 1) / cp, t = (pages_for(st.len_text) + cp - 1) / cp;
        cv += v;
        ct += t;
        slots = std::max(slots, v + t);
      }
      if (max_slots) *max_slots = slots;
      return (cv * c->n_visual_jobs + ct * c->n_text_jobs) * c->items_per_chunk;
    };
    const int64_t twice_per_worker = c->plan_per < 0 ? 3 : 10;
    // (a query group writes one partial row per head and chunk: its chunks stay at 128 keys or more)
    const int floor_pages = c->group > 1 ? std::max(c->min_chunk_pages, 8) : c->min_chunk_pages;
    int64_t work = 0;   // tiles of the step
    int longest_v = 0, longest_t = 0, w_v = 0, w_t = 0;
    for (int i = 0; i < n_seqs; ++i) {
      const SeqState& st = c->seqs[seq_ids[i]];
      const int v = pages_for(st.len_vis), t = pages_for(st.len_text);
      work += (v * c->visual_row_reads + t * c->text_row_reads) * c->items_per_chunk;
      longest_v = std::max(longest_v, v);
      longest_t = std::max(longest_t, t);
    }
    for (const LaunchGroup& g : c->groups) {
      w_v = std::max(w_v, g.w_max_v);
      w_t = std::max(w_t, g.w_max_t);
    }
    auto balanced = [&](int cp) {
      const int64_t heaviest = std::max(w_v * std::min(cp, longest_v), w_t * std::min(cp, longest_t));
      return work >= (cp >= std::max(longest_v, longest_t) ? 2 : 3) * heaviest * workers;
    };
    int pick = floor_pages;
    for (int cp = kMaxChunkPages; cp > floor_pages; cp /= 2) {
      if (c->plan_per < 0 || c->group > 1 ? 2 * items_at(cp, nullptr) >= twice_per_worker * workers : balanced(cp)) {
        pick = cp;
        break;
      }
    }
    if (c->groups.size() > 1) {
      int slots = 0;
      items_at(pick, &slots);
      while (slots > 24 && pick * 2 <= kMaxChunkPages && 2 * items_at(pick * 2, nullptr) >= 3 * workers) {
        pick *= 2;
        items_at(pick, &slots);
      }
    }
    c->chunk_pages = pick;
  }

  // ---- step descriptors: as a kernel argument when they are small and no page table entry
  // changes, otherwise through a pinned slot and one copy
  const bool inline_step = n_seqs <= kInlineSeqs && n_patches == 0;
  StepInline inl;
  StepSeq* h_seqs = inl.seqs;
  int slot = -1;
  uint8_t* hb = nullptr;
  if (!inline_step) {
    slot = c->stage_next;
    c->stage_next = (c->stage_next + 1) % kStageSlots;
    if (c->stage_used[slot]) QC_CUDA(cudaEventSynchronize(c->stage_done[slot]));   // its last copy must have run
    hb = c->pinned + static_cast<size_t>(slot) * c->lay.step_bytes;
    h_seqs = reinterpret_cast<StepSeq*>(hb + c->lay.step_seqs);
    if (n_patches) std::memcpy(hb + c->lay.step_patches, patches.data(), n_patches * sizeof(Patch));
  }
  // Static partition: the step's launches cut their work into equal ranges instead of claiming
  // items (by default whenever a step is several launches, whose short tails a few large items
  // per worker would dominate).
  bool use_static = c->static_partition == 1 || (c->static_partition < 0 && c->groups.size() > 1);
  int64_t tp_v = 0, tp_t = 0;                     // pages of the visual / text streams over the listed sequences
  int pmax_v = 0, pmax_t = 0;
  for (int i = 0; i < n_seqs; ++i) {
    const SeqState& st = c->seqs[seq_ids[i]];
    const int pv = pages_for(st.len_vis), pt = pages_for(st.len_text);
    tp_v += pv;
    tp_t += pt;
    pmax_v = std::max(pmax_v, pv);
    pmax_t = std::max(pmax_t, pt);
  }
  // Static ranges pay off for launches that leave a worker one or two ranges' worth of tiles (a
  // launch per layer or per lazy block); on larger launches claimed 512-key items were measured
  // faster (config 2, five blocks per launch: 0.89 against 1.05 ms per step; two blocks: 1.04
  // against 1.12).  Tile offsets are 32-bit.
  if (c->static_partition < 0) {
    const int64_t workers = static_cast<int64_t>(c->ctx->n_sms) * kWorkersPerSm;
    for (const LaunchGroup& g : c->groups) {
      const int64_t tiles = static_cast<int64_t>(c->items_per_chunk) * (g.wv * tp_v + g.wt * tp_t);
      if (tiles > workers * 60 * std::max(1, g.w_min)) use_static = false;
    }
  }
  for (const LaunchGroup& g : c->groups)
    if (static_cast<int64_t>(c->items_per_chunk) * (g.wv * tp_v + g.wt * tp_t + 64LL * n_seqs * (g.job_end - g.job_begin)) >= (1LL << 31))
      use_static = false;
  int64_t tot_v = 0, tot_t = 0, step_rows = 0;   // step_rows: K/V rows the step has to read (for the profile)
  int64_t pre_pv = 0, pre_pt = 0;
  for (int i = 0; i < n_seqs; ++i) {
    const int s = seq_ids[i];
    const SeqState& st = c->seqs[s];
    const int pv = pages_for(st.len_vis), pt = pages_for(st.len_text);
    const int ncv = (pv + c->chunk_pages - 1) / c->chunk_pages;
    const int nct = (pt + c->chunk_pages - 1) / c->chunk_pages;
    h_seqs[i] = StepSeq{s, st.len_text, st.len_vis, ncv + nct, static_cast<int32_t>(use_static ? pre_pv : tot_v),
                        static_cast<int32_t>(use_static ? pre_pt : tot_t), ncv, 0};
    tot_v += static_cast<int64_t>(ncv) * c->items_per_chunk;
    tot_t += static_cast<int64_t>(nct) * c->items_per_chunk;
    pre_pv += pv;
    pre_pt += pt;
    step_rows += st.len_vis * c->visual_row_reads + st.len_text * c->text_row_reads;
  }
  const int n_pos = static_cast<int>(c->plan.size());
  const int64_t n_items64 = c->plan_vis_before[n_pos] * tot_v + c->plan_text_before[n_pos] * tot_t;
  const int n_items = use_static ? 0 : static_cast<int>(n_items64);   // <= max_items: the item list was sized at allocation

  // ---- enqueue
  if (!inline_step) {
    QC_CUDA(cudaMemcpyAsync(c->ws + c->lay.step, hb, c->lay.step_bytes, cudaMemcpyHostToDevice, stream));
    QC_CUDA(cudaEventRecord(c->stage_done[slot], stream));
    c->stage_used[slot] = true;
  }

  Params p = base_params(c);
  p.q = static_cast<const uint16_t*>(q_dev);
  p.k = static_cast<const uint16_t*>(k_dev);
  p.v = static_cast<const uint16_t*>(v_dev);
  p.out = static_cast<uint16_t*>(out_dev);
  p.lse = lse_out_dev;
  p.n_seqs = n_seqs;
  p.n_pos = use_static ? 0 : n_pos;   // static ranges need no item list
  p.n_items = n_items;
  p.part_static = use_static ? 1 : 0;
  p.n_patches = n_patches;
  p.tot_v = static_cast<int32_t>(tot_v);
  p.tot_t = static_cast<int32_t>(tot_t);
  p.inline_seqs = inline_step ? 1 : 0;
  // the append reads the page table (not beside its patches) and every layer's k/v (not before
  // the host pipe has copied them)
  // in-order schedule: nothing of a layer is touched before its own launch (the worker that meets
  // the end of the layer's text stream takes the new rows from the inputs and stores them)
  const bool fold = want_per == -2 && c->fold_append;
  p.fold_append = fold ? 1 : 0;
  p.fused_append = (n_patches == 0 && !pipe && !open_only && !fold) ? 1 : 0;

  // Few output rows: a cluster of CTAs for each, if the options leave the schedule as it comes.
  const RowSplit by_rows = fold && use_static ? row_split_of(c, n_seqs, seq_ids) : RowSplit{0, 0};
  p.row_cluster = by_rows.cluster;
  p.row_warps = by_rows.warps;
  const bool planned = use_static && p.row_cluster == 0 && c->plan_ahead && c->groups.size() <= static_cast<size_t>(kMaxPlanLaunches) &&
                       c->groups.size() <= static_cast<size_t>(std::min(c->cfg.n_layers, kMaxPlanLaunches)) &&
                       c->ctx->n_sms * kWorkersPerSm <= kPlanWorkers;
  // static partition of every launch of the step (part_workers == 0: the launch has nothing to sweep)
  auto partition_of = [&](size_t gi) {
    const LaunchGroup& g = c->groups[gi];
    const int pb = c->group_pos[gi].first, pe = c->group_pos[gi].second;
    LaunchDesc L{};
    L.pos_begin = pb;
    L.pos_end = pe;
    L.part_row_cost = c->static_row_cost;
    L.layer = -1;
    if (planned && g.layer_end - g.layer_begin == 1) {
      L.layer = g.layer_begin;
      bool vis = false, text = false;   // swept here?
      for (int pos = pb; pos < pe; ++pos) (c->plan[pos].job.stream ? vis : text) = true;
      L.vis_launch = vis ? static_cast<int32_t>(gi) : c->leader[L.layer];
      L.text_launch = text ? static_cast<int32_t>(gi) : c->leader[L.layer];
    }
    const int64_t kv_tiles = static_cast<int64_t>(c->items_per_chunk) * (g.wv * tp_v + g.wt * tp_t);
    if (kv_tiles <= 0) return L;
    const int64_t T = kv_tiles + static_cast<int64_t>(c->items_per_chunk) * c->static_row_cost * n_seqs * (pe - pb);
    // tiles per page of the lightest / heaviest job that has any page, longest row in tiles
    const int w_min = (tp_v > 0 && tp_t > 0) ? g.w_min : g.w_max_v * (tp_v > 0) + g.w_max_t * (tp_t > 0);
    const int w_lo = std::max(1, std::min(w_min, g.w_min));
    const int64_t row_max = std::max<int64_t>(static_cast<int64_t>(pmax_v) * g.w_max_v,
                                              static_cast<int64_t>(pmax_t) * g.w_max_t);
    const int64_t q_max = 30LL * w_lo;
    // at least a page of the heaviest job, with query groups two (each of a row's pieces then is seven or
    // eight partial rows to merge: batch 1, 160 launches: one page 2.93 ms, two 2.45; batch 8 2.36 / 2.06)
    int64_t q_min = std::max<int64_t>(c->group > 1 ? 2 * g.w_max : g.w_max,
                                      (row_max + c->slots_per_stream - 3) / (c->slots_per_stream - 2));
    q_min = std::max<int64_t>(q_min, std::min<int64_t>(c->static_min_tiles, q_max / 2));
    const int64_t W = static_cast<int64_t>(c->ctx->n_sms) * kWorkersPerSm;
    int64_t k = 1, q;
    if (T > W * q_max) {   // several ranges per worker, each as long as a piece may be
      k = (T + W * q_max - 1) / (W * q_max);
      q = (T + W * k - 1) / (W * k);
    } else {
      q = std::max<int64_t>(q_min, (T + W - 1) / W);
    }
    const int64_t vw = (T + q - 1) / q;
    L.part_vw = static_cast<int32_t>(vw);
    L.part_k = static_cast<int32_t>(k);
    L.part_workers = static_cast<int32_t>((vw + k - 1) / k);
    L.part_q = static_cast<int32_t>(q);
    // few workers are spread over the chip rather than packed into few CTAs (batch 1: 13.2 against 13.5 ms)
    const int n_ctas = c->ctx->n_sms * kAttendCtasPerSm;
    L.part_wpc = std::min(kAttendWarps, std::max(1, (L.part_workers + n_ctas - 1) / n_ctas));
    L.part_wv = g.wv;
    L.part_wt = g.wt;
    // Who merges the rows of a launch of one layer.  With one query head per row and at most two rows per
    // CTA (592) the launch itself: 8 layers, time with its own merge over time with a merge launch, rows of 140 / 280 /
    // 600 / 1 200 keys: 64 rows 1.04 / 0.94 / 0.89 / 0.87, 224 rows 0.99 / 0.97 / 0.96 / 0.97, 480 rows 0.99 / 0.98 / 0.99 / 1.00,
    // 576 rows 0.99 / 0.99 / 0.99 / 1.00.  With query groups, whose every partial is seven or eight rows, a merge
    // launch over the whole chip (896 launches at batch 32: 19.1, the other way 20.4).
    if (L.layer >= 0 && c->fused_merge && c->group == 1 && static_cast<int64_t>(n_seqs) * c->hq <= 2LL * n_ctas)
      L.fused_merge = (L.part_workers + L.part_wpc - 1) / L.part_wpc <= kPlanCtas;
    return L;
  };
  LaunchList launches;
  if (use_static && p.row_cluster == 0)
    for (size_t gi = 0; gi < c->groups.size() && gi < static_cast<size_t>(kMaxPlanLaunches); ++gi)
      launches.launch[gi] = partition_of(gi);
  p.wdesc = planned ? reinterpret_cast<const WorkerDesc*>(c->ws + c->lay.wdesc) : nullptr;

  cudaEvent_t* ev = nullptr;
  if (c->profile && !open_only && c->ev_steps < kMaxProfileSteps) {
    if (static_cast<int>(c->ev.size()) < 4 * (c->ev_steps + 1)) {
      for (int i = 0; i < 4; ++i) {
        cudaEvent_t e;
        QC_CUDA(cudaEventCreate(&e));
        c->ev.push_back(e);
      }
    }
    ev = &c->ev[4 * c->ev_steps];
    QC_CUDA(cudaEventRecord(ev[0], stream));
  }
  QC_CUDA(launch_setup(p, inline_step ? &inl : nullptr, stream));
  c->kernel_launches++;
  if (!p.fused_append && !pipe && !open_only && !fold) {
    p.layer_begin = 0;
    p.layer_end = N;
    QC_CUDA(launch_append(p, stream));
    c->kernel_launches++;
  }
  if (planned) {
    QC_CUDA(launch_plan(p, launches, static_cast<int>(c->groups.size()), stream));
    c->kernel_launches++;
  }
  if (open_only) {   // qc_decode_begin: the launches follow layer by layer (qc_decode_layer)
    OpenStep& o = c->open;
    o.p = p;
    o.launches = launches;
    o.use_static = use_static;
    o.tot_v = tot_v;
    o.tot_t = tot_t;
    o.next_layer = 0;
    o.bytes = step_rows * c->hkv * c->D * 2;
    o.active = true;
    return QC_OK;
  }
  for (size_t gi = 0; gi < c->groups.size(); ++gi) {
    const int st = run_group(c, p, gi, launches, use_static, tot_v, tot_t, pipe != nullptr,
                             pipe ? pipe->in[gi] : nullptr, pipe ? pipe->done[gi] : nullptr, ev, stream);
    if (st != QC_OK) return st;
  }
  if (ev) {
    QC_CUDA(cudaEventRecord(ev[3], stream));
    c->ev_steps++;
    c->prof_bytes += step_rows * c->hkv * c->D * 2;
    c->prof_items += n_items;
  }
  c->decode_steps++;
  c->kv_bytes_swept += step_rows * c->hkv * c->D * 2;
  return QC_OK;
}

}  // namespace

extern "C" {

int32_t qc_decode_step(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const void* q_dev, const void* k_dev,
                       const void* v_dev, void* out_dev, float* lse_out_dev) {
  return decode_step_core(c, n_seqs, seq_ids, q_dev, k_dev, v_dev, out_dev, lse_out_dev, nullptr);
}

int32_t qc_decode_begin(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids) {
  return decode_step_core(c, n_seqs, seq_ids, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, true);
}

int32_t qc_decode_layer(qc_cache* c, int32_t layer, const void* q_dev, const void* k_dev, const void* v_dev,
                        void* out_dev, float* lse_out_dev) {
  if (!c || !q_dev || !k_dev || !v_dev || !out_dev) return QC_ERR_INVALID_ARG;
  const void* ptrs[4] = {q_dev, k_dev, v_dev, out_dev};
  for (const void* ptr : ptrs)
    if (reinterpret_cast<uintptr_t>(ptr) & 15) return QC_ERR_INVALID_ARG;
  OpenStep& o = c->open;
  if (!o.active || layer != o.next_layer) return QC_ERR_STATE;
  if (const int32_t dev_err = *static_cast<volatile int32_t*>(c->err_host)) return dev_err;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  // the kernels index a step's tensors as [layer][sequence]...: hand them this layer's slices at that place
  Params p = o.p;
  const uintptr_t q_off = static_cast<uintptr_t>(layer) * p.n_seqs * c->hq * c->D * 2;
  const uintptr_t kv_off = static_cast<uintptr_t>(layer) * p.n_seqs * c->hkv * c->D * 2;
  p.q = reinterpret_cast<const uint16_t*>(reinterpret_cast<uintptr_t>(q_dev) - q_off);
  p.k = reinterpret_cast<const uint16_t*>(reinterpret_cast<uintptr_t>(k_dev) - kv_off);
  p.v = reinterpret_cast<const uint16_t*>(reinterpret_cast<uintptr_t>(v_dev) - kv_off);
  p.out = reinterpret_cast<uint16_t*>(reinterpret_cast<uintptr_t>(out_dev) - q_off);
  p.lse = lse_out_dev ? reinterpret_cast<float*>(reinterpret_cast<uintptr_t>(lse_out_dev) -
                                                  static_cast<uintptr_t>(layer) * p.n_seqs * c->hq * sizeof(float))
                      : nullptr;
  const int st = run_group(c, p, static_cast<size_t>(layer), o.launches, o.use_static, o.tot_v, o.tot_t,
                           !p.fold_append, nullptr, nullptr, nullptr, c->ctx->stream);
  if (st != QC_OK) return st;
  if (++o.next_layer == c->cfg.n_layers) {
    o.active = false;
    c->decode_steps++;
    c->kv_bytes_swept += o.bytes;
  }
  return QC_OK;
}

int32_t qc_decode_step_host(qc_cache* c, int32_t n_seqs, const int32_t* seq_ids, const void* q_host,
                            const void* k_host, const void* v_host, void* out_host, float* lse_out_host) {
  if (!c || n_seqs < 0) return QC_ERR_INVALID_ARG;
  if (n_seqs == 0) return QC_OK;
  if (!q_host || !k_host || !v_host || !out_host || n_seqs > c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  cudaStream_t stream = c->ctx->stream;
  // The step runs as up to four launch groups of consecutive lazy blocks: while one group
  // computes, the inputs of the next are copied in and the outputs of the previous copied out.
  // (a small step is not worth cutting up: one group)
  const int nb = static_cast<int>(c->block_jobs.size());
  const size_t in_bytes = static_cast<size_t>(c->cfg.n_layers) * n_seqs * (c->hq + 2 * c->hkv) * c->D * 2;
  const int per = in_bytes < (1u << 20) ? nb : (nb + 3) / 4;
  if (c->plan_dirty || c->plan_per != per) {
    const int st = rebuild_plan(c, per);
    if (st != QC_OK) return st;
  }
  const size_t G = c->groups.size();
  if (!c->copy_in) {
    QC_CUDA(cudaStreamCreateWithFlags(&c->copy_in, cudaStreamNonBlocking));
    QC_CUDA(cudaStreamCreateWithFlags(&c->copy_out, cudaStreamNonBlocking));
  }
  while (c->ev_in.size() < G) {
    cudaEvent_t a, b;
    QC_CUDA(cudaEventCreateWithFlags(&a, cudaEventDisableTiming));
    QC_CUDA(cudaEventCreateWithFlags(&b, cudaEventDisableTiming));
    c->ev_in.push_back(a);
    c->ev_done.push_back(b);
  }
  const size_t q_layer = static_cast<size_t>(n_seqs) * c->hq * c->D * 2;    // bytes of one layer's q (and out)
  const size_t kv_layer = static_cast<size_t>(n_seqs) * c->hkv * c->D * 2;
  const size_t lse_layer = static_cast<size_t>(n_seqs) * c->hq * sizeof(float);
  uint8_t* dq = c->ws + c->lay.stage_q;
  uint8_t* dk = c->ws + c->lay.stage_k;
  uint8_t* dv = c->ws + c->lay.stage_v;
  uint8_t* dout = c->ws + c->lay.stage_out;
  uint8_t* dlse = c->ws + c->lay.stage_lse;
  const uint8_t* hq = static_cast<const uint8_t*>(q_host);
  const uint8_t* hk = static_cast<const uint8_t*>(k_host);
  const uint8_t* hv = static_cast<const uint8_t*>(v_host);
  for (size_t g = 0; g < G; ++g) {
    const size_t lb = c->groups[g].layer_begin, nl = c->groups[g].layer_end - lb;
    QC_CUDA(cudaMemcpyAsync(dq + lb * q_layer, hq + lb * q_layer, nl * q_layer, cudaMemcpyHostToDevice, c->copy_in));
    QC_CUDA(cudaMemcpyAsync(dk + lb * kv_layer, hk + lb * kv_layer, nl * kv_layer, cudaMemcpyHostToDevice, c->copy_in));
    QC_CUDA(cudaMemcpyAsync(dv + lb * kv_layer, hv + lb * kv_layer, nl * kv_layer, cudaMemcpyHostToDevice, c->copy_in));
    QC_CUDA(cudaEventRecord(c->ev_in[g], c->copy_in));
  }
  const HostPipe pipe{per, c->ev_in.data(), c->ev_done.data()};
  const int st = decode_step_core(c, n_seqs, seq_ids, dq, dk, dv, dout,
                                  lse_out_host ? reinterpret_cast<float*>(dlse) : nullptr, &pipe);
  if (st != QC_OK) {
    cudaStreamSynchronize(c->copy_in);
    cudaStreamSynchronize(stream);
    return st;
  }
  for (size_t g = 0; g < G; ++g) {
    const size_t lb = c->groups[g].layer_begin, nl = c->groups[g].layer_end - lb;
    QC_CUDA(cudaStreamWaitEvent(c->copy_out, c->ev_done[g], 0));
    QC_CUDA(cudaMemcpyAsync(static_cast<uint8_t*>(out_host) + lb * q_layer, dout + lb * q_layer, nl * q_layer,
                            cudaMemcpyDeviceToHost, c->copy_out));
    if (lse_out_host)
      QC_CUDA(cudaMemcpyAsync(reinterpret_cast<uint8_t*>(lse_out_host) + lb * lse_layer, dlse + lb * lse_layer,
                              nl * lse_layer, cudaMemcpyDeviceToHost, c->copy_out));
  }
  QC_CUDA(cudaStreamSynchronize(c->copy_out));
  QC_CUDA(cudaStreamSynchronize(stream));
  return QC_OK;
}

int32_t qc_free_seq(qc_cache* c, int32_t seq_id) {
  if (!c || seq_id < 0 || seq_id >= c->cfg.max_seqs) return QC_ERR_INVALID_ARG;
  SeqState& st = c->seqs[seq_id];
  if (!st.active || c->open.active) return QC_ERR_STATE;
  if (c->paged) {
    for (auto it = st.alloc_order.rbegin(); it != st.alloc_order.rend(); ++it) c->free_stack.push_back(*it);
    for (int l = 0; l < c->cfg.n_layers; ++l)
      for (int sm = 0; sm < 4; ++sm) {
        const size_t r = trow(c, l, sm, seq_id);
        std::fill(c->table.begin() + r, c->table.begin() + r + c->max_pages, -1);
      }
  }
  st = SeqState();
  return QC_OK;
}

int32_t qc_get_stats(qc_cache* c, qc_stats* out) {
  if (!c || !out) return QC_ERR_INVALID_ARG;
  std::memset(out, 0, sizeof(*out));
  const int N = c->cfg.n_layers;
  const int64_t row = static_cast<int64_t>(c->hkv) * c->D * 2;
  out->page_bytes = row * kPage;
  out->pages_total = c->n_pool_pages;
  int64_t rows = 0, rows_full = 0, pages = 0, pages_full = 0;
  for (const SeqState& st : c->seqs) {
    if (!st.active) continue;
    out->n_active_seqs++;
    for (int l = 0; l < N; ++l)
      for (int sm = 0; sm < 4; ++sm) {
        const int len = (sm & 1) ? st.len_vis : st.len_text;
        if (owns(c, l, sm)) {
          rows += len;
          pages += pages_for(len);
        }
        rows_full += len;
        pages_full += pages_for(len);
      }
  }
  out->pages_in_use = c->paged ? c->n_pool_pages - static_cast<int64_t>(c->free_stack.size()) : pages;
  out->kv_bytes_stored = rows * row;
  out->kv_bytes_all_full = rows_full * row;
  out->kv_bytes_stored_paged = pages * out->page_bytes;
  out->kv_bytes_all_full_paged = pages_full * out->page_bytes;
  out->qcache_bytes = static_cast<int64_t>(N) * c->cfg.max_seqs * c->hq * c->D * 2;
  out->decode_steps = c->decode_steps;
  out->attend_launches = c->attend_launches;
  out->kernel_launches = c->kernel_launches;
  out->kv_bytes_swept = c->kv_bytes_swept;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  int32_t err = 0;
  QC_CUDA(cudaMemcpyAsync(&err, c->ws + c->lay.err, sizeof(err), cudaMemcpyDeviceToHost, c->ctx->stream));
  QC_CUDA(cudaStreamSynchronize(c->ctx->stream));
  out->device_error = err;
  return QC_OK;
}

int32_t qc_debug_page_table(const qc_cache* c, int32_t layer, int32_t stream, int32_t seq_id, int32_t* page_ids,
                            int32_t cap, int32_t* n_pages, int32_t* n_tokens, int32_t* owner_layer) {
  if (!c || layer < 0 || layer >= c->cfg.n_layers || stream < 0 || stream > 3 || seq_id < 0 ||
      seq_id >= c->cfg.max_seqs || cap < 0 || (cap > 0 && !page_ids))
    return QC_ERR_INVALID_ARG;
  const SeqState& st = c->seqs[seq_id];
  int owner = -1, np = 0, nt = 0;
  if (st.active) {
    owner = owns(c, layer, stream) ? layer : c->leader[layer];
    nt = (stream & 1) ? st.len_vis : st.len_text;
    np = pages_for(nt);
    const size_t r = trow(c, owner, stream, seq_id);
    for (int i = 0; i < np && i < cap; ++i) page_ids[i] = c->table[r + i];
  }
  if (n_pages) *n_pages = np;
  if (n_tokens) *n_tokens = nt;
  if (owner_layer) *owner_layer = owner;
  return QC_OK;
}

int32_t qc_debug_read_qcache(qc_cache* c, int32_t layer, void* host_bf16) {
  if (!c || !host_bf16 || layer < 0 || layer >= c->cfg.n_layers) return QC_ERR_INVALID_ARG;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  const size_t bytes = static_cast<size_t>(c->cfg.max_seqs) * c->hq * c->D * 2;
  const uint8_t* src = c->ws + c->lay.qcache + static_cast<size_t>(c->leader[layer]) * bytes;
  QC_CUDA(cudaMemcpyAsync(host_bf16, src, bytes, cudaMemcpyDeviceToHost, c->ctx->stream));
  return sync_and_check(c);
}

int32_t qc_debug_read_row(qc_cache* c, int32_t layer, int32_t stream, int32_t seq_id, int32_t token,
                          int32_t kv_head, void* host_bf16) {
  if (!c || !host_bf16 || layer < 0 || layer >= c->cfg.n_layers || stream < 0 || stream > 3 || seq_id < 0 ||
      seq_id >= c->cfg.max_seqs || kv_head < 0 || kv_head >= c->hkv)
    return QC_ERR_INVALID_ARG;
  const SeqState& st = c->seqs[seq_id];
  if (!st.active) return QC_ERR_STATE;
  const int len = (stream & 1) ? st.len_vis : st.len_text;
  if (token < 0 || token >= len) return QC_ERR_INVALID_ARG;
  const int owner = owns(c, layer, stream) ? layer : c->leader[layer];
  const int32_t pid = c->table[trow(c, owner, stream, seq_id) + token / kPage];
  if (pid < 0 || pid >= c->n_pool_pages) return QC_ERR_STATE;
  const size_t off = ((static_cast<size_t>(pid) * c->hkv + kv_head) * kPage + token % kPage) * c->D;
  QC_CUDA(cudaSetDevice(c->ctx->device));
  QC_CUDA(cudaMemcpyAsync(host_bf16, c->pool + off, c->D * 2, cudaMemcpyDeviceToHost, c->ctx->stream));
  return sync_and_check(c);
}

int32_t qc_set_option(qc_cache* c, const char* key, int64_t value) {
  if (!c || !key) return QC_ERR_INVALID_ARG;
  const std::string k(key);
  if (k == "split_tokens") {
    if (value == 0) {   // back to the per-step choice
      c->auto_split = true;
      return QC_OK;
    }
    if (value % 16 || value < 16 || value > 16 * kMaxChunkPages) return QC_ERR_INVALID_ARG;
    const int cp = static_cast<int>(value / 16);
    if (cp < c->min_chunk_pages) return QC_ERR_INVALID_ARG;   // the workspace was sized for the initial split
    c->chunk_pages = cp;
    c->auto_split = false;
    return QC_OK;
  }
  if (k == "layers_per_launch") {
    if (value < 0 || value > c->cfg.n_layers) return QC_ERR_INVALID_ARG;
    c->layers_per_launch = static_cast<int>(value);
    c->plan_dirty = true;
    return QC_OK;
  }
  if (k == "per_layer_logit_cache") {   // one launch per layer; followers take shared scores from the logit cache
    c->layers_per_launch = value ? -1 : 0;
    c->plan_dirty = true;
    return QC_OK;
  }
  if (k == "in_order_launches") {   // one launch per layer; a leader's launch also sweeps its followers' cached V
    c->layers_per_launch = value ? -2 : 0;
    c->plan_dirty = true;
    return QC_OK;
  }
  if (k == "fused_merge") {   // 0: partial rows are merged by a launch of their own
    c->fused_merge = value != 0;
    return QC_OK;
  }
  if (k == "static_partition") {
    if (value < -1 || value > 1) return QC_ERR_INVALID_ARG;
    c->static_partition = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "debug_drop_tile") {   // test hook, see qc.h
    c->debug_drop_tile = value != 0;
    return QC_OK;
  }
  if (k == "fold_append") {
    c->fold_append = value != 0;
    return QC_OK;
  }
  if (k == "plan_ahead") {
    c->plan_ahead = value != 0;
    return QC_OK;
  }
  if (k == "row_warps") {
    if (value != 0 && value != 1 && value != 2 && value != 3 && value != 4 && value != 6) return QC_ERR_INVALID_ARG;
    c->row_warps = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "row_cluster") {
    if (value < -1 || value > 8) return QC_ERR_INVALID_ARG;
    c->row_cluster = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "static_row_cost") {
    if (value < 0 || value > 64) return QC_ERR_INVALID_ARG;
    c->static_row_cost = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "static_min_tiles") {
    if (value < 1 || value > 4096) return QC_ERR_INVALID_ARG;
    c->static_min_tiles = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "prefill_shared_scores") {
    if (value < 0 || value > 2) return QC_ERR_INVALID_ARG;
    c->prefill_shared = static_cast<int>(value);
    return QC_OK;
  }
  if (k == "prefill_pair_min_tokens") {
    if (value < 0) return QC_ERR_INVALID_ARG;
    c->prefill_pair_min_tokens = static_cast<int>(std::min<int64_t>(value, 1 << 30));
    return QC_OK;
  }
  if (k == "prefill_tcgen05") {
    c->prefill_tcgen05 = value != 0;
    return QC_OK;
  }
  if (k == "profile") {
    if (value < 0 || value > 2) return QC_ERR_INVALID_ARG;
    c->profile = static_cast<int>(value);
    return QC_OK;
  }
  return QC_ERR_INVALID_ARG;
}

int32_t qc_get_profile(qc_cache* c, qc_profile* out) {
  if (!c || !out) return QC_ERR_INVALID_ARG;
  std::memset(out, 0, sizeof(*out));
  QC_CUDA(cudaSetDevice(c->ctx->device));
  QC_CUDA(cudaStreamSynchronize(c->ctx->stream));
  for (int s = 0; s < c->ev_steps; ++s) {
    float a = 0.f, t = 0.f;
    QC_CUDA(cudaEventElapsedTime(&a, c->ev[4 * s + 1], c->ev[4 * s + 2]));
    QC_CUDA(cudaEventElapsedTime(&t, c->ev[4 * s + 0], c->ev[4 * s + 3]));
    out->attend_ms += a;
    out->step_ms += t;
  }
  for (int i = 0; i < c->ev_prefill_calls; ++i) {
    float a = 0.f;
    QC_CUDA(cudaEventElapsedTime(&a, c->ev_prefill[2 * i], c->ev_prefill[2 * i + 1]));
    out->prefill_attend_ms += a;
  }
  out->prefill_calls = c->ev_prefill_calls;
  out->prefill_flops = c->prof_prefill_flops;
  c->ev_prefill_calls = 0;
  c->prof_prefill_flops = 0.0;
  for (int i = 0; i < c->ev_launches; ++i) {
    float a = 0.f;
    QC_CUDA(cudaEventElapsedTime(&a, c->ev_launch[2 * i], c->ev_launch[2 * i + 1]));
    out->attend_kernel_ms += a;
  }
  out->attend_kernel_launches = c->ev_launches;
  c->ev_launches = 0;
  out->steps = c->ev_steps;
  out->kv_bytes_read = c->prof_bytes;
  out->items = c->prof_items;
  c->ev_steps = 0;
  c->prof_bytes = 0;
  c->prof_items = 0;
  return QC_OK;
}

}  // extern "C"
