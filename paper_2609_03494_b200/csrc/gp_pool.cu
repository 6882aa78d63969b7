// Host side of the C ABI, the blob layout, and the small bookkeeping kernels:
// step plan, admission, prompt ingest, release, debug gathers.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/growpage.h"
#include "gp_dev.cuh"

#define GP_PLAN_THREADS 1024       // threads of the plan kernel for batches of up to GP_MAX_REQ requests (a thread each) ...
#define GP_PLAN_SMALL 256          // ... and for batches of up to this many: its time is block barriers, which 8 warps pass faster than 32
#define PLAN_STATES 512            // requests of a pool whose counters the plan kernel reads ahead (8 KB: it starts beside the boundary kernel)
enum { LAUNCH_RUNS = 1, LAUNCH_CAPTURED = 2 };     // a launch now, or one into the graph that its stream is captured into
#define GP_NEVER (-(1 << 30))      // bstep of a request that has not reached a boundary

struct gp_pool {
  gp_config cfg;
  int device;
  GpDev dev;
  // asynchronous boundary mode: steps alternate between two sets of the scratch that a step's boundary chain
  // still reads while the next step runs (dev, dev_alt); the chain of a step is launched behind the attention
  // kernel of the next step (or by whatever call needs the pool's pages settled first)
  GpDev dev_alt;
  int chain_pending;                                // the last step's boundary chain has not been launched yet
  int attn_grid_async, chain_grid;
  int attn_grid_ov, chain_grid_ov;                  // synchronous mode with the boundary work beside the attention kernel
  long long serial;                                 // decode steps issued so far
  void* blob;
  size_t bytes;
  std::vector<uint8_t> live;      // host mirror of the slot free list
  int num_sms, attn_grid, sel_grid, compact_grid;
  int chain_grid_max;                               // thread blocks of the one-kernel boundary path that are resident at once
  int chain_grid_long;                              // ... in clusters that share out units of many candidates (0: this pool never has such)
  bool chain_clusters;                              // the path is launched that way where a request may be that long
  // A live request holds at most as many tokens as it was admitted with and steps have been issued since, unless a captured step is replayed.
  std::vector<long long> began;                     // of each: tokens admitted with, less the steps issued before
  long long began_max;                              // ... the most of the live ones
  bool captured;                                    // a step was captured
  int step_open, step_n_req, step_layers_done;      // per-layer entry points: a step begun and not yet ended
  int plain_plan;                                   // a request was released or a step abandoned since the last plan: the next launch
                                                    // of one that runs (LAUNCH_RUNS) or is captured (LAUNCH_CAPTURED) waits for it
  std::vector<uint8_t> step_layer_seen;             // layers gp_attn_layer has run in the open step
  cudaStream_t layer_stream;                        // stream of the last of them
  // error bits set by the kernels (GP_E_*): one int of page-locked host memory that the device addresses directly,
  // so that the host reads it without a copy once the work that could set it has completed
  int* h_err;
  // staging for the host-pointer entry point (inside the blob)
  int* st_ids; void* st_q; void* st_k; void* st_v; float* st_out; int* st_act;
  // The host entry points fetch a step's inputs on a stream of their own into one of two staging sets, so that the
  // fetch of step t + 1 runs beside the kernels of step t when the caller issues steps ahead.
  int* st2_ids; void* st2_q; void* st2_k; void* st2_v;
  cudaStream_t fetch_stream;                        // inputs in, beside the steps on the caller's stream
  cudaEvent_t ev_fetch[2], ev_used[2], ev_out[2];   // set fetched; its step has run; its results are in the caller's buffers
  long long host_steps;                             // steps issued through the host entry points
  long long host_waited;                            // gp_decode_step_host_async calls whose results have been waited for
  long long host_async_issued;                      // ... and issued
  int host_async_set[2];                            // the staging sets of the (at most two) calls not yet waited for
  // small device words
  int* d_status;
  uint8_t* dbg;                   // gather target of the debug getters
  // measurement
  int profiling;
  cudaStream_t last_stream;       // stream of the last decode step
  int early_plan;                 // gp_set_early_plan: the plan kernel reads the caller's inputs before its wait
  int first_plain;                // the step's first kernel follows a kernel of another kind: plain launch
  int32_t* actions_copy;          // host entry points: the caller's (mapped) array the boundary kernel copies the actions to
  cudaEvent_t ev[GP_N_KERNELS + 1];
  float ms[GP_N_KERNELS];
  int64_t launches[GP_N_KERNELS];
  int64_t launch_count;
};


namespace {

struct Layout {
  size_t kv, tok, rank, refcount, free_stack, words, page_table, shadow, reqi, pos, summ, Kx, Hx, delta, rc,
      merge_cnt, bnd_info, bnd_acc, free_peek, cmp_info, cmp_off, zbuf, zstat, sum_par, inv_freq, tickets, rope_f,
      unit_ready, shard_sums, bnd_info2, bnd_acc2, zbuf2, zstat2, rc2, rope_cs2, rope_f2,
      evict, evict2, cflags, rope_cs, partials, scores, counters, dbg,
      st_ids, st_q, st_k, st_v, st_out, st_act, st2_ids, st2_q, st2_k, st2_v, total;
  int max_rc;
  long long max_batch_tokens, max_boundary_tokens;
};

inline size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

// Pages per attention work item: 64 (two page ids per producer lane), and half of that for requests at their
// capacity boundary, whose pages also pay for the fp64 logits (the plan kernel has the two exceptions).  When an attention launch has less than one such
// item of work per CTA (small batches, short sequences; a layer-by-layer launch, which covers one layer's heads
// only), smaller items (32 and 8 pages) keep more CTAs busy (measured when a layer was three launches: the 36-layer shape
// with 16 requests, layer by layer, 1030 us per step that way, 1252 with the large items; a layer is one launch now, 900 us).
constexpr int GP_CHUNK = 64, GP_BCHUNK = 32;
constexpr int GP_FINE_CHUNK = 32, GP_FINE_BCHUNK = 8;
constexpr int GP_WIDE_BCHUNK = 16;       // few boundary tiles of groups of eight (see the plan kernel)
int chunk_pages_setting() { return GP_CHUNK; }
int bchunk_pages_setting() { return GP_BCHUNK; }

bool valid_config(const gp_config* c) {
  if (!c) return false;
  if (c->n_layers < 1 || c->n_kv_heads < 1 || c->n_q_heads < 1) return false;
  if (c->n_q_heads % c->n_kv_heads) return false;
  const int G = c->n_q_heads / c->n_kv_heads;
  if (G > 8 || (G & (G - 1))) return false;
  if (c->head_dim != 64 && c->head_dim != 128) return false;
  // page_size: 16, 32, ..., 256 tokens; the protected window is one 16-token tile (so it equals the page at 16)
  if (c->page_size < GP_PAGE || c->page_size > GP_MAX_BLK || (c->page_size & (c->page_size - 1))) return false;
  if (c->recent_window != GP_PAGE) return false;
  const long long sub = c->page_size / GP_PAGE;
  if (c->max_requests < 1 || c->max_requests > GP_MAX_REQ) return false;
  if (c->max_pages_per_req < 1 || c->max_pages_per_req * sub > (1 << 20)) return false;
  if (c->max_pages_per_req * sub > GP_MAX_TILES_PER_REQ) return false;
  if (c->n_pages < 1 || c->n_pages * sub > 0x7fffffffLL / GP_PAGE) return false;
  if (c->k_loc < 0 || c->k_loc > c->page_size) return false;
  if (c->max_batch_tokens < 0 || c->max_boundary_tokens < 0) return false;
  if (c->demand_metric < GP_METRIC_TOP_P || c->demand_metric > GP_METRIC_ENTROPY) return false;
  if (c->async_boundary < 0 || c->async_boundary > 1 || c->async_slots < 0 || c->async_slots > 4096) return false;
  if (c->overlap_slots < -2 || c->overlap_slots > 4096) return false;
  if (c->kv_shard_count < 1 || c->kv_shard_count > 64 || c->reserved != 0) return false;
  // spread over several pools, the mean of Eq. 8 is completed by adding up integers; the entropy variant sums doubles
  if (c->kv_shard_count > 1 && (c->demand_metric != GP_METRIC_TOP_P || c->async_boundary)) return false;
  if (!(c->beta_s >= 0.0 && c->beta_s < 1.0 && c->beta_l >= 0.0 && c->beta_l < 1.0)) return false;
  if (!(c->top_p > 0.0 && c->top_p < 1.0)) return false;
  if (!(c->rope_theta >= 0.0)) return false;
  if (c->policy < GP_POLICY_DEMAND || c->policy > GP_POLICY_SHRINK) return false;
  if (!(c->p_compress >= 0.0 && c->p_compress <= 1.0)) return false;
  if (c->min_capacity < 0 || !(c->shrink_below == c->shrink_below)) return false;
  return true;
}

Layout make_layout(const gp_config& c) {
  Layout L;
  // everything below is in physical (16-token) pages: a page of the method is `sub` of them
  const size_t sub = (size_t)c.page_size / GP_PAGE, blk = (size_t)c.page_size;
  const size_t M = c.max_requests, cap = (size_t)c.max_pages_per_req * sub, b = GP_PAGE, d = c.head_dim;
  const size_t LH = (size_t)c.n_layers * c.n_kv_heads, G = c.n_q_heads / c.n_kv_heads;
  const size_t np = (size_t)c.n_pages * sub;
  L.max_batch_tokens = c.max_batch_tokens > 0 ? c.max_batch_tokens : (long long)(np * b);
  // candidate tokens of one step's boundary requests: by default every request of a batch may be at its boundary
  // (equal prompts reach it together); a caller that knows better sizes the boundary scratch smaller
  L.max_boundary_tokens = c.max_boundary_tokens > 0 ? c.max_boundary_tokens : L.max_batch_tokens;
  if (L.max_boundary_tokens < (long long)(cap * b) && L.max_batch_tokens >= (long long)(cap * b)) L.max_boundary_tokens = (long long)(cap * b);
  const size_t Tb = (size_t)L.max_boundary_tokens;
  const int ch = chunk_pages_setting();
  int bch = bchunk_pages_setting() < ch ? bchunk_pages_setting() : ch;
  if (bch > GP_FINE_BCHUNK) bch = GP_FINE_BCHUNK;            // small launches cut finer
  L.max_rc = (int)((size_t)L.max_batch_tokens / (b * bch) + 2 * M + 1);
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes); return at; };
  L.kv = take(LH * np * 2 * b * d * 2);
  L.tok = take(LH * np * b * 4);
  L.rank = take(LH * np * b * 4);
  L.refcount = take(np * 4);
  L.free_stack = take(np * 4);
  L.words = take(256 * 4);                       // free_top, err, plan header, status
  L.page_table = take(M * cap * 4);
  L.shadow = take(M * cap * 4);
  L.reqi = take(8 * M * 4);                      // P, n, started, sum_par, live, n_pristine, bstep, last_act
  L.pos = take(M * 8);
  L.summ = take((size_t)c.n_layers * M * 2 * 2 * c.n_q_heads * d * 8);
  L.Kx = take(M * LH * 2 * 4);
  L.Hx = take(c.demand_metric == GP_METRIC_ENTROPY ? M * LH * 2 * 8 : 16);
  L.delta = take(M * 8);
  L.rc = take((size_t)L.max_rc * GP_DESC_INTS * 4);
  L.merge_cnt = take((size_t)L.max_rc * LH * 4);
  L.bnd_info = take(M * 32);
  L.bnd_acc = take(M * 16);
  L.unit_ready = take((size_t)M * LH * 4);
  L.shard_sums = take((size_t)M * 2 * 4);
  L.free_peek = take((M + 1) * 4);
  L.cmp_info = take((M + 1) * 16);
  L.cmp_off = take(M * 8);
  L.zbuf = take(LH * (Tb + b) * 2 * G * 8);
  L.zstat = take(LH * (Tb / b + 1) * 2 * G * 2 * 8);
  L.evict = take(M * LH * blk * 4);
  L.evict2 = take(c.policy == GP_POLICY_SHRINK ? M * LH * 2 * blk * 4 : 16);
  L.cflags = take(LH * ((Tb + M * b) / (1 << GP_PART_LOG_MIN) + 2 * M + 1) * 4);
  L.inv_freq = take(d / 2 * 8);
  L.tickets = take((size_t)c.n_layers * 2 * 4);
  L.rope_f = take(M * (d / 2) * 2 * 4);
  L.rope_cs = take(M * (d / 2) * 2 * 8);
  L.partials = take((size_t)L.max_rc * LH * G * (d + 2) * 4);
  L.scores = take(3 * LH * Tb * 8);                // a whole unit uses two regions, a job of one task the one of its number
  if (c.async_boundary) {                        // the second set of what a boundary chain reads beside the next step
    L.bnd_info2 = take(M * 32);
    L.bnd_acc2 = take(M * 16);
    L.zbuf2 = take(LH * (Tb + b) * 2 * G * 8);
    L.zstat2 = take(LH * (Tb / b + 1) * 2 * G * 2 * 8);
    // and of what the plan of a step writes while the attention kernel of the step before may still read its own
    L.rc2 = take((size_t)L.max_rc * GP_DESC_INTS * 4);
    L.rope_cs2 = take(M * (d / 2) * 2 * 8);
    L.rope_f2 = take(M * (d / 2) * 2 * 4);
  } else {
    L.bnd_info2 = L.bnd_acc2 = L.zbuf2 = L.zstat2 = L.rc2 = L.rope_cs2 = L.rope_f2 = 0;
  }
  L.counters = take(16 * 8);
  L.dbg = take(cap * b * (4 + 2 * d * 2));
  if (c.host_staging) {
    L.st_ids = take(M * 4);
    L.st_q = take((size_t)c.n_layers * M * c.n_q_heads * d * 2);
    L.st_k = take((size_t)c.n_layers * M * c.n_kv_heads * d * 2);
    L.st_v = take((size_t)c.n_layers * M * c.n_kv_heads * d * 2);
    L.st2_ids = take(M * 4);
    L.st2_q = take((size_t)c.n_layers * M * c.n_q_heads * d * 2);
    L.st2_k = take((size_t)c.n_layers * M * c.n_kv_heads * d * 2);
    L.st2_v = take((size_t)c.n_layers * M * c.n_kv_heads * d * 2);
    L.st_out = take((size_t)c.n_layers * M * c.n_q_heads * d * 4);
    L.st_act = take(M * 4);
  } else {
    L.st_ids = L.st_q = L.st_k = L.st_v = L.st_out = L.st_act = L.st2_ids = L.st2_q = L.st2_k = L.st2_v = 0;
  }
  L.total = o;
  return L;
}

// ---------------------------------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------------------------------
__global__ void gp_init_kernel(GpDev p) {
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // page 0 is handed out first
  for (long long i = i0; i < p.n_pages; i += stride) p.free_stack[i] = (int)(p.n_pages - 1 - i);
  for (long long i = i0; i < (long long)p.M * p.cap; i += stride) p.shadow[i] = -1;
  for (long long i = i0; i < p.M; i += stride) p.bstep[i] = GP_NEVER;
  for (long long i = i0; i < p.d / 2; i += stride) p.inv_freq[i] = p.rope_theta != 0.0 ? pow(p.rope_theta, -2.0 * (double)i / (double)p.d) : 0.0;
  if (i0 == 0) *p.free_top = (int)p.n_pages;
}

// exclusive scan over the CTA (up to 32 warps) of two ints and a long long, with the totals: one barrier (every warp scans the
// warps' sums for itself).  The arrays are free again after the caller's next barrier.
struct PlanScan { int a[32], b[32]; long long w[32]; };
__device__ __forceinline__ void plan_scan(PlanScan& S, int a, int b, long long w, int& ea, int& eb, long long& ew, int& ta, int& tb,
                                          long long& tw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto scan = [&](int& x, int& y, long long& z) {          // inclusive, over the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int x2 = __shfl_up_sync(0xffffffffu, x, off), y2 = __shfl_up_sync(0xffffffffu, y, off);
      const long long z2 = __shfl_up_sync(0xffffffffu, z, off);
      if (lane >= off) { x += x2; y += y2; z += z2; }
    }
  };
  int ia = a, ib = b; long long iw = w;
  scan(ia, ib, iw);
  if (lane == 31) { S.a[warp] = ia; S.b[warp] = ib; S.w[warp] = iw; }
  __syncthreads();
  const bool has = lane < (int)(blockDim.x >> 5);
  int xa = has ? S.a[lane] : 0, xb = has ? S.b[lane] : 0; long long xw = has ? S.w[lane] : 0;
  scan(xa, xb, xw);
  ta = __shfl_sync(0xffffffffu, xa, 31); tb = __shfl_sync(0xffffffffu, xb, 31); tw = __shfl_sync(0xffffffffu, xw, 31);
  const int pa = __shfl_sync(0xffffffffu, xa, (warp + 31) & 31), pb = __shfl_sync(0xffffffffu, xb, (warp + 31) & 31);
  const long long pw = __shfl_sync(0xffffffffu, xw, (warp + 31) & 31);
  ea = ia - a + (warp ? pa : 0); eb = ib - b + (warp ? pb : 0); ew = iw - w + (warp ? pw : 0);
}

// Step plan: validates the batch, cuts every stepped request into chunks and writes one work descriptor
// per chunk for the attention kernel, lists the requests that reach their capacity boundary with this
// step's append (trailing check: n + 1 == P b) and hands each a slice of the logit scratch.  With rotary embeddings the other
// CTAs write the cosines and sines of the requests' positions.
// What bounds it: two dependent round trips (request ids; descriptors out) and six block barriers between them.  (With the counters read
// behind the ids, three scans and a scan of the cost bins of 45 dependent steps: 12.3 us between events for 64 requests, now 10.2;
// 16 steps of four requests 317 us, now 280.)
// Loops that one request in a few hundred makes longer than a trip are not unrolled: instruction fetch (26 KB of them, now 20; us a step, two requests
// 17.9 / 17.5, 16 with rotary embeddings 30.4 / 30.0, 20 in groups of one 32.9 / 32.6, 64 62.9 / 62.9).
__global__ void __launch_bounds__(GP_PLAN_THREADS)
gp_plan_kernel(const __grid_constant__ GpDev p, const int* __restrict__ req_ids, int n_req, int* __restrict__ actions, int early,
               int cp_norm, int cp_bnd, int launch_units, int launch_grid, int serial) {
  // serial: number of this decode step (asynchronous boundary mode: a request that reached its boundary at
  // step serial - 1 sits this step out; its counters and pages belong to that step's boundary chain, which may
  // still be running)
  // cp_norm, cp_bnd: pages per work item, for requests in general and for those at their capacity boundary, when
  // the attention launch has work for large items; launch_units: (layer, head) units per request in one
  // attention launch; launch_grid: its CTAs
  // early: the caller's request ids may be read before the wait for the preceding kernel (see below)
  __shared__ PlanScan s_scan[2];
  __shared__ __align__(16) int s_first[GP_MAX_REQ];      // lowest batch index naming a request; then cost classes and items
  __shared__ int s_bin[GP_COST_BINS], s_binbase[GP_COST_BINS], s_pages, s_bpages;
  // .x slots in use, .y pages, .z position, .w: 1 live, 2 has decoded, 4 summary buffer in use, 8 sits this step out
  __shared__ int4 s_state[PLAN_STATES];
  const int i = threadIdx.x;
  const bool in = i < n_req;
  // What runs before the wait for the kernel before this one.  In a whole-step launch that kernel is the
  // compaction of the step before (or something the caller put in between, which could not start before that): this
  // grid became schedulable only after that step's decisions had completed, and compaction touches neither the
  // requests' counters nor anything the plan writes except the step stamp.  So the counters of the pool's requests are read before
  // the wait.  (In the asynchronous mode the chain kernel before this one writes counters until it ends.)
  // The caller's request ids are read before it only where the caller says that they were complete before the
  // preceding kernel could signal (`early`); CTA 0 then plans the whole step first and waits only before it looks at the free list
  // (which compaction's last CTA may still change) and stamps the step.  CTA 0 does
  // wait, so the grid as a whole still ends after everything before it.  The next kernel may be scheduled
  // as soon as every CTA of this grid has started; it waits for this grid's end at its own top.
  auto load_state = [&](int r) {                         // from the L2: before the wait
    const int live = __ldcg(p.live + r), started = __ldcg(p.started + r), par = __ldcg(p.sum_par + r);
    const int held = p.async && __ldcg(p.bstep + r) == serial - 1;
    return make_int4(__ldcg(p.n + r), __ldcg(p.P + r), (int)__ldcg(p.pos + r), (live ? 1 : 0) | (started ? 2 : 0) | (par ? 4 : 0) | (held ? 8 : 0));
  };
  const bool preloaded = !p.async && p.M <= PLAN_STATES;
  if (blockIdx.x == 0) {
    if (preloaded) {
#pragma unroll 1
      for (int t = i; t < p.M; t += blockDim.x) s_state[t] = load_state(t);
    }
#pragma unroll 1
    for (int t = i; t < p.M; t += blockDim.x) s_first[t] = 0x7fffffff;
#pragma unroll 1
    for (int t = i; t < GP_COST_BINS; t += blockDim.x) s_bin[t] = 0;
    if (i == 0) s_pages = s_bpages = 0;
    __syncthreads();
  }
  if (!early) gp_pdl_wait();
  gp_pdl_launch_dependents();
  if (blockIdx.x > 0) {                       // cos / sin of the step's position (from the L2: these CTAs may run before the wait)
    const int half = p.d / 2;
    const int idx = ((int)blockIdx.x - 1) * (int)blockDim.x + i;
    if (idx < n_req * half) {
      const int r = req_ids[idx / half];
      if (r >= 0 && r < p.M) {
        double sn, cs;
        sincos((double)__ldcg(p.pos + r) * p.inv_freq[idx % half], &sn, &cs);
        *reinterpret_cast<double2*>(p.rope_cs + (size_t)idx * 2) = make_double2(cs, sn);
        *reinterpret_cast<float2*>(p.rope_f + (size_t)idx * 2) = make_float2((float)cs, (float)sn);
      }
    }
    return;
  }
  int r = -1;
  if (in) r = req_ids[i];
  // The number this step goes by: the host's count of decode steps in the asynchronous mode (the two scratch sets
  // count on their own); otherwise the pool's own counter on the device, so that a step replayed from a CUDA graph
  // still gets a number of its own.
  const int hdr_step = __ldcg(p.hdr + HDR_STEP);           // (this kernel alone writes it)
  const int step_no = p.async ? serial : hdr_step;
  const int free_top0 = early ? 0 : __ldcg(p.free_top);
  const bool inrange = in && r >= 0 && r < p.M;
  if (inrange) atomicMin(&s_first[r], i);
  int4 st = make_int4(0, 0, 0, 0);
  if (inrange) st = preloaded ? s_state[r] : load_state(r);
  // the attention kernel draws its items from these (the one of the step before, the last to draw, has ended: that step's
  // decisions waited for it, or, where it was abandoned before it had any, this launch did)
#pragma unroll 1
  for (int idx = threadIdx.x; idx < 2 * p.L; idx += blockDim.x) p.tickets[idx] = 0;
  if (i == 0) p.hdr[HDR_WORK_SPLIT] = p.hdr[HDR_WORK_SEL] = 0;           // (the boundary work before drew from these until it let this kernel be scheduled)
  __syncthreads();
  int chunks = 0, pages = 0, act = GP_ACT_NONE;
  const int n_old = st.x, Pr = st.y, pos = st.z;
  long long nc = 0;
  int isb = 0;
  int cp = cp_norm;                       // pages per work item of this request
  if (in) {
    const bool valid = inrange && (st.w & 1) && s_first[r] == i;
    if (!valid) {
      act = GP_ACT_INVALID;
    } else if (st.w & 8) {
      act = GP_ACT_HELD;                  // its boundary chain may still be running: nothing of it is looked at
    } else if (n_old >= Pr * GP_PAGE) {
      act = GP_ACT_STALLED;
    } else {
      pages = n_old / GP_PAGE + 1;
      if (n_old + 1 == Pr * GP_PAGE) { isb = 1; nc = (long long)(Pr - 1) * GP_PAGE; }
    }
  }
  {
    // Large items when an attention launch has at least one of them per CTA (pages of the batch x units per
    // request / CTAs >= an item), fine ones otherwise: small batches, short sequences, layer-by-layer launches.
    // Measured on one layer of the 8B shape: 8 to 48 requests of 30 to 50 pages are 2 to 8 us per step faster
    // with fine items, 64 requests of 44 pages and more 3 us faster with large ones.
    const int warp_pages = __reduce_add_sync(0xffffffffu, pages);
    if ((i & 31) == 0 && warp_pages) atomicAdd(&s_pages, warp_pages);
    if (isb) atomicAdd(&s_bpages, pages);
    __syncthreads();
    // Boundary requests in large items as well where that leaves two of them per CTA: each item works out its q~ anew, which its consumer warps wait for
    // (groups of eight: 24 000 cycles an item, 3000 a tile in items of 32).  us of the attention kernel, items of 32 / 64: 64 layers x 32 requests, groups of
    // eight, two at a boundary 1636 / 1573, four 1843 / 1782; 36 x 256, 16 at a boundary 3884 / 3866, 22 4046 / 3972.  With few of them the items are
    // too long for the selection behind them: one layer x 64, four at a boundary 46 / 57; 36 x 4, one, 77.4 / 77.9 us a step.
    // In small items for groups of eight, whose boundary tiles take a consumer warp 15 000 cycles each, where there are few of them: what the step then waits
    // for is the longest (64 requests of 128 to 1400 tokens on one layer 84.4 / 79.8 us a step; 20 on eight layers 153.4 / 154.8 if it were not for
    // the bound; groups of four 62.9 / 64.3).  At d = 64 as well, items of 32 / 16: 70.2 / 65.6, 32 of 500 to 9000 on two KV heads 112.7 / 103.3 (d = 128 125.2 / 114.1), 8 on
    // four layers 78.9 / 77.3 (98.3 / 97.0); 120 requests on one layer 93.3 / 94.0, the most it costs.
    if (p.G == 8 && cp_bnd > GP_WIDE_BCHUNK && (long long)s_bpages * launch_units < 8LL * launch_grid && s_pages / GP_WIDE_BCHUNK + n_req <= p.max_rc)
      cp_bnd = GP_WIDE_BCHUNK;
    // (Not where the items, cut the smaller way, might not fit the scratch: who is refused below stays who was.)
    if ((long long)s_bpages * launch_units >= 2LL * cp_norm * launch_grid && s_pages / cp_bnd + n_req <= p.max_rc) cp_bnd = cp_norm;
    if ((long long)s_pages * launch_units < (long long)cp_norm * launch_grid) { cp_norm = GP_FINE_CHUNK; cp_bnd = GP_FINE_BCHUNK; }
  }
  if (pages > 0) {
    // a page of a boundary request also pays for the fp64 summary logits: its items are smaller, by the rules above (32 in general: 16, 24, 40 and 48
    // pages against 64 for the others, whatever the step, were all slower)
    cp = isb ? cp_bnd : cp_norm;
    chunks = (pages + cp - 1) / cp;
    cp = (pages + chunks - 1) / chunks;              // equal sizes: chunks of cp pages, the last one shorter
  }
  // (boundary requests and stepped requests in one word: at most GP_MAX_REQ of each)
  int rc_off, n_rc, both, both_tot; long long tok_off, tok_tot;
  plan_scan(s_scan[0], chunks, isb << 16 | (chunks > 0), nc, rc_off, both, tok_off, n_rc, both_tot, tok_tot);
  // A batch whose summed lengths exceed max_batch_tokens (the caller's bound; with shared prompt pages the sum
  // can exceed what the pool holds) does not fit the scratch: a request whose boundary logits or whose work
  // items do not fit is not stepped (its state stays as it is, it can be stepped again in a later batch).  The
  // offsets are then taken again over what is left, so that the item list has no holes.
  if (tok_tot > p.max_boundary_tokens || n_rc > p.max_rc) {         // (the same for every thread)
    if (chunks > 0 && ((isb && tok_off + nc > p.max_boundary_tokens) || rc_off + chunks > p.max_rc)) {
      chunks = 0; isb = 0; nc = 0; act = GP_ACT_SCRATCH;
    }
    plan_scan(s_scan[1], chunks, isb << 16 | (chunks > 0), nc, rc_off, both, tok_off, n_rc, both_tot, tok_tot);
  }
  const int bnd_idx = both >> 16, n_bnd = both_tot >> 16, n_active = both_tot & 0xffff;
  // Work items are listed by descending cost (pages), those of boundary requests, which also pay for the fp64 logits, before the
  // others: the attention kernel draws from the two parts in that order, largest first.  Counting sort.
  const int key = chunks > 0 ? cp + (isb ? GP_COST_BINS / 2 : 0) : 0;
  // Items of equal cost keep the batch's order (a rank counted over the earlier batch slots, not the order in
  // which atomics land), so that the same batch gives the same numbered list every time.  An item's number says which of a
  // block's warps takes which of its tiles, and split outputs are merged in chunk order: with the numbers fixed, the attention outputs
  // repeat bit for bit whichever thread block draws an item.
  s_first[i] = chunks > 0 ? (key << 16) | chunks : 0;        // s_first has served its purpose
  if (chunks > 0) atomicAdd(&s_bin[key], chunks);
  __syncthreads();
  if (threadIdx.x < 32) {                             // descending exclusive scan over the cost bins, five to a lane
    constexpr int PER = GP_COST_BINS / 32;
    int v[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { v[j] = s_bin[GP_COST_BINS - 1 - ((int)threadIdx.x * PER + j)]; sum += v[j]; }
    int inc = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, inc, off);
      if ((int)threadIdx.x >= off) inc += a;
    }
    int at = inc - sum;
#pragma unroll
    for (int j = 0; j < PER; ++j) { s_binbase[GP_COST_BINS - 1 - ((int)threadIdx.x * PER + j)] = at; at += v[j]; }
  }
  int within = 0;
  if (chunks > 0) {
    const int4* e4 = reinterpret_cast<const int4*>(s_first);
    int j = 0;
    for (; j + 4 <= i; j += 4) {
      const int4 e = e4[j >> 2];
      within += ((e.x >> 16) == key ? (e.x & 0xffff) : 0) + ((e.y >> 16) == key ? (e.y & 0xffff) : 0) +
                ((e.z >> 16) == key ? (e.z & 0xffff) : 0) + ((e.w >> 16) == key ? (e.w & 0xffff) : 0);
    }
#pragma unroll 1
    for (; j < i; ++j) { const int e = s_first[j]; within += (e >> 16) == key ? (e & 0xffff) : 0; }
  }
  __syncthreads();
  const int sorted0 = s_binbase[key] + within;
  if (in) {
    if (isb) { p.bstep[r] = step_no; if (p.async) act = GP_ACT_PENDING; }
    actions[i] = act;
    if (isb) {
      p.bnd_info[2 * bnd_idx] = make_int4(i, r, Pr, pos);     // pos: position of this step's token
      // .z: reports the attention kernel makes per (layer, head) unit of this request (one per consumer warp and item)
      p.bnd_info[2 * bnd_idx + 1] = make_int4((int)(unsigned)(tok_off & 0xffffffffLL), (int)(tok_off >> 32), GP_ATTN_CONSUMERS * chunks, 0);
      reinterpret_cast<int4*>(p.bnd_acc)[bnd_idx] = make_int4(0, 0, 0, 0);
    }
    // descriptors of this request's chunks: four 16-byte stores each
    const int flags = isb | (st.w & 2);
#pragma unroll 1
    for (int c = 0; c < chunks; ++c) {
      const int pg0 = c * cp;
      int4* d = reinterpret_cast<int4*>(p.rcx + (size_t)(sorted0 + c) * GP_DESC_INTS);
      d[0] = make_int4(i, r, pg0, min(cp, pages - pg0));
      d[1] = make_int4(c, chunks, n_old, pos);
      d[2] = make_int4(flags, Pr, (int)(unsigned)(tok_off & 0xffffffffLL), (int)(tok_off >> 32));
      d[3] = make_int4((st.w >> 2) & 1, rc_off + c, 0, isb ? bnd_idx : 0);
    }
  }
  // the attention kernel counts, per unit of a boundary request, the work items its consumer warps have finished
  if (p.report_units) {
#pragma unroll 1
    for (int idx = threadIdx.x; idx < n_bnd * p.L * p.Hkv; idx += blockDim.x) p.unit_ready[idx] = 0;
  }
  if (threadIdx.x == 0) {
    p.hdr[HDR_N_RC] = n_rc;
    p.hdr[HDR_N_BRC] = s_binbase[GP_COST_BINS / 2] + s_bin[GP_COST_BINS / 2];
    p.hdr[HDR_N_BND] = n_bnd;
    p.hdr[HDR_N_ACTIVE] = n_active;
  }
  // ---- from here on the kernel before this one has completed --------------------------------------------
  gp_pdl_wait();
  if (!p.async) {
    // the top of the free list, one page per boundary request: what this step's grants can take.  (In the
    // asynchronous mode the free list belongs to the boundary chains, which run one after the other: the
    // decision step reads it itself.)
    const int top = early ? __ldcg(p.free_top) : free_top0;
    if (in && isb && bnd_idx < top) p.free_peek[1 + bnd_idx] = __ldcg(p.free_stack + top - 1 - bnd_idx);
    if (threadIdx.x == 0) p.free_peek[0] = top;
  }
  if (threadIdx.x == 0) p.hdr[HDR_STEP] = hdr_step + 1;
}

constexpr int ADMIT_THREADS = 256;

// `status` on the device (the ingest kernel behind this one looks at it) and, for the host, in page-locked memory
__global__ void __launch_bounds__(ADMIT_THREADS)
gp_admit_kernel(const __grid_constant__ GpDev p, int r, int share_from, int n_shared, int n_tail, int P_target, int* status,
                volatile int* host_status) {
  gp_pdl_launch_dependents();
  const int t = threadIdx.x;
  const int need = P_target - n_shared;
  const int top = *p.free_top;
  // refusals in a fixed order: what is wrong with the arguments, then the slot, then the pages
  int st = GP_OK;
  if (n_shared > 0 && (!p.live[share_from] || p.n_pristine[share_from] < n_shared)) st = GP_ERR_INVALID;
  else if (r < 0) st = GP_ERR_NO_SLOT;
  else if (need > top || P_target > p.cap) st = GP_ERR_NO_PAGES;
  __syncthreads();                                            // everybody has seen the state the answer is taken from
  if (st == GP_OK) {
    int* table = p.page_table + (size_t)r * p.cap;
    for (int j = t; j < n_shared; j += ADMIT_THREADS) {
      const int page = p.page_table[(size_t)share_from * p.cap + j];
      table[j] = page;
      atomicAdd(&p.refcount[page], 1);
    }
    for (int j = t; j < need; j += ADMIT_THREADS) {
      const int page = p.free_stack[top - 1 - j];
      table[n_shared + j] = page;
      p.refcount[page] = 1;
    }
    if (t == 0) {
      const int n0 = n_shared * GP_PAGE + n_tail;
      *p.free_top = top - need;
      p.P[r] = P_target; p.n[r] = n0; p.pos[r] = n0; p.started[r] = 0; p.live[r] = 1;
      p.bstep[r] = GP_NEVER; p.last_act[r] = GP_ACT_NONE;
      p.n_pristine[r] = (n0 / p.blk) * p.sub;                 // only full pages of the method can be shared
    }
  }
  if (t == 0) { *status = st; *host_status = st; }
}

// Copies the private part of a prompt into its pages.  A thread block takes the keys or the values of one (layer, 16-token
// tile): up to 32 KB that are contiguous in the prompt and go to the tile's H_kv contiguous pieces.  Bound by memory; what
// it needs of the source is asked for before the admission kernel's page table is (that kernel runs meanwhile), eight 16-byte
// pieces per thread in flight.  (One piece per thread and iteration, its place found by 64-bit divisions: 56 us for 600 tokens of
// 36 layers, half the copy rate.  With the tile's address and the piece's place by division for every piece: 27.5 us for 496 tokens, and eight requests
// of 100 to 1024, admitted, decoded once and released, 583 us; with shifts where a token's pieces are a power of two, 552.)
constexpr int INGEST_THREADS = 256, INGEST_PIECES = 8;
__global__ void __launch_bounds__(INGEST_THREADS)
gp_ingest_kernel(const __grid_constant__ GpDev p, int r, int n_shared, int n_tail, const __nv_bfloat16* __restrict__ k_tail,
                 const __nv_bfloat16* __restrict__ v_tail, const int* status) {
  const int CH = p.d / 8;
  const int tiles = (n_tail + GP_PAGE - 1) / GP_PAGE;
  const int isv = (int)(blockIdx.x & 1), tile = (int)((blockIdx.x >> 1) % tiles), l = (int)((blockIdx.x >> 1) / tiles);
  const int n_tok = min(GP_PAGE, n_tail - tile * GP_PAGE);      // tokens of the tile
  const int per_tok = p.Hkv * CH, total = n_tok * per_tok;      // 16-byte pieces: of a token, of the tile
  const uint4* src = reinterpret_cast<const uint4*>((isv ? v_tail : k_tail) + ((size_t)l * n_tail + (size_t)tile * GP_PAGE) * p.Hkv * p.d);
  const int ch_log = CH == 16 ? 4 : 3, tok_log = (per_tok & (per_tok - 1)) == 0 ? 31 - __clz(per_tok) : -1;
  bool ready = false;
  uint8_t* dst = nullptr;                                       // the tile of the page's first head, and its token words
  size_t at = 0;
  for (int i0 = threadIdx.x; i0 - (int)threadIdx.x < total; i0 += INGEST_PIECES * INGEST_THREADS) {
    uint4 val[INGEST_PIECES];
#pragma unroll
    for (int e = 0; e < INGEST_PIECES; ++e) {
      const int i = i0 + e * INGEST_THREADS;
      if (i < total) val[e] = __ldcs(src + i);
    }
    if (!ready) {
      gp_pdl_wait();
      if (__ldcg(status) != GP_OK) return;
      const int page = __ldcg(p.page_table + (size_t)r * p.cap + n_shared + tile);
      dst = reinterpret_cast<uint8_t*>(p.kv + gp_tile_off(p, l, page, 0));
      at = gp_tok_off(p, l, page, 0);
      ready = true;
    }
#pragma unroll
    for (int e = 0; e < INGEST_PIECES; ++e) {
      const int i = i0 + e * INGEST_THREADS;
      if (i < total) {
        const int s = tok_log >= 0 ? i >> tok_log : i / per_tok, rest = i - s * per_tok, h = rest >> ch_log, c = rest - (h << ch_log);
        *reinterpret_cast<uint4*>(dst + (size_t)((((2 * h + isv) * GP_PAGE + s) << ch_log) + (c ^ (s & 7))) * 16) = val[e];
        if (isv == 0 && c == 0) p.tok[at + h * GP_PAGE + s] = p.rank[at + h * GP_PAGE + s] = (n_shared + tile) * GP_PAGE + s;
      }
    }
  }
}

// Drops the request's references, a thread per page; the pages nobody else holds go back to the free list in table order.
// (One warp: 6.7 us for 130 pages.)
__global__ void __launch_bounds__(ADMIT_THREADS)
gp_release_kernel(const __grid_constant__ GpDev p, int r) {
  __shared__ int s_warp[ADMIT_THREADS / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int Pr = p.P[r];
  const int* table = p.page_table + (size_t)r * p.cap;
  int top = *p.free_top;
  for (int j0 = 0; j0 < Pr; j0 += ADMIT_THREADS) {
    const int j = j0 + t;
    int page = -1;
    bool freed = false;
    if (j < Pr) {
      page = table[j];
      freed = (atomicSub(&p.refcount[page], 1) == 1);
    }
    const unsigned mask = __ballot_sync(0xffffffffu, freed);
    if (lane == 0) s_warp[warp] = __popc(mask);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < ADMIT_THREADS / 32; ++w) { all += s_warp[w]; before += w < warp ? s_warp[w] : 0; }
    if (freed) p.free_stack[top + before + __popc(mask & ((1u << lane) - 1u))] = page;
    top += all;
    __syncthreads();
  }
  __syncthreads();                                            // everybody has read the pages and the top
  if (t == 0) {
    *p.free_top = top;
    p.live[r] = 0; p.P[r] = 0; p.n[r] = 0; p.started[r] = 0; p.n_pristine[r] = 0; p.bstep[r] = GP_NEVER;
  }
}

// debug: token ids and un-swizzled K, V rows of one (layer, head) stream into the gather buffer, in the order of the tokens
__global__ void gp_gather_kernel(GpDev p, int r, int l, int h, int n, int* tok_out, uint4* k_out, uint4* v_out) {
  const int CH = p.d / 8;
  const int row_bytes = p.d * 2;
  const long long total = (long long)n * 2 * CH;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(idx % CH);
    const int isv = (int)((idx / CH) % 2);
    const int slot = (int)(idx / (2 * CH));
    const int page = p.page_table[(size_t)r * p.cap + slot / GP_PAGE];
    const int s = slot % GP_PAGE;
    const uint8_t* src = reinterpret_cast<const uint8_t*>(p.kv + gp_tile_off(p, l, page, h)) +
                         isv * GP_PAGE * row_bytes + s * row_bytes + ((c ^ (s & 7)) << 4);
    const int at = p.rank[gp_tok_off(p, l, page, h) + s];
    if (at < 0 || at >= n) continue;                         // (a wait that gave up: the pool's error word says so)
    (isv ? v_out : k_out)[(size_t)at * CH + c] = *reinterpret_cast<const uint4*>(src);
    if (isv == 0 && c == 0) tok_out[at] = p.tok[gp_tok_off(p, l, page, h) + s];
  }
}

#define GP_CUDA(x)                      \
  do {                                  \
    if ((x) != cudaSuccess) return GP_ERR_CUDA; \
  } while (0)

void pool_free(gp_pool* pool) {
  if (pool->h_err) cudaFreeHost(pool->h_err);
  if (pool->fetch_stream) {
    cudaStreamDestroy(pool->fetch_stream);
    for (int i = 0; i < 2; ++i) { cudaEventDestroy(pool->ev_fetch[i]); cudaEventDestroy(pool->ev_used[i]); cudaEventDestroy(pool->ev_out[i]); }
  }
  delete pool;
}

// Asynchronous boundary mode: launches the boundary chain of the last decode step on `s` if it has not been
// launched yet (it normally rides behind the next step's attention kernel).  Everything that looks at the pool's
// pages, counters or free list from outside a decode step calls this first.
int flush_chain(gp_pool* pool, cudaStream_t s) {
  if (!pool->cfg.async_boundary || !pool->chain_pending) return GP_OK;
  const long long t = pool->serial - 1;                       // the step the chain belongs to
  const GpDev& d = (t & 1) ? pool->dev_alt : pool->dev;
  gp_launch_chain(d, 0, (int)(t & 0x3fffffff), 1, pool->chain_grid, s, false);
  pool->chain_pending = 0;
  pool->launch_count += 1;
  return cudaGetLastError() == cudaSuccess ? GP_OK : GP_ERR_CUDA;
}

// the kernels' error bits, once the work that could set them has completed
int kernel_status(const gp_pool* pool) {
  return *reinterpret_cast<volatile const int*>(pool->h_err) ? GP_ERR_CUDA : GP_OK;
}

bool misaligned(const void* ptr, uintptr_t a) { return (reinterpret_cast<uintptr_t>(ptr) & (a - 1)) != 0; }

int check_req(gp_pool* pool, int32_t req) {
  if (!pool) return GP_ERR_INVALID;
  if (req < 0 || req >= pool->cfg.max_requests || !pool->live[req]) return GP_ERR_INVALID;
  return GP_OK;
}

}  // namespace

// ===================================================================================================
// C ABI
// ===================================================================================================
extern "C" {

int gp_config_default(gp_config* cfg) {
  if (!cfg) return GP_ERR_INVALID;
  memset(cfg, 0, sizeof(*cfg));
  cfg->page_size = GP_PAGE;
  cfg->max_requests = 512;
  cfg->recent_window = GP_PAGE;
  cfg->kv_shard_count = 1;
  cfg->k_loc = GP_PAGE / 4;          // a quarter of the page; the paper's 64 at its page size of 256
  cfg->beta_s = 0.9;
  cfg->beta_l = 0.999;
  cfg->top_p = 0.99;
  cfg->tau = 0.0;
  cfg->rope_theta = 0.0;
  cfg->policy = GP_POLICY_DEMAND;
  cfg->policy_seed = 0;
  cfg->p_compress = 0.7;
  cfg->shrink_below = -0.005;
  cfg->min_capacity = 1024;
  return GP_OK;
}

size_t gp_pool_bytes(const gp_config* cfg) {
  if (!valid_config(cfg)) return 0;
  return make_layout(*cfg).total;
}

int gp_pool_create(const gp_config* cfg, void* dev_blob, size_t bytes, int device, gp_pool** out) {
  if (!out) return GP_ERR_INVALID;
  *out = nullptr;
  if (!valid_config(cfg) || !dev_blob || ((uintptr_t)dev_blob & 255)) return GP_ERR_INVALID;
  const Layout L = make_layout(*cfg);
  if (bytes < L.total) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(device));
  gp_pool* pool = new (std::nothrow) gp_pool();
  if (!pool) return GP_ERR_STATE;
  pool->cfg = *cfg;
  pool->device = device;
  pool->blob = dev_blob;
  pool->bytes = bytes;
  pool->live.assign(cfg->max_requests, 0);
  pool->began.assign(cfg->max_requests, 0);
  pool->began_max = 0;
  pool->captured = false;
  pool->profiling = 0;
  pool->early_plan = 0;
  pool->first_plain = 0;
  pool->step_open = 0; pool->step_n_req = 0; pool->step_layers_done = 0; pool->plain_plan = 0;
  pool->step_layer_seen.assign(cfg->n_layers, 0);
  pool->h_err = nullptr;
  pool->launch_count = 0;
  pool->serial = 0;
  memset(pool->ms, 0, sizeof(pool->ms));
  memset(pool->launches, 0, sizeof(pool->launches));
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) { pool_free(pool); return GP_ERR_CUDA; }
  pool->num_sms = prop.multiProcessorCount;
  pool->attn_grid = pool->num_sms * gp_attention_ctas_per_sm(cfg->head_dim);

  uint8_t* base = static_cast<uint8_t*>(dev_blob);
  GpDev& d = pool->dev;
  d.L = cfg->n_layers; d.Hq = cfg->n_q_heads; d.Hkv = cfg->n_kv_heads; d.G = cfg->n_q_heads / cfg->n_kv_heads;
  d.sub = cfg->page_size / GP_PAGE; d.blk = cfg->page_size;
  d.d = cfg->head_dim; d.M = cfg->max_requests; d.cap = cfg->max_pages_per_req * d.sub; d.k_loc = cfg->k_loc;
  d.chunk_pages = chunk_pages_setting(); d.max_rc = L.max_rc;
  d.bchunk_pages = bchunk_pages_setting();
  d.n_pages = cfg->n_pages * d.sub; d.max_batch_tokens = L.max_batch_tokens;
  d.max_boundary_tokens = L.max_boundary_tokens;
  d.async = cfg->async_boundary;
  d.spin_limit = GP_SPIN_LIMIT;
  d.withhold = 0;
  d.z_stride = (L.max_boundary_tokens + GP_PAGE - 1) / GP_PAGE * GP_PAGE;
  d.beta_s = cfg->beta_s; d.beta_l = cfg->beta_l; d.top_p = cfg->top_p; d.tau = cfg->tau; d.rope_theta = cfg->rope_theta;
  d.policy = cfg->policy; d.policy_seed = (unsigned long long)(unsigned)cfg->policy_seed; d.p_compress = cfg->p_compress;
  d.shrink_below = cfg->shrink_below;
  {
    const long long mp = (cfg->min_capacity + GP_PAGE - 1) / GP_PAGE;      // (P - 1) b >= min_capacity, and P >= 3
    d.min_pages_after_shrink = (int)(mp > (1 << 21) ? (1 << 21) : (mp < 2 * d.sub ? 2 * d.sub : mp));
  }
  d.p_fix = (unsigned long long)llrint(cfg->top_p * 4611686018427387904.0);
  d.kv = reinterpret_cast<__nv_bfloat16*>(base + L.kv);
  d.tok = reinterpret_cast<int*>(base + L.tok);
  d.rank = reinterpret_cast<int*>(base + L.rank);
  d.refcount = reinterpret_cast<int*>(base + L.refcount);
  d.free_stack = reinterpret_cast<int*>(base + L.free_stack);
  int* words = reinterpret_cast<int*>(base + L.words);
  d.free_top = words + 0;
  {
    void* herr = nullptr; void* derr = nullptr;
    if (cudaHostAlloc(&herr, 64, cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer(&derr, herr, 0) != cudaSuccess) {
      if (herr) cudaFreeHost(herr);
      pool_free(pool);
      return GP_ERR_CUDA;
    }
    memset(herr, 0, 64);
    pool->h_err = static_cast<int*>(herr);
    d.err = static_cast<int*>(derr);
  }
  pool->d_status = words + 2;
  d.hdr = words + 64;
  d.page_table = reinterpret_cast<int*>(base + L.page_table);
  d.shadow = reinterpret_cast<int*>(base + L.shadow);
  int* reqi = reinterpret_cast<int*>(base + L.reqi);
  const int M = cfg->max_requests;
  d.P = reqi; d.n = reqi + M; d.started = reqi + 2 * M; d.sum_par = reqi + 3 * M;
  d.live = reqi + 4 * M; d.n_pristine = reqi + 5 * M; d.bstep = reqi + 6 * M; d.last_act = reqi + 7 * M;
  d.pos = reinterpret_cast<long long*>(base + L.pos);
  d.summ = reinterpret_cast<double*>(base + L.summ);
  d.Kx = reinterpret_cast<int*>(base + L.Kx);
  d.Hx = reinterpret_cast<double*>(base + L.Hx);
  d.metric = cfg->demand_metric;
  d.delta = reinterpret_cast<double*>(base + L.delta);
  d.rcx = reinterpret_cast<int*>(base + L.rc);
  d.merge_cnt = reinterpret_cast<int*>(base + L.merge_cnt);
  d.bnd_info = reinterpret_cast<int4*>(base + L.bnd_info);
  d.bnd_acc = reinterpret_cast<int*>(base + L.bnd_acc);
  d.unit_ready = reinterpret_cast<int*>(base + L.unit_ready);
  d.shard_sums = reinterpret_cast<int*>(base + L.shard_sums);
  d.units_total = cfg->n_layers * cfg->n_kv_heads * cfg->kv_shard_count;
  d.free_peek = reinterpret_cast<int*>(base + L.free_peek);
  d.cmp_info = reinterpret_cast<int4*>(base + L.cmp_info);
  d.cmp_off = reinterpret_cast<long long*>(base + L.cmp_off);
  d.zbuf = reinterpret_cast<double*>(base + L.zbuf);
  d.zstat = reinterpret_cast<double*>(base + L.zstat);
  d.evict = reinterpret_cast<int*>(base + L.evict);
  d.evict2 = reinterpret_cast<int*>(base + L.evict2);
  d.cflags = reinterpret_cast<int*>(base + L.cflags);
  d.inv_freq = reinterpret_cast<double*>(base + L.inv_freq);
  d.tickets = reinterpret_cast<int*>(base + L.tickets);
  d.rope_f = reinterpret_cast<float*>(base + L.rope_f);
  d.rope_cs = reinterpret_cast<double*>(base + L.rope_cs);
  d.partials = reinterpret_cast<float*>(base + L.partials);
  d.scores = reinterpret_cast<double*>(base + L.scores);
  d.counters = reinterpret_cast<long long*>(base + L.counters);
  gp_attention_setup(d);
  gp_boundary_setup(d, pool->num_sms, &pool->sel_grid, &pool->compact_grid, &pool->chain_grid_max, &pool->chain_grid_long);
  pool->dev_alt = d;
  pool->chain_pending = 0;
  pool->last_stream = nullptr;
  if (cfg->async_boundary) {
    GpDev& a = pool->dev_alt;
    a.hdr = words + 128;
    a.bnd_info = reinterpret_cast<int4*>(base + L.bnd_info2);
    a.bnd_acc = reinterpret_cast<int*>(base + L.bnd_acc2);
    a.zbuf = reinterpret_cast<double*>(base + L.zbuf2);
    a.zstat = reinterpret_cast<double*>(base + L.zstat2);
    a.rcx = reinterpret_cast<int*>(base + L.rc2);
    a.rope_f = reinterpret_cast<float*>(base + L.rope_f2);
    a.rope_cs = reinterpret_cast<double*>(base + L.rope_cs2);
    // the chain kernel runs beside the attention kernel on the room it leaves: `slots` of its thread blocks
    int slots = cfg->async_slots > 0 ? cfg->async_slots : 64;
    if (slots > pool->attn_grid / 2) slots = pool->attn_grid / 2;
    pool->attn_grid_async = pool->attn_grid - slots;
    pool->chain_grid = slots;
  }
  pool->attn_grid_ov = pool->attn_grid;
  pool->chain_grid_ov = 0;
  pool->chain_clusters = false;
  // How the boundary work of a step is launched where the caller leaves it open.  One kernel behind the attention kernel saves a kernel
  // boundary and starts its jobs while the attention kernel drains (us per step, four kernels / one, layers x requests, 8 KV heads:
  // 1 x 64 73.5 / 65.7; 8 x 16 91 / 87; 36 x 4 84 / 83; 36 x 16 314 / 310); from about ten thousand units on the two kernels'
  // larger grids are worth as much (64 x 32: 1790 / 1810; 36 x 64: 1177 / 1180; 36 x 256: 4388 / 4420).
  const long long units = (long long)cfg->n_layers * cfg->n_kv_heads * cfg->max_requests;
  int slots = cfg->overlap_slots;
  if (slots == 0) slots = units <= 8192 ? -2 : -1;
  if (!cfg->async_boundary && slots == -2) {
    pool->chain_clusters = pool->chain_grid_long > 0;
    pool->chain_grid_ov = pool->chain_grid_max;    // the whole grid, behind the attention kernel's
  } else if (!cfg->async_boundary && slots > 0) {
    if (slots > pool->attn_grid / 2) slots = pool->attn_grid / 2;
    pool->attn_grid_ov = pool->attn_grid - slots;
    pool->chain_grid_ov = slots;
  }
  pool->dev.report_units = pool->dev_alt.report_units = pool->chain_grid_ov > 0;
  const int cmp_ctas = cfg->async_boundary ? pool->chain_grid : pool->chain_grid_ov > 0 ? pool->chain_grid_ov : pool->compact_grid;
  pool->dev.copy_share = pool->dev_alt.copy_share = (float)(cfg->n_layers * cfg->n_kv_heads) / (float)cmp_ctas;
  pool->dbg = base + L.dbg;
  if (cfg->host_staging) {
    pool->st_ids = reinterpret_cast<int*>(base + L.st_ids);
    pool->st_q = base + L.st_q; pool->st_k = base + L.st_k; pool->st_v = base + L.st_v;
    pool->st2_ids = reinterpret_cast<int*>(base + L.st2_ids);
    pool->st2_q = base + L.st2_q; pool->st2_k = base + L.st2_k; pool->st2_v = base + L.st2_v;
    pool->st_out = reinterpret_cast<float*>(base + L.st_out);
    pool->st_act = reinterpret_cast<int*>(base + L.st_act);
  } else {
    pool->st_ids = nullptr; pool->st_q = pool->st_k = pool->st_v = nullptr; pool->st_out = nullptr; pool->st_act = nullptr;
  }
  // Stale pages are read (masked) by the attention kernel, so they must hold finite numbers.
  if (cudaMemset(dev_blob, 0, L.total) != cudaSuccess) { pool_free(pool); return GP_ERR_CUDA; }
  gp_init_kernel<<<1024, 256>>>(d);
  pool->launch_count++;
  for (int i = 0; i <= GP_N_KERNELS; ++i) {
    if (cudaEventCreate(&pool->ev[i]) != cudaSuccess) { pool_free(pool); return GP_ERR_CUDA; }
  }
  if (cudaDeviceSynchronize() != cudaSuccess) { pool_free(pool); return GP_ERR_CUDA; }
  *out = pool;
  return GP_OK;
}

int gp_pool_destroy(gp_pool* pool) {
  if (!pool) return GP_ERR_INVALID;
  cudaSetDevice(pool->device);
  cudaDeviceSynchronize();
  for (int i = 0; i <= GP_N_KERNELS; ++i) cudaEventDestroy(pool->ev[i]);
  pool_free(pool);
  return GP_OK;
}

static int launch_kind(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) (void)cudaGetLastError();      // (the legacy stream beside a capture: runs)
  return st == cudaStreamCaptureStatusNone ? LAUNCH_RUNS : LAUNCH_CAPTURED;
}

int gp_request_add(gp_pool* pool, int32_t share_from, int32_t n_shared_pages, const void* k_tail, const void* v_tail,
                   int32_t n_tail, int32_t initial_pages, void* stream, int32_t* out_req) {
  if (!pool || !out_req || n_tail < 0 || n_shared_pages < 0 || initial_pages < 0) return GP_ERR_INVALID;
  if (n_tail > 0 && (!k_tail || !v_tail || misaligned(k_tail, 16) || misaligned(v_tail, 16))) return GP_ERR_INVALID;
  *out_req = -1;
  if (pool->step_open) return GP_ERR_STATE;      // the open step's plan holds a snapshot of the free list
  if (n_shared_pages > 0 && check_req(pool, share_from) != GP_OK) return GP_ERR_INVALID;
  const gp_config& c = pool->cfg;
  int slot = -1;
  for (int i = 0; i < c.max_requests; ++i)
    if (!pool->live[i]) { slot = i; break; }
  if (slot < 0 && n_shared_pages == 0) return GP_ERR_NO_SLOT;
  const int sub = c.page_size / GP_PAGE;
  const long long n_prompt = (long long)n_shared_pages * c.page_size + n_tail;
  long long P = n_prompt / c.page_size + 1;
  if (initial_pages > P) P = initial_pages;
  // with shared pages the donor's count of shareable pages lives on the device: the kernel below gives the
  // refusals in the documented order (invalid arguments, no slot, no pages)
  if (P > c.max_pages_per_req && n_shared_pages == 0) return GP_ERR_NO_PAGES;
  if (P > c.max_pages_per_req) P = (long long)c.max_pages_per_req + 1;      // still refused, and fits an int
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (flush_chain(pool, s) != GP_OK) return GP_ERR_CUDA;       // the free list belongs to the last step's boundary chain first
  // The kernels count in physical pages.  The ingest is launched behind the admission and looks at its status itself, so
  // that the host waits once: for the status, and so that the caller may free the prompt buffers on return.
  volatile int* h_status = pool->h_err + 1;
  *h_status = GP_ERR_CUDA;
  gp_admit_kernel<<<1, ADMIT_THREADS, 0, s>>>(pool->dev, slot, share_from, n_shared_pages * sub, n_tail, (int)(P * sub), pool->d_status,
                                              pool->dev.err + 1);
  pool->launch_count++;
  GP_CUDA(cudaGetLastError());
  if (n_tail > 0 && slot >= 0 && P <= c.max_pages_per_req) {       // (otherwise the admission refuses: nothing to copy, and no bound on n_tail)
    const long long blocks = 2LL * ((n_tail + GP_PAGE - 1) / GP_PAGE) * c.n_layers;
    GP_CUDA(gp_launch(gp_ingest_kernel, (int)blocks, INGEST_THREADS, 0, s, true, pool->dev, slot, n_shared_pages * sub, (int)n_tail,
                      static_cast<const __nv_bfloat16*>(k_tail), static_cast<const __nv_bfloat16*>(v_tail),
                      static_cast<const int*>(pool->d_status)));
    pool->launch_count++;
  }
  GP_CUDA(cudaStreamSynchronize(s));
  const int st = *h_status;
  if (st != GP_OK) return st;
  pool->live[slot] = 1;
  pool->began[slot] = n_prompt - pool->serial;
  if (pool->began[slot] > pool->began_max) pool->began_max = pool->began[slot];
  *out_req = slot;
  return GP_OK;
}

static const GpNorm kNoNorm = {nullptr, nullptr, 0.0};

// CTA 0 plans; the others fill the table of cosines and sines (a thread per entry).  The plan reads the requests' counters before
// its wait, so what writes them has to be done when it starts.  Behind the kernels of a step it is; behind a release or an abandoned
// step the launch is a plain one, without early planning: only the wait would show the plan what a release has written, and an abandoned
// step's kernels let their dependents go at their top and no decision waited for them, so that a plan beside them would take the items
// they still draw and the counters they draw from.  (An admission is waited for on the host.)
static void launch_plan(gp_pool* pool, const int32_t* ids, int32_t n_req, int32_t* actions, bool early, cudaStream_t s, bool pdl,
                        bool by_layer = false, const GpDev* dev = nullptr, int attn_grid = 0) {
  const GpDev& d = dev ? *dev : pool->dev;
  const int threads = n_req <= GP_PLAN_SMALL ? GP_PLAN_SMALL : GP_PLAN_THREADS;
  const int table = d.rope_theta != 0.0 ? (n_req * (d.d / 2) + threads - 1) / threads : 0;
  if (pool->plain_plan) {
    const int mine = launch_kind(s);
    if (pool->plain_plan & mine) { early = false; pdl = false; pool->plain_plan &= ~mine; }
  }
  if (pool->chain_clusters && !pool->captured) pool->captured = launch_kind(s) == LAUNCH_CAPTURED;
  gp_launch(gp_plan_kernel, 1 + table, threads, 0, s, pdl, d, ids, n_req, actions, early ? 1 : 0, d.chunk_pages, d.bchunk_pages,
            by_layer ? d.Hkv : d.L * d.Hkv, attn_grid ? attn_grid : pool->attn_grid, (int)(pool->serial & 0x3fffffff));
}

int gp_decode_step(gp_pool* pool, const int32_t* dev_req_ids, int32_t n_req, const void* q, const void* k,
                   const void* v, void* out, int32_t* dev_actions, void* stream) {
  if (!pool || n_req < 0 || n_req > pool->cfg.max_requests) return GP_ERR_INVALID;
  if (pool->step_open) return GP_ERR_STATE;
  if (n_req == 0) return GP_OK;
  if (!dev_req_ids || !q || !k || !v || !out || !dev_actions) return GP_ERR_INVALID;
  // the kernels move query, key and value rows with 16-byte copies and write `out` in 8-byte pieces
  if (misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(out, 16) ||
      misaligned(dev_req_ids, 4) || misaligned(dev_actions, 4)) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool prof = pool->profiling != 0;
  const bool pdl = !prof;                      // events between the kernels need them serialised the plain way
  const int serial = (int)(pool->serial & 0x3fffffff);
  if (!pool->cfg.async_boundary) {
    const GpDev& d = pool->dev;
    const int LH = d.L * d.Hkv;
    if (prof) cudaEventRecord(pool->ev[0], s);
    // first_plain: the kernel before the plan on the stream is not one of this library's (the host entry point's
    // fetch of the inputs): no programmatic dependence on it
    if (pool->chain_grid_ov > 0) {
      // Three kernels.  The boundary work of the step (selection jobs, decisions, compaction) is one kernel behind the
      // attention kernel.  Its thread blocks take their places as that
      // kernel's leave (or, with overlap_slots > 0, run beside it on slots its grid leaves free), and a selection job
      // starts as soon as the attention kernel has reported its unit's summary logits complete.
      launch_plan(pool, dev_req_ids, n_req, dev_actions, pool->early_plan != 0, s, pdl && !pool->first_plain, false, nullptr,
                  pool->attn_grid_ov);
      if (prof) cudaEventRecord(pool->ev[1], s);
      gp_launch_attention(d, n_req, q, k, v, static_cast<float*>(out), pool->attn_grid_ov, s, pdl, 0, LH, 0, false, false, kNoNorm);
      if (prof) cudaEventRecord(pool->ev[2], s);
      // In clusters where a request may be long enough for one to share out its units: blocks that find their places eight at a time and draw their
      // jobs are slower where none is.  us a step with requests of up to 1400 tokens that might grow to 16 000, in clusters / not, layers x
      // requests: 1 x 64 65.8 / 62.7, at d = 64 54.4 / 51.3; four short ones 17.4 / 16.7; 36 x 16 312.5 / 295.2.  Replays of a captured step are not
      // counted, so from the first capture on every launch is one in clusters.  The results are those of the other form.
      const bool clusters = pool->chain_clusters && (pool->captured || pool->began_max + pool->serial > GP_SHARED_FROM);
      gp_launch_chain(d, n_req, serial, 1, clusters ? pool->chain_grid_long : pool->chain_grid_ov, s, pdl, dev_req_ids, dev_actions, pool->actions_copy,
                      clusters);
      if (prof) { cudaEventRecord(pool->ev[3], s); cudaEventRecord(pool->ev[4], s); }    // the last interval stays empty
      pool->launch_count += 3;
    } else {
      // Four kernels, one after the other (overlap_slots = -1): the selection and compaction kernels of the
      // layer-by-layer step
      launch_plan(pool, dev_req_ids, n_req, dev_actions, pool->early_plan != 0, s, pdl && !pool->first_plain);
      if (prof) cudaEventRecord(pool->ev[1], s);
      gp_launch_attention(d, n_req, q, k, v, static_cast<float*>(out), pool->attn_grid, s, pdl, 0, LH, 0, false, false, kNoNorm);
      if (prof) cudaEventRecord(pool->ev[2], s);
      gp_launch_boundary(d, dev_req_ids, n_req, dev_actions, false, pool->sel_grid, pool->compact_grid, s,
                         prof ? pool->ev[3] : nullptr, pdl, serial);
      if (prof) cudaEventRecord(pool->ev[4], s);
      pool->launch_count += GP_N_KERNELS;
    }
  } else {
    // Asynchronous boundary work, all on the caller's stream: plan and attention of this step, then one kernel
    // with the boundary chain of the step before (working sets, decisions, compaction), which runs beside the
    // attention kernel and ends after it.  Step t uses scratch set t mod 2.
    const int par = (int)(pool->serial & 1);
    const GpDev& d = par ? pool->dev_alt : pool->dev;
    const GpDev& dprev = par ? pool->dev : pool->dev_alt;
    const int LH = d.L * d.Hkv;
    if (prof) cudaEventRecord(pool->ev[0], s);
    // no early planning here: the plan reads the pages and slots of the requests that return from their step out,
    // which the chain kernel of the step before (the kernel before this one on the stream) has just written
    launch_plan(pool, dev_req_ids, n_req, dev_actions, false, s, pdl && !pool->first_plain, false, &d, pool->attn_grid_async);
    if (prof) cudaEventRecord(pool->ev[1], s);
    gp_launch_attention(d, n_req, q, k, v, static_cast<float*>(out), pool->attn_grid_async, s, pdl, 0, LH, 0, false, false, kNoNorm);
    if (prof) cudaEventRecord(pool->ev[2], s);
    // the decisions of the step before set pages and slots of requests that sit this step out: nothing else of
    // this step looks at those words
    gp_launch_chain(dprev, n_req, (int)((pool->serial - 1) & 0x3fffffff), pool->chain_pending, pool->chain_grid, s, pdl);
    if (prof) { cudaEventRecord(pool->ev[3], s); cudaEventRecord(pool->ev[4], s); }
    pool->chain_pending = 1;
    pool->last_stream = s;
    pool->launch_count += 3;
  }
  pool->serial += 1;
  GP_CUDA(cudaGetLastError());
  if (prof) {
    GP_CUDA(cudaEventSynchronize(pool->ev[GP_N_KERNELS]));
    for (int i = 0; i < GP_N_KERNELS; ++i) {
      float t = 0.f;
      GP_CUDA(cudaEventElapsedTime(&t, pool->ev[i], pool->ev[i + 1]));
      pool->ms[i] += t;
      pool->launches[i] += 1;
    }
  }
  return GP_OK;
}

int gp_async_join(gp_pool* pool, void* stream) {
  if (!pool) return GP_ERR_INVALID;
  if (!pool->cfg.async_boundary) return GP_OK;
  GP_CUDA(cudaSetDevice(pool->device));
  return flush_chain(pool, static_cast<cudaStream_t>(stream));
}

int gp_boundary_outcome(gp_pool* pool, int32_t req, int32_t* action, int64_t* step) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  int a = 0, b = 0;
  GP_CUDA(cudaMemcpy(&a, pool->dev.last_act + req, 4, cudaMemcpyDeviceToHost));
  GP_CUDA(cudaMemcpy(&b, pool->dev.bstep + req, 4, cudaMemcpyDeviceToHost));
  if (b == GP_NEVER) a = GP_ACT_NONE;
  if (action) *action = a;
  if (step) *step = b == GP_NEVER ? -1 : (int64_t)((pool->serial & ~0x3fffffffLL) | (long long)b);
  return GP_OK;
}

// ---- the same step, layer by layer: a model's forward pass has layer l + 1's query only after layer l's
// attention output ---------------------------------------------------------------------------------------
int gp_step_begin(gp_pool* pool, const int32_t* dev_req_ids, int32_t n_req, int32_t* dev_actions, void* stream) {
  if (!pool || n_req < 0 || n_req > pool->cfg.max_requests) return GP_ERR_INVALID;
  if (pool->step_open || pool->cfg.async_boundary) return GP_ERR_STATE;
  if (n_req == 0) return GP_OK;
  if (!dev_req_ids || !dev_actions || misaligned(dev_req_ids, 4) || misaligned(dev_actions, 4)) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  launch_plan(pool, dev_req_ids, n_req, dev_actions, false, static_cast<cudaStream_t>(stream), true, true);
  pool->launch_count += 1;
  pool->step_open = 1;
  pool->step_n_req = n_req;
  pool->step_layers_done = 0;
  pool->step_layer_seen.assign(pool->cfg.n_layers, 0);
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

// A layer behind another layer's launch on the same stream may start before that one has ended: the plan it reads has (that
// launch waited for it), and layers share nothing else (see gp_attn_kernel).
static void launch_layer(gp_pool* pool, int n_req, const void* q, const void* k, const void* v, float* out, int layer, cudaStream_t s,
                         const GpNorm& nm) {
  const GpDev& d = pool->dev;
  const bool planned = pool->step_layers_done > 0 && s == pool->layer_stream;
  pool->layer_stream = s;
  gp_launch_attention(d, n_req, q, k, v, out, pool->attn_grid, s, true, layer * d.Hkv, d.Hkv, -1, true, planned, nm);
}

int gp_attn_layer(gp_pool* pool, int32_t layer, const int32_t* dev_req_ids, int32_t n_req, const void* q, const void* k,
                  const void* v, void* out, void* stream) {
  if (!pool || pool->step_open != 1 || n_req != pool->step_n_req) return pool && pool->step_open != 1 ? GP_ERR_STATE : GP_ERR_INVALID;
  if (layer < 0 || layer >= pool->cfg.n_layers || !dev_req_ids || !q || !k || !v || !out) return GP_ERR_INVALID;
  if (misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(out, 16) || misaligned(dev_req_ids, 4))
    return GP_ERR_INVALID;
  if (pool->step_layer_seen[layer]) return GP_ERR_STATE;          // every layer once
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const GpDev& d = pool->dev;
  // The kernels index their per-step tensors as [layer][request][head][d]: a layer's own tensors are handed over
  // as the base such an array would have (the kernels only touch this layer's part of it).
  const size_t qs = (size_t)layer * n_req * d.Hq * d.d, ks = (size_t)layer * n_req * d.Hkv * d.d;
  const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(reinterpret_cast<uintptr_t>(q) - qs * 2);
  const __nv_bfloat16* kb = reinterpret_cast<const __nv_bfloat16*>(reinterpret_cast<uintptr_t>(k) - ks * 2);
  const __nv_bfloat16* vb = reinterpret_cast<const __nv_bfloat16*>(reinterpret_cast<uintptr_t>(v) - ks * 2);
  float* ob = reinterpret_cast<float*>(reinterpret_cast<uintptr_t>(out) - qs * 4);
  launch_layer(pool, n_req, qb, kb, vb, ob, layer, s, kNoNorm);
  pool->launch_count += 1;
  pool->step_layers_done += 1;
  pool->step_layer_seen[layer] = 1;
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

int gp_attn_layer_qknorm(gp_pool* pool, int32_t layer, const int32_t* dev_req_ids, int32_t n_req, const void* q_raw,
                         const void* k_raw, const void* v, const float* q_weight, const float* k_weight, double eps, void* out,
                         void* stream) {
  if (!pool || pool->step_open != 1 || n_req != pool->step_n_req) return pool && pool->step_open != 1 ? GP_ERR_STATE : GP_ERR_INVALID;
  if (layer < 0 || layer >= pool->cfg.n_layers || !dev_req_ids || !q_raw || !k_raw || !v || !out || !q_weight || !k_weight)
    return GP_ERR_INVALID;
  if (misaligned(q_raw, 16) || misaligned(k_raw, 16) || misaligned(v, 16) || misaligned(out, 16) || misaligned(dev_req_ids, 4) ||
      misaligned(q_weight, 4) || misaligned(k_weight, 4) || !(eps >= 0.0))
    return GP_ERR_INVALID;
  if (pool->step_layer_seen[layer]) return GP_ERR_STATE;          // every layer once
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const GpDev& d = pool->dev;
  const size_t qs = (size_t)layer * n_req * d.Hq * d.d, ks = (size_t)layer * n_req * d.Hkv * d.d;
  auto shifted = [](const void* ptr, size_t bytes) { return reinterpret_cast<uintptr_t>(ptr) - bytes; };
  const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(shifted(q_raw, qs * 2));
  const __nv_bfloat16* vb = reinterpret_cast<const __nv_bfloat16*>(shifted(v, ks * 2));
  float* ob = reinterpret_cast<float*>(shifted(out, qs * 4));
  const __nv_bfloat16* kb = reinterpret_cast<const __nv_bfloat16*>(shifted(k_raw, ks * 2));
  const GpNorm nm = {q_weight, k_weight, eps};
  launch_layer(pool, n_req, qb, kb, vb, ob, layer, s, nm);
  pool->launch_count += 1;
  pool->step_layers_done += 1;
  pool->step_layer_seen[layer] = 1;
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

int gp_step_end(gp_pool* pool, const int32_t* dev_req_ids, int32_t n_req, int32_t* dev_actions, void* stream) {
  if (!pool || pool->step_open != 1) return pool ? GP_ERR_STATE : GP_ERR_INVALID;
  if (n_req != pool->step_n_req || !dev_req_ids || !dev_actions) return GP_ERR_INVALID;
  if (pool->step_layers_done != pool->cfg.n_layers) return GP_ERR_STATE;       // layers missing: run them, or gp_step_abort
  GP_CUDA(cudaSetDevice(pool->device));
  gp_launch_boundary(pool->dev, dev_req_ids, n_req, dev_actions, true, pool->sel_grid, pool->compact_grid,
                     static_cast<cudaStream_t>(stream), nullptr, true, (int)(pool->serial & 0x3fffffff));
  pool->serial += 1;
  pool->launch_count += 2;
  pool->step_open = 0;
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

int gp_step_abort(gp_pool* pool) {
  if (!pool) return GP_ERR_INVALID;
  if (pool->step_open != 1) return GP_ERR_STATE;        // (a step begun with gp_decode_step_local has to be finished)
  // Nothing of an open step is committed before gp_step_end: the requests' counters are untouched, rows appended
  // by the layers that ran lie beyond the occupied slots, and the summaries went to the buffer not in use.
  pool->step_open = 0;
  pool->plain_plan = LAUNCH_RUNS | LAUNCH_CAPTURED;
  return GP_OK;
}

// ---- the step of a pool that holds a part of the model's KV heads --------------------------------------------
int gp_decode_step_local(gp_pool* pool, const int32_t* dev_req_ids, int32_t n_req, const void* q, const void* k,
                         const void* v, void* out, int32_t* dev_actions, void* stream) {
  if (!pool || n_req < 0 || n_req > pool->cfg.max_requests) return GP_ERR_INVALID;
  if (pool->step_open || pool->cfg.async_boundary) return GP_ERR_STATE;
  if (n_req == 0) return GP_OK;
  if (!dev_req_ids || !q || !k || !v || !out || !dev_actions) return GP_ERR_INVALID;
  if (misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(out, 16) ||
      misaligned(dev_req_ids, 4) || misaligned(dev_actions, 4)) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const GpDev& d = pool->dev;
  const int LH = d.L * d.Hkv;
  const int serial = (int)(pool->serial & 0x3fffffff);
  launch_plan(pool, dev_req_ids, n_req, dev_actions, false, s, true);
  gp_launch_attention(d, n_req, q, k, v, static_cast<float*>(out), pool->attn_grid, s, true, 0, LH, 0, false, false, kNoNorm);
  gp_launch_select_only(d, dev_req_ids, n_req, dev_actions, pool->sel_grid, s, true, serial);
  pool->launch_count += 3;
  pool->step_open = 2;                           // between the two halves the pool takes nothing else
  pool->step_n_req = n_req;
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

int gp_shard_sums(gp_pool* pool, int32_t** dev_sums, int64_t* n_ints) {
  if (!pool || !dev_sums || !n_ints) return GP_ERR_INVALID;
  *dev_sums = pool->dev.shard_sums;
  *n_ints = 2LL * pool->cfg.max_requests;
  return GP_OK;
}

int gp_decode_step_finish(gp_pool* pool, const int32_t* dev_req_ids, int32_t n_req, int32_t* dev_actions, void* stream) {
  if (!pool) return GP_ERR_INVALID;
  if (pool->step_open != 2) return GP_ERR_STATE;
  if (n_req != pool->step_n_req || !dev_req_ids || !dev_actions) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  gp_launch_decide_compact(pool->dev, dev_req_ids, n_req, dev_actions, pool->compact_grid, static_cast<cudaStream_t>(stream),
                           (int)(pool->serial & 0x3fffffff));
  pool->serial += 1;
  pool->launch_count += 2;
  pool->step_open = 0;
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

// The step's inputs, read from page-locked mapped host memory over the bus by one kernel: the request ids word
// by word, queries, keys and values in 16-byte pieces, every piece its own load, all in flight together (four
// separate copies cost their set-up four times).
__global__ void gp_fetch_inputs_kernel(int* __restrict__ d_ids, const int* __restrict__ s_ids, int n_ids,
                                       uint4* __restrict__ d1, const uint4* __restrict__ s1, long long n1,
                                       uint4* __restrict__ d2, const uint4* __restrict__ s2, long long n2,
                                       uint4* __restrict__ d3, const uint4* __restrict__ s3, long long n3) {
  const long long total = n1 + n2 + n3;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid < n_ids) d_ids[tid] = s_ids[tid];
  for (long long i = tid; i < total; i += (long long)gridDim.x * blockDim.x) {
    if (i < n1) d1[i] = s1[i];
    else if (i < n1 + n2) d2[i - n1] = s2[i - n1];
    else d3[i - n1 - n2] = s3[i - n1 - n2];
  }
}

extern "C" int gp_decode_step_host_wait(gp_pool* pool);
static int host_step(gp_pool* pool, const int32_t* host_req_ids, int32_t n_req, const void* q, const void* k,
                     const void* v, void* out, int32_t* actions, void* stream, bool wait) {
  if (!pool || n_req < 0 || n_req > pool->cfg.max_requests) return GP_ERR_INVALID;
  if (!pool->st_ids || pool->step_open) return GP_ERR_STATE;
  if (n_req == 0) return GP_OK;
  if (!host_req_ids || !q || !k || !v || !out || !actions) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const gp_config& c = pool->cfg;
  const size_t qb = (size_t)c.n_layers * n_req * c.n_q_heads * c.head_dim * 2;
  const size_t kb = (size_t)c.n_layers * n_req * c.n_kv_heads * c.head_dim * 2;
  // Inputs: from mapped page-locked buffers one kernel fetches all four over the bus into one of two staging sets.
  // When the caller issues steps ahead (gp_decode_step_host_async) the fetch runs on a stream of its own, beside
  // the kernels of the step before it: it waits until the step that last used the set has read it, and the step
  // waits for its fetch.  The call that waits for its step fetches on the caller's stream (nothing to overlap
  // with).  Pageable memory: four copies on the caller's stream.
  const int set = (int)(pool->host_steps & 1);
  bool staged_async = false;                 // inputs by the copy engine on the side stream (the call that does not wait)
  int* st_ids = set ? pool->st2_ids : pool->st_ids;
  void* st_q = set ? pool->st2_q : pool->st_q;
  void* st_k = set ? pool->st2_k : pool->st_k;
  void* st_v = set ? pool->st2_v : pool->st_v;
  {
    void *mi = nullptr, *mq = nullptr, *mk = nullptr, *mv = nullptr;
    const bool mapped = ((uintptr_t)host_req_ids % 4 == 0) && ((uintptr_t)q % 16 == 0) && ((uintptr_t)k % 16 == 0) &&
                        ((uintptr_t)v % 16 == 0) &&
                        cudaHostGetDevicePointer(&mi, const_cast<int32_t*>(host_req_ids), 0) == cudaSuccess &&
                        cudaHostGetDevicePointer(&mq, const_cast<void*>(q), 0) == cudaSuccess &&
                        cudaHostGetDevicePointer(&mk, const_cast<void*>(k), 0) == cudaSuccess &&
                        cudaHostGetDevicePointer(&mv, const_cast<void*>(v), 0) == cudaSuccess;
    if (mapped && wait) {
      const long long pieces = (long long)(qb + 2 * kb) / 16;         // a row is 128 or 256 bytes: whole pieces
      int grid = (int)((pieces + 255) / 256);
      if (grid > pool->num_sms * 8) grid = pool->num_sms * 8;
      if (grid * 256 < n_req) grid = (n_req + 255) / 256;
      gp_fetch_inputs_kernel<<<grid, 256, 0, s>>>(st_ids, static_cast<const int*>(mi), n_req,
                                                 static_cast<uint4*>(st_q), static_cast<const uint4*>(mq), (long long)qb / 16,
                                                 static_cast<uint4*>(st_k), static_cast<const uint4*>(mk), (long long)kb / 16,
                                                 static_cast<uint4*>(st_v), static_cast<const uint4*>(mv), (long long)kb / 16);
      pool->launch_count++;
    } else if (mapped) {
      if (!pool->fetch_stream) {
        GP_CUDA(cudaStreamCreateWithFlags(&pool->fetch_stream, cudaStreamNonBlocking));
        for (int i = 0; i < 2; ++i) {
          GP_CUDA(cudaEventCreateWithFlags(&pool->ev_fetch[i], cudaEventDisableTiming));
          GP_CUDA(cudaEventCreateWithFlags(&pool->ev_used[i], cudaEventDisableTiming));
          GP_CUDA(cudaEventCreateWithFlags(&pool->ev_out[i], cudaEventDisableTiming));
          GP_CUDA(cudaEventRecord(pool->ev_used[i], s));
          GP_CUDA(cudaEventRecord(pool->ev_out[i], s));
        }
      }
      cudaStream_t fs = pool->fetch_stream;
      GP_CUDA(cudaStreamWaitEvent(fs, pool->ev_used[set], 0));
      // Copies by the copy engine here, not the fetch kernel: they run beside the step before, whose attention
      // kernel fills every SM's registers; a kernel that reads over the bus for 15 us held some of them and kept
      // that step's attention thread blocks from starting (11 us per step).  The copies' set-up time, which is
      // what the fetch kernel saves the call that waits, is hidden here.
      GP_CUDA(cudaMemcpyAsync(st_ids, host_req_ids, (size_t)n_req * 4, cudaMemcpyHostToDevice, fs));
      GP_CUDA(cudaMemcpyAsync(st_q, q, qb, cudaMemcpyHostToDevice, fs));
      GP_CUDA(cudaMemcpyAsync(st_k, k, kb, cudaMemcpyHostToDevice, fs));
      GP_CUDA(cudaMemcpyAsync(st_v, v, kb, cudaMemcpyHostToDevice, fs));
      GP_CUDA(cudaEventRecord(pool->ev_fetch[set], fs));
      GP_CUDA(cudaStreamWaitEvent(s, pool->ev_fetch[set], 0));
      staged_async = true;
    } else {
      (void)cudaGetLastError();                    // pageable memory: not an error
      GP_CUDA(cudaMemcpyAsync(st_ids, host_req_ids, (size_t)n_req * 4, cudaMemcpyHostToDevice, s));
      GP_CUDA(cudaMemcpyAsync(st_q, q, qb, cudaMemcpyHostToDevice, s));
      GP_CUDA(cudaMemcpyAsync(st_k, k, kb, cudaMemcpyHostToDevice, s));
      GP_CUDA(cudaMemcpyAsync(st_v, v, kb, cudaMemcpyHostToDevice, s));
    }
  }
  pool->host_steps += 1;
  // Outputs: when the caller's buffers are page-locked and mapped (the usual pinned allocation), the kernels
  // write them over the bus while they run and nothing is left to copy when the step ends.  (The same was tried
  // for the inputs and was slower: rows read over the bus by the kernels stall the pipelines that wait for them.)
  void* d_out = nullptr;
  void* d_act = nullptr;
  const bool direct = cudaHostGetDevicePointer(&d_out, out, 0) == cudaSuccess &&
                      cudaHostGetDevicePointer(&d_act, actions, 0) == cudaSuccess;
  if (!direct) (void)cudaGetLastError();           // pageable memory: not an error, the staged path takes over
  // (Results through a staging set and the copy engine on a third stream, beside the next step, were tried for the
  // call that does not wait: a megabyte takes the copy engine and the event that reports it 60 us, longer than the
  // host may lag behind when it reads every step's results before it issues the step after the next: 92 us per
  // step against 78 with the kernels writing the rows over the bus themselves.)
  float* st_out = pool->st_out;
  int* st_act = pool->st_act;
  if (staged_async && pool->host_async_issued - pool->host_waited >= 2) {          // two calls outstanding: the older first
    const int st0 = gp_decode_step_host_wait(pool);
    if (st0 != GP_OK) return st0;
  }
  // The inputs arrive by the fetch kernel or the copies above, which end before the plan kernel starts: that
  // kernel is launched the plain way here (not as a programmatic dependent of the fetch kernel, whose stores it
  // reads), so planning ahead of its wait, which is then no wait at all, is safe whatever the option says.
  const int early = pool->early_plan;
  pool->early_plan = 1;
  pool->first_plain = 1;
  // The actions: the plan kernel writes them all and the decisions overwrite some; written straight to host memory
  // they made the plan kernel wait for the bus.  With the boundary work in one kernel they stay on the device and
  // that kernel copies them to the caller's array once they are final (beside its compaction).
  const bool act_late = direct && !pool->cfg.async_boundary && pool->chain_grid_ov > 0;
  pool->actions_copy = act_late ? static_cast<int32_t*>(d_act) : nullptr;
  const int st = gp_decode_step(pool, st_ids, n_req, st_q, st_k, st_v,
                                direct ? d_out : static_cast<void*>(st_out),
                                direct && !act_late ? static_cast<int32_t*>(d_act) : st_act, stream);
  pool->actions_copy = nullptr;
  pool->early_plan = early;
  pool->first_plain = 0;
  if (st != GP_OK) return st;
  if (pool->fetch_stream) GP_CUDA(cudaEventRecord(pool->ev_used[set], s));       // the set may be fetched into again
  if (!direct) {
    GP_CUDA(cudaMemcpyAsync(out, st_out, qb * 2, cudaMemcpyDeviceToHost, s));
    GP_CUDA(cudaMemcpyAsync(actions, st_act, (size_t)n_req * 4, cudaMemcpyDeviceToHost, s));
  }
  if (staged_async) {                          // what gp_decode_step_host_wait waits for: this call's work on `stream`
    GP_CUDA(cudaEventRecord(pool->ev_out[set], s));
    pool->host_async_set[pool->host_async_issued & 1] = set;
    pool->host_async_issued += 1;
  }
  if (!wait) return GP_OK;
  GP_CUDA(cudaStreamSynchronize(s));
  return kernel_status(pool);
}

int gp_decode_step_host(gp_pool* pool, const int32_t* host_req_ids, int32_t n_req, const void* q, const void* k,
                        const void* v, void* out, int32_t* actions, void* stream) {
  return host_step(pool, host_req_ids, n_req, q, k, v, out, actions, stream, true);
}

int gp_decode_step_host_async(gp_pool* pool, const int32_t* host_req_ids, int32_t n_req, const void* q, const void* k,
                              const void* v, void* out, int32_t* actions, void* stream) {
  return host_step(pool, host_req_ids, n_req, q, k, v, out, actions, stream, false);
}

int gp_decode_step_host_wait(gp_pool* pool) {
  if (!pool) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (pool->host_waited < pool->host_async_issued) {
    GP_CUDA(cudaEventSynchronize(pool->ev_out[pool->host_async_set[pool->host_waited & 1]]));
    pool->host_waited += 1;
  } else {
    GP_CUDA(cudaDeviceSynchronize());        // nothing of that kind outstanding: whatever else the pool has in flight
  }
  return kernel_status(pool);
}

int gp_pool_status(gp_pool* pool, int32_t* error_bits) {
  if (!pool) return GP_ERR_INVALID;
  const int e = *reinterpret_cast<volatile const int*>(pool->h_err);
  if (error_bits) *error_bits = e;
  return e ? GP_ERR_CUDA : GP_OK;
}

int gp_release(gp_pool* pool, int32_t req, void* stream) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  if (pool->step_open) return GP_ERR_STATE;      // the open step's plan holds a snapshot of the free list
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, static_cast<cudaStream_t>(stream)) != GP_OK) return GP_ERR_CUDA;
  gp_release_kernel<<<1, ADMIT_THREADS, 0, static_cast<cudaStream_t>(stream)>>>(pool->dev, req);
  pool->launch_count++;
  pool->plain_plan |= launch_kind(static_cast<cudaStream_t>(stream));
  pool->live[req] = 0;
  if (pool->chain_clusters && pool->began[req] == pool->began_max) {
    pool->began_max = -pool->serial;
    for (int i = 0; i < pool->cfg.max_requests; ++i)
      if (pool->live[i] && pool->began[i] > pool->began_max) pool->began_max = pool->began[i];
  }
  GP_CUDA(cudaGetLastError());
  return GP_OK;
}

const char* gp_strerror(int status) {
  switch (status) {
    case GP_OK: return "ok";
    case GP_ERR_INVALID: return "invalid argument or request id";
    case GP_ERR_NO_SLOT: return "no free request slot";
    case GP_ERR_NO_PAGES: return "not enough free pages or per-request cap exceeded";
    case GP_ERR_CUDA: return "CUDA error or internal kernel error";
    case GP_ERR_STATE: return "call not possible in this state";
    case GP_ERR_TOO_LARGE: return "problem exceeds the fixed scratch of the no-allocation entry point";
    default: return "unknown status";
  }
}

// ---- introspection ---------------------------------------------------------------------------------
int gp_debug_request(gp_pool* pool, int32_t req, int32_t* P, int32_t* n, int64_t* pos, int32_t* page_table) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  int Pv = 0, nv = 0; long long pv = 0;
  GP_CUDA(cudaMemcpy(&Pv, pool->dev.P + req, 4, cudaMemcpyDeviceToHost));
  GP_CUDA(cudaMemcpy(&nv, pool->dev.n + req, 4, cudaMemcpyDeviceToHost));
  GP_CUDA(cudaMemcpy(&pv, pool->dev.pos + req, 8, cudaMemcpyDeviceToHost));
  if (P) *P = Pv / (pool->cfg.page_size / GP_PAGE);
  if (n) *n = nv;
  if (pos) *pos = pv;
  if (page_table && Pv > 0)
  {
    // pages of the method: the group of tiles that starts at table entry j * sub (see gp_debug_pool)
    const int sub = pool->cfg.page_size / GP_PAGE;
    std::vector<int> tiles((size_t)Pv);
    GP_CUDA(cudaMemcpy(tiles.data(), pool->dev.page_table + (size_t)req * pool->dev.cap, (size_t)Pv * 4, cudaMemcpyDeviceToHost));
    for (int j = 0; j < Pv / sub; ++j) page_table[j] = tiles[(size_t)j * sub] / sub;
  }
  return GP_OK;
}

int gp_debug_state(gp_pool* pool, int32_t* P, int32_t* n) {
  if (!pool) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  const int M = pool->cfg.max_requests;
  const size_t nb = (size_t)M * 4;
  if (P) GP_CUDA(cudaMemcpy(P, pool->dev.P, nb, cudaMemcpyDeviceToHost));
  if (n) GP_CUDA(cudaMemcpy(n, pool->dev.n, nb, cudaMemcpyDeviceToHost));
  if (P) for (int i = 0; i < M; ++i) P[i] /= pool->cfg.page_size / GP_PAGE;
  return GP_OK;
}

static int gather_stream(gp_pool* pool, int32_t req, int32_t layer, int32_t kv_head, int* n_out) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  if (layer < 0 || layer >= pool->cfg.n_layers || kv_head < 0 || kv_head >= pool->cfg.n_kv_heads) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  int nv = 0;
  GP_CUDA(cudaMemcpy(&nv, pool->dev.n + req, 4, cudaMemcpyDeviceToHost));
  *n_out = nv;
  if (nv == 0) return GP_OK;
  const size_t cap_tok = (size_t)pool->cfg.max_pages_per_req * pool->cfg.page_size;
  int* tok = reinterpret_cast<int*>(pool->dbg);
  uint4* kk = reinterpret_cast<uint4*>(pool->dbg + cap_tok * 4);
  uint4* vv = reinterpret_cast<uint4*>(pool->dbg + cap_tok * 4 + cap_tok * pool->cfg.head_dim * 2);
  gp_gather_kernel<<<148, 256>>>(pool->dev, req, layer, kv_head, nv, tok, kk, vv);
  pool->launch_count++;
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  return GP_OK;
}

int gp_debug_retained(gp_pool* pool, int32_t req, int32_t layer, int32_t kv_head, int32_t* token_ids) {
  if (!token_ids) return GP_ERR_INVALID;
  int n = 0;
  const int st = gather_stream(pool, req, layer, kv_head, &n);
  if (st != GP_OK) return st;
  if (n > 0) GP_CUDA(cudaMemcpy(token_ids, pool->dbg, (size_t)n * 4, cudaMemcpyDeviceToHost));
  return GP_OK;
}

int gp_debug_kv(gp_pool* pool, int32_t req, int32_t layer, int32_t kv_head, void* k_rows, void* v_rows) {
  int n = 0;
  const int st = gather_stream(pool, req, layer, kv_head, &n);
  if (st != GP_OK) return st;
  const size_t cap_tok = (size_t)pool->cfg.max_pages_per_req * pool->cfg.page_size;
  const size_t rowb = (size_t)pool->cfg.head_dim * 2;
  if (n > 0 && k_rows) GP_CUDA(cudaMemcpy(k_rows, pool->dbg + cap_tok * 4, n * rowb, cudaMemcpyDeviceToHost));
  if (n > 0 && v_rows)
    GP_CUDA(cudaMemcpy(v_rows, pool->dbg + cap_tok * 4 + cap_tok * rowb, n * rowb, cudaMemcpyDeviceToHost));
  return GP_OK;
}

int gp_debug_summaries(gp_pool* pool, int32_t req, double* out) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  if (!out) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  const gp_config& c = pool->cfg;
  int par = 0;
  GP_CUDA(cudaMemcpy(&par, pool->dev.sum_par + req, 4, cudaMemcpyDeviceToHost));
  const size_t per = (size_t)2 * c.n_q_heads * c.head_dim;
  for (int l = 0; l < c.n_layers; ++l)
    GP_CUDA(cudaMemcpy(out + (size_t)l * per, pool->dev.summ + (((size_t)l * c.max_requests + req) * 2 + par) * per,
                       per * 8, cudaMemcpyDeviceToHost));
  return GP_OK;
}

int gp_debug_boundary(gp_pool* pool, int32_t req, int32_t* K_S, int32_t* K_L, double* delta) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  const int LH = pool->cfg.n_layers * pool->cfg.n_kv_heads;
  std::vector<int> kx((size_t)LH * 2);
  GP_CUDA(cudaMemcpy(kx.data(), pool->dev.Kx + (size_t)req * LH * 2, (size_t)LH * 8, cudaMemcpyDeviceToHost));
  for (int i = 0; i < LH; ++i) {
    if (K_S) K_S[i] = kx[2 * i];
    if (K_L) K_L[i] = kx[2 * i + 1];
  }
  if (delta) GP_CUDA(cudaMemcpy(delta, pool->dev.delta + req, 8, cudaMemcpyDeviceToHost));
  return GP_OK;
}

int gp_debug_entropy(gp_pool* pool, int32_t req, double* H_S, double* H_L) {
  const int st = check_req(pool, req);
  if (st != GP_OK) return st;
  if (pool->cfg.demand_metric != GP_METRIC_ENTROPY) return GP_ERR_STATE;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  const int LH = pool->cfg.n_layers * pool->cfg.n_kv_heads;
  std::vector<double> hx((size_t)LH * 2);
  GP_CUDA(cudaMemcpy(hx.data(), pool->dev.Hx + (size_t)req * LH * 2, (size_t)LH * 16, cudaMemcpyDeviceToHost));
  for (int i = 0; i < LH; ++i) {
    if (H_S) H_S[i] = hx[2 * i];
    if (H_L) H_L[i] = hx[2 * i + 1];
  }
  return GP_OK;
}

int gp_debug_pool(gp_pool* pool, int64_t* n_free, int32_t* refcounts, int64_t counters[12]) {
  if (!pool) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  int top = 0;
  GP_CUDA(cudaMemcpy(&top, pool->dev.free_top, 4, cudaMemcpyDeviceToHost));
  const int err = *reinterpret_cast<volatile const int*>(pool->h_err);
  if (n_free) *n_free = top / (pool->cfg.page_size / GP_PAGE);
  if (refcounts) {
    // One count per page of the method.  Its 16-token tiles are taken from the free list, shared and returned
    // together and in whole aligned groups (the list starts in tile order and every pop and push is a multiple of
    // the group), so page i is tiles [i * sub, (i + 1) * sub) and its count is that of its first tile.
    const int sub = pool->cfg.page_size / GP_PAGE;
    std::vector<int> ref((size_t)pool->dev.n_pages);
    GP_CUDA(cudaMemcpy(ref.data(), pool->dev.refcount, ref.size() * 4, cudaMemcpyDeviceToHost));
    for (long long i = 0; i < pool->cfg.n_pages; ++i) refcounts[i] = ref[(size_t)i * sub];
  }
  if (counters) {
    long long c[12];
    GP_CUDA(cudaMemcpy(c, pool->dev.counters, 96, cudaMemcpyDeviceToHost));
    for (int i = 0; i < 12; ++i) counters[i] = c[i];
    counters[4] /= pool->cfg.page_size / GP_PAGE;          // copy-on-write: counted per 16-token tile, reported per page
    counters[7] = err;
  }
  return GP_OK;
}

int gp_test_withhold(gp_pool* pool, int32_t what, int32_t spin_limit) {
  if (!pool || what < 0 || what > 63 || spin_limit < 0) return GP_ERR_INVALID;
  GpDev* views[2] = {&pool->dev, &pool->dev_alt};
  for (GpDev* v : views) {
    v->withhold = what;
    v->spin_limit = spin_limit > 0 ? (unsigned)spin_limit : GP_SPIN_LIMIT;
  }
  return GP_OK;
}

int gp_set_early_plan(gp_pool* pool, int32_t enable) {
  if (!pool) return GP_ERR_INVALID;
  pool->early_plan = enable ? 1 : 0;
  return GP_OK;
}

int gp_set_profiling(gp_pool* pool, int32_t enable) {
  if (!pool) return GP_ERR_INVALID;
  pool->profiling = enable ? 1 : 0;
  memset(pool->ms, 0, sizeof(pool->ms));
  memset(pool->launches, 0, sizeof(pool->launches));
  return GP_OK;
}

int gp_get_kernel_times(gp_pool* pool, float* ms, int64_t* launches) {
  if (!pool) return GP_ERR_INVALID;
  GP_CUDA(cudaSetDevice(pool->device));
  if (flush_chain(pool, pool->last_stream) != GP_OK) return GP_ERR_CUDA;
  GP_CUDA(cudaDeviceSynchronize());
  for (int i = 0; i < GP_N_KERNELS; ++i) {
    if (ms) ms[i] = pool->ms[i];
    if (launches) launches[i] = pool->launches[i];
  }
  memset(pool->ms, 0, sizeof(pool->ms));
  memset(pool->launches, 0, sizeof(pool->launches));
  return GP_OK;
}

int64_t gp_launch_count(gp_pool* pool) { return pool ? pool->launch_count : 0; }

}  // extern "C"
