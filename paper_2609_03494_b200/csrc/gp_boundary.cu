// Capacity-boundary work (Sec. 3.2 - 3.3, App. D.1, App. D.2), every step, behind the attention kernel.
// That kernel leaves, for every (request at a boundary, layer, KV head) unit and both calibrated summaries,
// exp(logit - the page's maximum logit) of every candidate key, and per 16-token page the maximum and the sum of
// those exponentials.  The work on them, in the order of its dependences:
//
//   selection         per unit, one CTA: per-head softmax over the candidate set and group mean -> a^S and a^L;
//                     then, side by side on warps of their own, the working-set sizes K^S and K^L (Eq. 7) and,
//                     speculatively, the b slots a compression would evict (Eq. 9, Eq. 10).  Under the Shrink policy
//                     the 2b slots a Shrink would evict as well (Eq. 13).
//   decisions         by the CTA that finishes its jobs last: Eq. 8 per request, the action (grow, compress,
//                     shrink), the device allocator: grants first, then copy-on-write targets, each in ascending
//                     request id.
//   compaction        per compressing unit: stable in-place compaction into (P-1) b slots ((P-2) b at a Shrink):
//                     the rows behind the new end fill the evicted slots before it, the order of the tokens is kept in
//                     a word per slot; shared pages are copied to their targets.  Work is claimed from a
//                     ticket counter.  The last CTA swaps in the target pages, drops the references to the replaced ones
//                     and returns the last page of every request that shrank.
//
// It comes in two shapes that run the same device functions:
//   gp_chain_kernel                       all of it in one kernel (the deciding CTA tells the others through a flag):
//                                         behind the attention kernel of its own step, with every job waiting for the
//                                         attention kernel's report that its unit is complete (synchronous mode), or
//                                         beside the attention kernel of the next step (asynchronous mode);
//   gp_bsel_kernel, gp_compact_kernel     selection + decisions, then compaction, as kernels of their own
//   (and gp_decide_kernel)                (large pools, the layer-by-layer step; with the KV heads spread over several
//                                         pools the decisions wait for the sums of all pools in a kernel of their own).
//
// Everything that decides an integer outcome is fp64.  Top-p counting and the eviction cut work on the IEEE bit
// patterns of the (non-negative) scores: a radix descent, 8 bits per level from the first bit in which the unit's
// scores differ, until the bin with the crossing point holds at most 32 scores, which one warp sorts.  The top-p mass
// is accumulated in 2^62 fixed point with integer atomics, so the result does not depend on the order in which
// threads add.
//
// Size of the code: a step of a few units runs these functions once per thread block, and what they then cost is the fetch of their
// instructions.  So loops whose trips are not the point are kept from being unrolled (`unroll 1`; the compiler unrolled the loop over the two
// supports, and the decisions' loops four to eight times): gp_chain_kernel<128, 4> 258 -> 170 KB (its form in clusters, which holds both ways of taking a unit,
// 272), the compaction 62 -> 52, the decisions 26 -> 17.  us a pass before / now: one layer x 64 requests, 16 steps, 1067 / 1039; four requests, 16 steps, 267 / 259; 256 requests copied
// on write in one of 24 steps 14 315 / 13 979; 36 layers x 16, 16 steps, 4912 / 4897.
#include "../../include/growpage.h"
#include "gp_dev.cuh"

namespace {

constexpr double TWO62 = 4611686018427387904.0;
constexpr int SEL_T = 256;           // threads of the selection kernel
constexpr int SEL_NW = SEL_T / 32;
constexpr int SEL_CAP = 5120;        // candidate tokens whose scores (both views) are kept in shared memory, at most
constexpr int CT = 256;              // threads of the compaction kernel
constexpr int CMP_SHRINK = 1 << 30;       // flag on a compressing request's boundary index: the action is a Shrink
constexpr int CMP_LOG = 16;               // ... and from this bit on log2 of the slots of a ticket
static_assert(GP_MAX_REQ <= 1 << CMP_LOG, "a boundary index fits below");

__device__ __forceinline__ unsigned long long to_fix(double a) {
  return (unsigned long long)__double2ll_rn(a * TWO62);
}

// log2 of the slots of a compaction ticket (test support: see GP_WITHHOLD_CHUNK).  A unit's last ticket has what lies behind its new end too.
__device__ __forceinline__ int part_log_of(const GpDev& p, int want) {
  if (p.withhold & GP_TEST_COMPACT_BY_UNIT) return GP_PART_LOG_UNIT;
  return (p.withhold & (GP_WITHHOLD_CHUNK | GP_TEST_COMPACT_BY_PART)) ? GP_PART_LOG_MIN : want;
}

// ------------------------------------------------------------------------------------------------------
// decision + allocator, run by the last CTA of the selection kernel
// ------------------------------------------------------------------------------------------------------
__device__ void decide_and_allocate(const GpDev& p, const int* req_ids, int n_req, int n_bnd, int* actions, int* s_arr,
                                    int serial, bool from_sums = false) {
  // from_sums: the sums of K^S and K^L come from shard_sums (summed over the pools that hold the model's other KV
  // heads) instead of this pool's own accumulators
  // In the asynchronous boundary mode this runs beside the next decode step: it touches only the requests at
  // this step's boundary (which sit that step out), reads the free list itself (the boundary chains run one
  // after the other and nothing else takes or returns pages meanwhile) and reports through last_act only
  // (`actions` is null: the caller's array belongs to a step that has ended).
  int* s_want = s_arr;
  int* s_ksh = s_arr + GP_MAX_REQ;
  int* s_P = s_arr + 2 * GP_MAX_REQ;
  int* s_order = s_arr + 3 * GP_MAX_REQ;
  int* s_req = s_arr + 4 * GP_MAX_REQ;
  int* s_base = s_arr + 5 * GP_MAX_REQ;
  int* s_bi = s_arr + 6 * GP_MAX_REQ;
  int* s_free = s_arr + 7 * GP_MAX_REQ;      // the free pages the grants of this step can take, top first
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarp = blockDim.x >> 5;
  // everything the decisions need arrives in one round trip: the jobs summed K^S and K^L per request, a job
  // counted its shared pages, and the plan kernel copied the top of the free list
  const int LH = p.L * p.Hkv;
  const int n_active = p.hdr[HDR_N_ACTIVE];
  int top0 = 0;
  if (n_bnd > 0) {
    top0 = p.async ? __ldcg(p.free_top) : __ldcg(p.free_peek);
#pragma unroll 1
    for (int e = tid; e < n_bnd; e += blockDim.x) {
      const int4 inf = p.bnd_info[2 * e], inf2 = p.bnd_info[2 * e + 1];
      int4 acc = __ldcg(reinterpret_cast<const int4*>(p.bnd_acc) + e);
      if (from_sums) { acc.x = __ldcg(p.shard_sums + 2 * e); acc.y = __ldcg(p.shard_sums + 2 * e + 1); }
      s_free[e] = p.async ? (e < top0 ? __ldcg(p.free_stack + top0 - 1 - e) : 0) : __ldcg(p.free_peek + 1 + e);
      const int r = inf.y, Pr = inf.z;
      const int nC = (Pr - p.sub) * GP_PAGE;                // |C_t| of Eq. 7: history minus the newest page of the method
      // Eq. 8 with a common |C|: Delta = (sum K^S - sum K^L) / (N |C|), one division of exact integers
      double delta = 0.0;
      int want = 1;
      if (nC > 0) {
        delta = (double)((long long)acc.x - (long long)acc.y) / ((double)p.units_total * (double)nC);
        if (p.metric == GP_METRIC_ENTROPY) {
          // the same mean with H / ln |C| in the place of K / |C|, summed unit by unit in (layer, head) order
          const double* hx = p.Hx + (size_t)r * LH * 2;
          double accd = 0.0;
#pragma unroll 1
          for (int u2 = 0; u2 < LH; ++u2) accd += __ldcg(hx + 2 * u2) - __ldcg(hx + 2 * u2 + 1);
          delta = nC > 1 ? accd / ((double)LH * log((double)nC)) : 0.0;
        }
        want = delta > p.tau;
        if (p.policy == 1) {                                  // the reversed reading of the demand signal
          want = !want;
        } else if (p.policy == 2) {                           // frequency-matched random control
          unsigned long long zz = p.policy_seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(r + 1) +
                                  0xBF58476D1CE4E5B9ull * (unsigned long long)inf.w;
          zz = (zz ^ (zz >> 30)) * 0xBF58476D1CE4E5B9ull;
          zz = (zz ^ (zz >> 27)) * 0x94D049BB133111EBull;
          zz ^= zz >> 31;
          want = !((double)(zz >> 11) * (1.0 / 9007199254740992.0) < p.p_compress);
        } else if (p.policy == GP_POLICY_SHRINK) {            // Eq. 13: the third action, where it is admissible
          if (!want && delta < p.shrink_below && Pr - p.sub >= p.min_pages_after_shrink) want = 16;
        }
      }
      p.delta[r] = delta;
      // pages and slots as the step left them (full); the allocator below changes what the decision changes.  In
      // the asynchronous mode the plan of the step in between leaves these two words of a held request alone.
      p.P[r] = Pr; p.n[r] = Pr * GP_PAGE;
      p.cmp_off[e] = (long long)(unsigned)inf2.x | ((long long)inf2.y << 32);
      s_want[e] = want; s_ksh[e] = acc.z; s_P[e] = Pr; s_req[e] = r; s_bi[e] = inf.x;
    }
  }
  if (tid == 0) {
    atomicAdd(reinterpret_cast<unsigned long long*>(p.counters + 5), 1ull);
    atomicAdd(reinterpret_cast<unsigned long long*>(p.counters + 6), (unsigned long long)n_active);
    p.hdr[HDR_WORK_CMP] = 0;
    if (n_bnd == 0) { p.hdr[HDR_N_CMP] = 0; p.hdr[HDR_N_CITEM] = 0; p.hdr[HDR_N_COW] = 0; }
  }
  if (n_bnd == 0) return;
  __syncthreads();
#pragma unroll 1
  for (int e = tid; e < n_bnd; e += blockDim.x) {
    int rank = 0;
#pragma unroll 2
    for (int f = 0; f < n_bnd; ++f) rank += (s_req[f] < s_req[e]);
    s_order[rank] = e;
  }
  __syncthreads();
  auto report = [&](int bi, int r, int act) {
    if (actions) actions[bi] = act;
    p.last_act[r] = act;
  };
  if (tid == 0) {                                        // sequential allocator: shared memory only
    int top = top0;
    int n_cmp = 0, chunks = 0;
    unsigned long long grow = 0, comp = 0, fall = 0, stall = 0, cow = 0, scored = 0, shr = 0;
    const int sub = p.sub;
#pragma unroll 1
    for (int k = 0; k < n_bnd; ++k) {                    // pass 1: grants, ascending request id
      const int e = s_order[k];
      const int r = s_req[e], Pr = s_P[e], bi = s_bi[e];
      scored += (unsigned long long)(Pr - sub) * GP_PAGE;
      if ((s_want[e] & 1) && Pr + sub <= p.cap && top >= sub) {
        // one page of the method: `sub` tiles from the top of the free list
#pragma unroll 1
        for (int t = 0; t < sub; ++t) {
          const int page = (sub == 1 && !p.async) ? s_free[top0 - top] : p.free_stack[top - 1];
          --top;
          p.refcount[page] = 1;
          p.page_table[(size_t)r * p.cap + Pr + t] = page;
        }
        p.P[r] = Pr + sub;
        report(bi, r, GP_ACT_GROW);
        s_want[e] |= 2;
        ++grow;
      } else if (Pr == sub) {
        report(bi, r, GP_ACT_STALLED);
        s_want[e] |= 4;
        ++stall;
      }
    }
    int copies = -1;                                     // tiles per (layer, KV head) that this pass may have copied
    // Units whose pages are shared are copied tile by tile, 8 KB each at d = 128.  Where they are too few for the grid (one has more than
    // twice a thread block's even share of the tiles) they are cut into parts of about a quarter of that share, of eight tiles at least.
    // Requests of 2048 tokens that share a prompt, us of the step in which all are copied, by units / cut (one layer, 8 KV heads): 2 requests
    // 127 / 88, 4 148 / 106, 8 173 / 141, 16 227 / 211; cut all the same: 32 312 / 320, 4 layers x 16 494 / 519.
#pragma unroll 1
    for (int k = 0; k < n_bnd; ++k) {                    // pass 2: copy-on-write targets
      const int e = s_order[k];
      if (s_want[e] & 6) continue;
      const int r = s_req[e], bi = s_bi[e];
      if (s_ksh[e] > top) {
        report(bi, r, GP_ACT_STALLED);
        ++stall;
        continue;
      }
      s_base[e] = top;
      top -= s_ksh[e];
      cow += s_ksh[e];
      const bool shrink = (s_want[e] & 16) != 0;
      int log = GP_PART_LOG;
      if (s_ksh[e] > 8) {
        if (copies < 0) {
          copies = 0;
#pragma unroll 1
          for (int f = 0; f < n_bnd; ++f) copies += (s_want[f] & 6) ? 0 : s_ksh[f];
        }
        const float share = (float)copies * p.copy_share;
        if ((float)s_ksh[e] > 2.f * share) log = min(log, max(7, 33 - __clz((int)(1.5f * share))));
      }
      log = part_log_of(p, log);
      p.cmp_info[n_cmp] = make_int4(r, s_P[e], e | log << CMP_LOG | (shrink ? CMP_SHRINK : 0), chunks);
      chunks += ((s_P[e] - (shrink ? 2 : 1) * sub) * GP_PAGE + (1 << log) - 1) >> log;
      ++n_cmp;
      if (s_want[e] & 1) { report(bi, r, GP_ACT_COMPRESS_FALLBACK); ++fall; }
      else if (shrink) { report(bi, r, GP_ACT_SHRINK); ++shr; }
      else { report(bi, r, GP_ACT_COMPRESS); ++comp; }
      // a compression frees one page worth of slots; a Shrink frees two and gives the last page back (the
      // compaction kernel returns it once nothing reads it any more)
      p.n[r] = (s_P[e] - (shrink ? 2 : 1) * sub) * GP_PAGE;
      if (shrink) p.P[r] = s_P[e] - sub;
      p.n_pristine[r] = 0;
      s_want[e] |= 8;
    }
    p.cmp_info[n_cmp] = make_int4(0, 0, 0, chunks);
    if (top < 0) atomicOr(p.err, GP_E_FREELIST);
    *p.free_top = top;
    p.hdr[HDR_N_CMP] = n_cmp;
    p.hdr[HDR_N_CITEM] = chunks * LH;
    p.hdr[HDR_N_COW] = (int)(cow + shr);           // page-table work left for the compaction kernel's last CTA
    unsigned long long* cn = reinterpret_cast<unsigned long long*>(p.counters);
    if (grow) atomicAdd(cn + 0, grow);
    if (comp) atomicAdd(cn + 1, comp);
    if (fall) atomicAdd(cn + 2, fall);
    if (stall) atomicAdd(cn + 3, stall);
    if (cow) atomicAdd(cn + 4, cow);
    if (shr) atomicAdd(cn + 10, shr);
    atomicAdd(cn + 9, scored);
  }
  __syncthreads();
#pragma unroll 1
  for (int e = warp; e < n_bnd; e += nwarp) {             // fill in the targets, in table order
    if (!(s_want[e] & 8) || s_ksh[e] == 0) continue;
    const int r = s_req[e], Pr = s_P[e], base = s_base[e];
    const int* table = p.page_table + (size_t)r * p.cap;
    int* shadow = p.shadow + (size_t)r * p.cap;
    int running = 0;
#pragma unroll 1
    for (int j0 = 0; j0 < Pr - p.sub; j0 += 32) {
      const int j = j0 + lane;
      const bool sh = j < Pr - p.sub && p.refcount[table[j]] > 1;
      const unsigned mask = __ballot_sync(0xffffffffu, sh);
      if (sh) {
        const int newp = p.free_stack[base - 1 - (running + __popc(mask & ((1u << lane) - 1u)))];
        shadow[j] = newp;
        p.refcount[newp] = 1;
      }
      running += __popc(mask);
    }
  }
}

// L2 loads the compiler may not sink towards their first use: the selection issues all loads of a phase together and
// only then waits (a plain load is free to drift past the block barriers in between)
__device__ __forceinline__ double2 ld_early2(const double* ptr) {
  double2 v;
  asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(ptr));
  return v;
}
// the GG values of one token and view: 8, 16, 32 or 64 contiguous bytes
template <int GG>
__device__ __forceinline__ void ld_early_row(const double* ptr, double* v) {
  if (GG == 1) asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v[0]) : "l"(ptr));
  else if (GG == 2) asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1 % GG]) : "l"(ptr));
  else {
#pragma unroll
    for (int i = 0; i < GG; i += 4)
      asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];"
                   : "=d"(v[i]), "=d"(v[(i + 1) % GG]), "=d"(v[(i + 2) % GG]), "=d"(v[(i + 3) % GG]) : "l"(ptr + i));
  }
}

// max or sum over the block of one value per thread, separately for each of `ncols` interleaved columns
// (thread t belongs to column t % ncols); fixed shuffle tree, so the sum does not depend on timing
template <bool IS_MAX>
__device__ __forceinline__ void column_reduce(double v, int ncols, double* red, double* result) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int off = ncols; off < 32; off <<= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, v, off);
    v = IS_MAX ? fmax(v, o) : v + o;
  }
  if (lane < ncols) red[warp * 16 + lane] = v;
  __syncthreads();
  if (threadIdx.x < ncols) {
    double r = red[threadIdx.x];
#pragma unroll 1
    for (int w = 1; w < SEL_T / 32; ++w) r = IS_MAX ? fmax(r, red[w * 16 + threadIdx.x]) : r + red[w * 16 + threadIdx.x];
    result[threadIdx.x] = r;
  }
  __syncthreads();
}

// shared memory of the selection; the arrays of scores come last, their size follows the pool's page cap
constexpr int BIN_STRIDE = 256 + 32;              // 256 bins at b + (b >> 3): a lane's 8 bins and its neighbours' in other banks
#define BIDX(b) ((b) + ((b) >> 3))
constexpr int SEL_F = 1024;                       // page factors in shared memory at a time
struct SelMisc {
  double red[SEL_NW * 16];
  double sM[16], sZ[16];                          // per column (view, head): maximum logit, 1 / (G sum of exponentials)
  unsigned long long list[3][32], list_fix[2][32];     // members of the crossing bin, per task: bit pattern, fixed-point mass
  int list_slot[32];
  unsigned rng[3][2];                             // smallest and largest high word of a^S, a^L and max(a^S, a^L)
  long long res[3][4];                            // crossing bin, members and mass before it, members in it
  int cnt[4];                                     // evicted slots listed, list members per task
  int K[2];
  int s_i[8];
  int ev[2 * GP_MAX_BLK];
  unsigned bins[3][3][BIN_STRIDE];                // per task: members, mass (low, high word)
  double gM[16], gR[16];                          // a unit shared out over a cluster: the maxima and factors of the whole unit ...
  unsigned grng[3][2];                            // ... and the range of its scores' high words
  unsigned shared_out[GP_MAX_REQ / 32];           // a bit per boundary request: its units are shared out
  int n_shared, ticket;
  alignas(16) double F[SEL_F];                    // page factors; of a unit shared out, after that, the cluster's bins
};
static_assert(SEL_F * sizeof(double) >= (3 * 4 + 2 * 8) * BIN_STRIDE, "the cluster's bins fit");
struct SelSmem {
  SelMisc* m;
  unsigned* loc;                     // [cap * 16 / 32 + 2] block-local picks, one bit per candidate
  double* sS;                        // [SEL_CAP or fewer] a^S, then as many of a^L
  double* sL;
  int n_cap;                         // candidates they have room for
};
__host__ __device__ inline int sel_n_cap(long long cap) { return cap * GP_PAGE < SEL_CAP ? (int)(cap * GP_PAGE) : SEL_CAP; }
__host__ __device__ inline size_t sel_loc_bytes(long long cap) { return (((size_t)cap * GP_PAGE / 32 + 2) * 4 + 15) / 16 * 16; }
constexpr size_t DECIDE_SMEM = 8 * GP_MAX_REQ * 4;          // the decisions' scratch takes the place of bitmap and scores
__device__ __forceinline__ SelSmem sel_smem_at(uint8_t* smem, int cap) {      // smem: 16-byte aligned, gp_sel_smem bytes
  SelSmem S;
  S.m = reinterpret_cast<SelMisc*>(smem);
  uint8_t* at = smem + (sizeof(SelMisc) + 15) / 16 * 16;
  S.loc = reinterpret_cast<unsigned*>(at);
  S.n_cap = sel_n_cap(cap);
  S.sS = reinterpret_cast<double*>(at + sel_loc_bytes(cap));
  S.sL = S.sS + S.n_cap;
  return S;
}

__device__ __forceinline__ unsigned long long key_of(double v) { return (unsigned long long)__double_as_longlong(v); }

// Per-head softmax over the first `ntile` pages of the candidates and the group mean (Sec. 3.2): a^S and a^L of every
// candidate, in the order of the tokens (`ord`; the logits lie in the order of the slots).  The attention kernel left, per 16-token page t and column c (view, head), the page's maximum logit m_tc
// and s_tc = sum of exp(z - m_tc), and per token x = exp(z - m_tc).  With M_c the maximum over pages and
// f_tc = exp(m_tc - M_c):  softmax = x f_tc / Z_c,  Z_c = sum_t s_tc f_tc.  So this pass takes one exponential per page
// and column instead of one per token and column; the factors f_tc / (G Z_c) of SEL_F / 2G pages at a time sit in
// shared memory.  A thread takes whole tokens (a view's values of a token are contiguous).  All loads of the prologue
// (page partials and the first tokens) are issued together.  `views`: bit 0 a^S, bit 1 a^L (a job that needs one view
// reads only that one's logits).  Also leaves the range of the scores' high words.
struct UnitOrder {          // the unit's order indices: of slot s, rank[table[s / 16] * page_stride + s % 16]
  const int* table; const int* rank;
  size_t page_stride;
};
template <int GG>
__device__ __forceinline__ void unit_softmax(const SelSmem& S, const double* __restrict__ x, size_t view_stride,
                                             const double* __restrict__ zs, double* __restrict__ aS, double* __restrict__ aL, int ntile,
                                             int views, const UnitOrder& ord) {
  constexpr int NC = 2 * GG;                             // columns
  constexpr int U = GG >= 4 ? 2 : 4;                     // tokens per thread in flight
  constexpr int KEEP = 2;                                // page partials per thread held in registers
  constexpr int FT = SEL_F / NC;                         // pages whose factors are in shared memory at a time
  SelMisc& m = *S.m;
  const int tid = threadIdx.x;
  const int myc = tid % NC;                              // SEL_T is a multiple of NC
  const int t0 = tid / NC;
  constexpr int TSTEP = SEL_T / NC;
  double2 keep[KEEP];
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    const int t = t0 + k * TSTEP;
    keep[k] = make_double2(-INFINITY, 0.0);
    if (t < ntile) keep[k] = ld_early2(zs + ((size_t)t * NC + myc) * 2);
  }
  double xv[U][2][GG];
  int pg[U], at[U];                                      // page of a token (of the next pass of the loop), its place in the order
  auto load_pages = [&](int tok0) {
#pragma unroll
    for (int u = 0; u < U; ++u) { const int t = (tok0 + tid + u * SEL_T) / GP_PAGE; pg[u] = t < ntile ? __ldg(ord.table + t) : 0; }
  };
  auto load_order = [&](int tok0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int tok = tok0 + tid + u * SEL_T;
      if (tok < ntile * GP_PAGE) at[u] = __ldcg(ord.rank + (size_t)pg[u] * ord.page_stride + tok % GP_PAGE);
    }
  };
  load_pages(0);
  auto load = [&](int tok0, int n_tok) {                 // tokens tok0 + tid, tok0 + tid + SEL_T, ... of both views
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int tok = tok0 + tid + u * SEL_T;
      if (tok < n_tok) {
        if (views & 1) ld_early_row<GG>(x + (size_t)tok * GG, xv[u][0]);
        if (views & 2) ld_early_row<GG>(x + view_stride + (size_t)tok * GG, xv[u][1]);
      }
    }
  };
  const int n = ntile * GP_PAGE;
  load(0, n);
  double mx = fmax(keep[0].x, keep[1].x);
#pragma unroll 8
  for (int t = t0 + KEEP * TSTEP; t < ntile; t += TSTEP) mx = fmax(mx, __ldcg(zs + ((size_t)t * NC + myc) * 2));
  load_order(0);
  load_pages(U * SEL_T);
  column_reduce<true>(mx, NC, m.red, m.sM);
  const double mc = m.sM[myc];
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    const int t = t0 + k * TSTEP;
    if (t < ntile) {
      const double f = exp(keep[k].x - mc);
      acc += keep[k].y * f;
      if (t < FT) m.F[t * NC + myc] = f;
    }
  }
#pragma unroll 1
  for (int tb = t0 + KEEP * TSTEP; tb < ntile; tb += 4 * TSTEP) {
    double2 ms[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = tb + k * TSTEP;
      ms[k] = t < ntile ? ld_early2(zs + ((size_t)t * NC + myc) * 2) : make_double2(-INFINITY, 0.0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = tb + k * TSTEP;
      if (t < ntile) {
        const double f = exp(ms[k].x - mc);
        acc += ms[k].y * f;
        if (t < FT) m.F[t * NC + myc] = f;
      }
    }
  }
  column_reduce<false>(acc, NC, m.red, m.sZ);
  const double rz = 1.0 / ((double)GG * m.sZ[myc]);        // group mean and normaliser in one factor
#pragma unroll 1
  for (int t = t0; t < min(ntile, FT); t += TSTEP) m.F[t * NC + myc] *= rz;       // (the thread that wrote the entry)
  __syncthreads();
  unsigned lo_w[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi_w[3] = {0u, 0u, 0u};
#pragma unroll 1
  for (int tb = 0; tb < ntile; tb += FT) {               // a set of pages whose factors are in shared memory
    const int k_begin = tb * GP_PAGE, k_end = min(n, k_begin + FT * GP_PAGE);
    if (tb) {
      load(k_begin, k_end);
      load_order(k_begin);
      load_pages(k_begin + U * SEL_T);
      __syncthreads();
#pragma unroll 1
      for (int t = tb + t0; t < min(ntile, tb + FT); t += TSTEP)
        m.F[(t - tb) * NC + myc] = exp(__ldcg(zs + ((size_t)t * NC + myc) * 2) - mc) * rz;
      __syncthreads();
    }
#pragma unroll 1
    for (int k0 = k_begin; k0 < k_end; k0 += U * SEL_T) {
      if (k0 != k_begin) { load(k0, k_end); load_order(k0); load_pages(k0 + U * SEL_T); }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tok = k0 + tid + u * SEL_T;
        if (tok < k_end) {
          const double* f = m.F + (tok / GP_PAGE - tb) * NC;
          double a[2] = {0.0, 0.0};
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if ((views >> q) & 1) {
              a[q] = xv[u][q][0] * f[q * GG];
#pragma unroll
              for (int g = 1; g < GG; ++g) a[q] += xv[u][q][g] * f[q * GG + g];
            }
          }
          // a job of one array; the larger score by its bits, as everywhere (one that is not a number is the largest)
          const int i = min(max(at[u], 0), n - 1);           // (within bounds whatever a wait that gave up left behind)
          if (aS == aL) aS[i] = views == 3 ? (key_of(a[0]) > key_of(a[1]) ? a[0] : a[1]) : a[views >> 1];
          else { aS[i] = a[0]; aL[i] = a[1]; }
          const unsigned w0 = (unsigned)__double2hiint(a[0]), w1 = (unsigned)__double2hiint(a[1]), w2 = max(w0, w1);
          lo_w[0] = min(lo_w[0], w0); lo_w[1] = min(lo_w[1], w1); lo_w[2] = min(lo_w[2], w2);
          hi_w[0] = max(hi_w[0], w0); hi_w[1] = max(hi_w[1], w1); hi_w[2] = max(hi_w[2], w2);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const unsigned a = __reduce_min_sync(0xffffffffu, lo_w[q]), b = __reduce_max_sync(0xffffffffu, hi_w[q]);
    if ((tid & 31) == 0) { atomicMin(&m.rng[q][0], a); atomicMax(&m.rng[q][1], b); }
  }
}

// Eq. 10, block-local quota: the kq best slots of every block of `blk` candidates (score desc, slot asc; the last block
// may be short) as bits of loc[].  Run by `nw` warps, warp w of them taking every nw-th 32 slots or block.
__device__ __forceinline__ void mark_local(const double* aS, const double* aL, int n, int blk, int kq, unsigned* loc, int w, int nw) {
  const int lane = threadIdx.x & 31;
  if (blk == GP_PAGE) {                                   // two blocks to a warp: every score against its block's others
#pragma unroll 1
    for (int b0 = w * 32; b0 < n; b0 += nw * 32) {
      const int i = b0 + lane;
      const unsigned long long key = i < n ? max(key_of(aS[i]), key_of(aL[i])) : 0ull;
      // by the high words; where two of a block share one (about one block in ten thousand), by the whole keys
      const unsigned hw = (unsigned)(key >> 32);
      int rank = 0;
      bool same = false;
#pragma unroll
      for (int o = 1; o < 16; ++o) {
        const unsigned t = __shfl_xor_sync(0xffffffffu, hw, o);
        rank += t > hw; same |= t == hw;
      }
      if (__any_sync(0xffffffffu, same && i < n)) {
        rank = 0;
#pragma unroll 1
        for (int o = 1; o < 16; ++o) {
          const unsigned long long t = __shfl_xor_sync(0xffffffffu, key, o);
          rank += t > key || (t == key && (lane ^ o) < lane);
        }
      }
      const unsigned bits = __ballot_sync(0xffffffffu, i < n && rank < kq);
      if (lane == 0) loc[b0 >> 5] = bits;
    }
    return;
  }
  // A warp to a block of 32 to 256: descends the bits of the kq-th largest score, counting with ballots; it may stop
  // where exactly kq scores lie at or above the candidate.
#pragma unroll 1
  for (int b0 = w * blk; b0 < n; b0 += nw * blk) {
    const int per = blk / 32, have = min(blk, n - b0);
    unsigned long long key[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = j * 32 + lane;
      key[j] = j < per && i < have ? max(key_of(aS[b0 + i]), key_of(aL[b0 + i])) + 1 : 0ull;        // 0: no candidate
    }
    auto count = [&](unsigned long long t) {
      int c = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) if (j < per) c += __popc(__ballot_sync(0xffffffffu, key[j] >= t));
      return c;
    };
    unsigned long long thr = 1ull;                        // every candidate
    bool exact = have <= kq;
    if (!exact) {
      thr = 0ull;
      unsigned top = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) top = max(top, (unsigned)(key[j] >> 32));
      top = __reduce_max_sync(0xffffffffu, top);
#pragma unroll 1
      for (int bit = top ? 63 - __clz((int)top) : 31; bit >= 0 && !exact; --bit) {
        const unsigned long long t = thr | (1ull << bit);
        const int c = count(t);
        if (c >= kq) { thr = t; exact = c == kq; }
      }
    }
    int spare = exact ? 0 : kq - count(thr + 1);           // scores equal to the threshold that still fit, lowest slots first
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < per) {
        const unsigned above = __ballot_sync(0xffffffffu, exact ? key[j] >= thr : key[j] > thr);
        const unsigned eq = exact ? 0u : __ballot_sync(0xffffffffu, key[j] == thr);
        const bool pick = (above >> lane & 1u) || ((eq >> lane & 1u) && __popc(eq & ((1u << lane) - 1u)) < spare);
        spare -= min(spare, __popc(eq));
        const unsigned bits = __ballot_sync(0xffffffffu, pick);
        if (lane == 0 && b0 + j * 32 < n) loc[(b0 >> 5) + j] = bits;
      }
    }
  }
}

// Selection of one boundary unit over its scores a^S, a^L (n candidates), all tasks side by side:
//   task 0, 1   warps 0-1, 2-3: K^S, K^L (Eq. 7): smallest k such that the k largest scores sum to at least p
//   task 2      warps 4-7: the `ne` lowest of max(a^S, a^L) outside the block-local quota (Eq. 10; score asc, slot desc)
// `tasks` is the set to run (bits); a single task gets all warps.  The descent goes level by level with block barriers, so
// the tasks stay in step.
// What bounds it: the latency of a level (members counted with shared-memory atomics, a scan by one warp); two or three
// levels for a thousand candidates.  Behind the attention kernel of 36 layers x 256 residents (4608 units) the selection
// takes 330 us, with a block per task and 4096-bin histograms it took 480; on 32 units of 20 000 candidates, groups of 8, 560 us
// against 1300 (scores in the pool's scratch: their loads are batched).
__device__ __forceinline__ void unit_select(const GpDev& p, const SelSmem& S, const double* aS, const double* aL, int n, int tasks,
                                         int ne, int kq, int* Kout, int* acc, int* evout) {
  SelMisc& m = *S.m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool alone = (tasks & (tasks - 1)) == 0;
  const int task = alone ? tasks >> 1 : warp < 2 ? 0 : (warp < 4 ? 1 : 2);
  const int T = alone ? SEL_T : task == 2 ? 128 : 64;                             // threads of the task, and this one's index
  const int gt = alone ? tid : task == 2 ? tid - 128 : tid & 63;
  const double* a = task == 1 ? aL : aS;
  const bool lead = gt < 32;                                                      // the task's first warp
  bool run = (tasks >> task) & 1;
  unsigned* bcnt = m.bins[task][0]; unsigned* blo = m.bins[task][1]; unsigned* bhi = m.bins[task][2];
  for (int i = tid; i < 3 * 3 * BIN_STRIDE; i += SEL_T) (&m.bins[0][0][0])[i] = 0;
  if (tid < 4) m.cnt[tid] = 0;
  __syncthreads();                                         // the scores are there
  if (tasks & 4) {
    if (kq > 0) mark_local(aS, aL, n, p.blk, kq, S.loc, warp, SEL_NW);
    else for (int i = tid; i < (n + 31) / 32; i += SEL_T) S.loc[i] = 0;
  }
  // (non-negative doubles order as their bit patterns do)
  auto key2 = [&](int i) { return max(key_of(aS[i]), key_of(aL[i])); };
  auto eligible = [&](int i) { return !((S.loc[i >> 5] >> (i & 31)) & 1u); };
  // keys agree above bit `shift + 8`
  const unsigned h0 = m.rng[task][0], h1 = m.rng[task][1];
  int shift = h0 == h1 ? 24 : max(0, 32 + (31 - __clz((int)(h0 ^ h1))) - 7);
  int width = 8;
  unsigned long long prefix = ((unsigned long long)h1 << 32) >> (shift + 8);
  unsigned before = 0;                                     // members before the crossing bin (above it; task 2: below it)
  unsigned long long mass = 0;
  unsigned in_bin = 0;
  int K = -1;
  bool ties = false, whole = false;
  __syncthreads();
  const bool mine = run;
  for (;;) {
    // four at a time: their loads, then their adds, in flight together
    const unsigned mask = (1u << width) - 1u;
    if (run && task != 2) {
#pragma unroll 1
      for (int i0 = gt; i0 < n; i0 += 4 * T) {
        unsigned long long f[4]; bool on[4]; int b[4]; unsigned old[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = i0 + e * T;
          const double v = a[i < n ? i : gt];
          const unsigned long long k = key_of(v) >> shift;
          on[e] = i < n && (k >> width) == prefix;
          b[e] = BIDX((int)((unsigned)k & mask));
          f[e] = to_fix(v);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          old[e] = 0u;
          if (on[e]) { atomicAdd(&bcnt[b[e]], 1u); old[e] = atomicAdd(&blo[b[e]], (unsigned)f[e]); }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {                      // the carry travels with the high word's add
          const unsigned up = (unsigned)(f[e] >> 32) + (old[e] + (unsigned)f[e] < old[e] ? 1u : 0u);
          if (on[e] && up) atomicAdd(&bhi[b[e]], up);
        }
      }
    } else if (run) {
#pragma unroll 1
      for (int i0 = gt; i0 < n; i0 += 4 * T) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = i0 + e * T, j = i < n ? i : gt;
          const unsigned long long k = key2(j) >> shift;
          if (i < n && (k >> width) == prefix && eligible(j)) atomicAdd(&bcnt[BIDX((int)((unsigned)k & mask))], 1u);
        }
      }
    }
    __syncthreads();
    if (run && lead) {                                     // lane owns bins [8 lane, 8 lane + 8)
      unsigned c8[8]; unsigned long long m8[8];
      unsigned c = 0; unsigned long long s = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int b = lane * 9 + j;                        // BIDX(8 lane + j)
        c8[j] = bcnt[b];
        m8[j] = task != 2 ? ((unsigned long long)bhi[b] << 32) + blo[b] : 0ull;
        c += c8[j]; s += m8[j];
      }
      unsigned ic = c; unsigned long long is = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (task != 2) {                                   // largest scores first
          const unsigned tc = __shfl_down_sync(0xffffffffu, ic, o);
          const unsigned long long ts = __shfl_down_sync(0xffffffffu, is, o);
          if (lane + o < 32) { ic += tc; is += ts; }
        } else {                                           // lowest scores first
          const unsigned tc = __shfl_up_sync(0xffffffffu, ic, o);
          if (lane >= o) ic += tc;
        }
      }
      unsigned rc = before + ic - c; unsigned long long rs = mass + is - s;
      bool hit = false;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int j = task != 2 ? 7 - jj : jj;
        const bool here = task != 2 ? rs < p.p_fix && rs + m8[j] >= p.p_fix : rc < (unsigned)ne && rc + c8[j] >= (unsigned)ne;
        if (here) { m.res[task][0] = lane * 8 + j; m.res[task][1] = rc; m.res[task][2] = (long long)rs; m.res[task][3] = c8[j]; hit = true; }
        rc += c8[j]; rs += m8[j];
      }
      if (!__any_sync(0xffffffffu, hit) && lane == 0) m.res[task][0] = -1;
    }
    __syncthreads();
    if (run) {
      const int bin = (int)m.res[task][0];
      if (bin < 0) {
        // rounding kept the total below p: everything.  (Task 2 has more than `ne` eligible candidates by the quota's size.)
        K = n; run = false;
        if (task == 2) {                                     // (scores that are not numbers: some list within bounds, and the error bit)
#pragma unroll 1
          for (int t = gt; t < ne; t += T) m.ev[t] = t;
          if (gt == 0) atomicOr(p.err, GP_E_BOUNDS);
        }
      } else {
        before = (unsigned)m.res[task][1]; mass = (unsigned long long)m.res[task][2]; in_bin = (unsigned)m.res[task][3];
        prefix = (prefix << width) | (unsigned long long)bin;
        if (task != 2 && in_bin == 1) { K = (int)before + 1; run = false; }
        else if (task == 2 && before + in_bin == (unsigned)ne) { whole = true; run = false; }       // the bin goes as a whole
        else if (in_bin <= 32) run = false;
        else if (shift == 0) { ties = true; run = false; }              // copies of one value
        else { width = min(8, shift); shift -= width; }
#pragma unroll 1
        for (int i = gt; i < BIN_STRIDE; i += T) { bcnt[i] = 0; blo[i] = 0; bhi[i] = 0; }
      }
    }
    if (!__syncthreads_or(run)) break;
  }
  // ---- the members of the crossing bin, one by one (keys >> shift == prefix) -----------------------------------------
  const bool listed = mine && K < 0 && !ties && !whole;
  if (mine && K < 0) {
    if (task != 2) {
      if (listed) {
#pragma unroll 4
        for (int i = gt; i < n; i += T) {
          const double v = a[i];
          if ((key_of(v) >> shift) == prefix) {
            const int at = atomicAdd(&m.cnt[1 + task], 1);
            m.list[task][at] = key_of(v); m.list_fix[task][at] = to_fix(v);
          }
        }
      }
    } else {
#pragma unroll 4
      for (int i = gt; i < n; i += T) {
        const unsigned long long full = key2(i), k = full >> shift;
        if (k <= prefix && eligible(i)) {
          if (k < prefix || whole) { const int at = atomicAdd(&m.cnt[0], 1); if (at < ne) m.ev[at] = i; }
          else if (listed) { const int at = atomicAdd(&m.cnt[3], 1); m.list[2][at] = full; m.list_slot[at] = i; }
        }
      }
    }
  }
  __syncthreads();
  if (mine && lead) {
    if (task != 2) {
      if (listed) {
        // every member's place in the descending order and the mass up to and including it
        const unsigned long long v = m.list[task][lane];
        int rank = 0;
        unsigned long long inc = 0;
#pragma unroll 4
        for (int j = 0; j < (int)in_bin; ++j) {
          const unsigned long long t = m.list[task][j];
          const bool first = t > v || (t == v && j <= lane);
          rank += first;
          inc += first ? m.list_fix[task][j] : 0ull;
        }
        K = (int)before + (int)__reduce_min_sync(0xffffffffu, lane < (int)in_bin && mass + inc >= p.p_fix ? (unsigned)rank : in_bin);
      } else if (ties) {
        const unsigned long long f = to_fix(__longlong_as_double((long long)prefix));
        unsigned long long j = f ? (p.p_fix - mass + f - 1) / f : 1ull;
        if (j < 1) j = 1;
        if (j > in_bin) j = in_bin;
        K = (int)before + (int)j;
      }
      if (lane == 0) {
        Kout[task] = K;
        atomicAdd(acc + task, K);                          // Eq. 8 needs only the sums over layers and heads
      }
    } else if (listed) {                                   // the lowest scores of the bin, later slots first among equals
      const unsigned long long v = m.list[2][lane];
      const int slot = m.list_slot[lane];
      int rank = 0;
#pragma unroll 4
      for (int j = 0; j < (int)in_bin; ++j) {
        const unsigned long long t = m.list[2][j];
        rank += t < v || (t == v && m.list_slot[j] > slot);
      }
      if (lane < (int)in_bin && rank < ne - (int)before) m.ev[before + rank] = slot;
    } else if (ties && lane == 0) {                        // rare: older (lower) slots win ties
      int at = (int)before;
#pragma unroll 1
      for (int i = n - 1; i >= 0 && at < ne; --i)
        if (key2(i) == prefix && eligible(i)) m.ev[at++] = i;
    }
  }
  if (!(tasks & 4)) return;
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < ne; t += SEL_T) {                    // the evicted slots in ascending order, by rank
    const int slot = m.ev[t];
    int rank = 0;
#pragma unroll 16
    for (int j = 0; j < ne; ++j) rank += (m.ev[j] < slot);           // (ne is a multiple of 16)
    evout[rank] = slot;
  }
}

// ------------------------------------------------------------------------------------------------------
// working sets + speculative eviction lists of a unit, one CTA; the last CTA decides
// ------------------------------------------------------------------------------------------------------
// Unit u = (boundary request bidx, layer and KV head lh): K^S and K^L go to Kx and, summed, to bnd_acc (Eq. 8), the `b`
// slots a compression would evict to evict, the 2b of a Shrink to evict2.  `want`: the tasks of unit_select, 7 for the whole
// unit; with few units a thread block takes one of its three tasks.
template <int GG>      // query heads per KV head
__device__ __forceinline__ void sel_unit(const GpDev& p, const SelSmem& S, int bidx, int lh, const int4 inf, const int4 inf2, int want) {
  SelMisc& m = *S.m;
  const int tid = threadIdx.x;
  constexpr int G = GG;
  const int LH = p.L * p.Hkv;
  const int r = inf.y, Pr = inf.z;
  const long long off = (long long)(unsigned)inf2.x | ((long long)inf2.y << 32);
  const size_t u = (size_t)bidx * LH + lh;
  int* Kout = p.Kx + ((size_t)r * LH + lh) * 2;
  int* acc = p.bnd_acc + 4 * bidx;
  // two supports (they coincide when the page is 16 tokens): the working sets of Eq. 7 leave out the newest page
  // of the method, the eviction candidates of Eq. 10 only the protected window, the newest 16-token tile
  const int nt_d = Pr - p.sub, nt_e = Pr - 1;
  if (nt_d == 0) {                           // one page of the method: nothing to estimate from, nothing to evict
    if (tid < 2 && ((want >> tid) & 1)) Kout[tid] = 0;
    return;
  }
  const size_t view_stride = (size_t)p.z_stride * G;
  const double* z = p.zbuf + (size_t)lh * 2 * view_stride + (size_t)off * G;       // [2 views][n][G] exp(logit - page max)
  const double* zs = p.zstat + ((size_t)lh * (p.max_boundary_tokens / GP_PAGE) + off / GP_PAGE) * 2 * G * 2;
  // the scores: in shared memory, or, for candidate sets too large for it, in the pool's scratch (three regions: a whole
  // unit uses two, one per view, a single job the one of its number).  A job that lists evictions keeps only
  // max(a^S, a^L), in the place of both.
  const bool single = want != 7;
  const bool small = nt_e * GP_PAGE <= (single ? 2 * S.n_cap : S.n_cap);
  double* aS = small ? S.sS : p.scores + ((size_t)(single ? want >> 1 : 0) * LH + lh) * p.max_boundary_tokens + off;
  double* aL = single ? aS : small ? S.sL : aS + (size_t)LH * p.max_boundary_tokens;
  const int views = want == 1 ? 1 : want == 2 ? 2 : 3;
  const UnitOrder ord = {p.page_table + (size_t)r * p.cap, p.rank + gp_tok_off(p, lh / p.Hkv, 0, lh % p.Hkv), (size_t)p.Hkv * GP_PAGE};
  const bool one_support = p.sub == 1;
  const bool entropy = p.metric == GP_METRIC_ENTROPY;
#pragma unroll 1
  for (int pass = 0; pass < (one_support ? 1 : 2); ++pass) {
    const int ntile = pass == 0 ? nt_d : nt_e, n = ntile * GP_PAGE;
    int tasks = want & (one_support ? 7 : pass == 0 ? 3 : 4);
    if (!tasks) continue;
    __syncthreads();                                       // the unit or pass before is done with the shared arrays
    if (tid < 3) { m.rng[tid][0] = 0xffffffffu; m.rng[tid][1] = 0u; }
    unit_softmax<GG>(S, z, view_stride, zs, aS, aL, ntile, views, ord);      // (its barriers order rng before the first use)
    if (entropy && (tasks & 3)) {
      __syncthreads();                                     // the scores are there
      // the ablation's other metric: H = -sum a ln a of the view, summed in a fixed order (per thread over its
      // strided candidates, then a fixed tree), so that the same input gives the same bits on every run
      double* Hout = p.Hx + ((size_t)r * LH + lh) * 2;
      for (int view = 0; view < 2; ++view) {
        if (!((tasks >> view) & 1)) continue;
        const double* a = view ? aL : aS;
        double hsum = 0.0;
#pragma unroll 1
        for (int i = tid; i < n; i += SEL_T) { const double v = a[i]; if (v > 0.0) hsum -= v * log(v); }
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) hsum += __shfl_xor_sync(0xffffffffu, hsum, o2);
        if ((tid & 31) == 0) m.red[tid >> 5] = hsum;
        __syncthreads();
        if (tid == 0) {
          double tot = 0.0;
#pragma unroll 1
          for (int w = 0; w < SEL_NW; ++w) tot += m.red[w];
          Kout[view] = 0;
          Hout[view] = tot;
        }
        __syncthreads();
      }
      tasks &= 4;
    }
    // the lists: b slots of a compression, then, where this boundary can be a Shrink, its 2b
    const bool shrink = p.policy == GP_POLICY_SHRINK && (tasks & 4) && Pr - p.sub >= p.min_pages_after_shrink;
    const int nblk = (n + p.blk - 1) / p.blk;
#pragma unroll 1
    for (int list = 0; list < (shrink ? 2 : 1); ++list) {
      const int ne = (list + 1) * p.blk;
      if (list || tasks)
        unit_select(p, S, aS, aL, n, list ? 4 : tasks, ne, min(p.k_loc, (n - ne) / nblk), Kout, acc,
                    list ? p.evict2 + u * ne : p.evict + u * ne);
    }
  }
}

// ------------------------------------------------------------------------------------------------------
// a unit of many candidates, shared out over the thread blocks of a cluster
// ------------------------------------------------------------------------------------------------------
// One thread block walks 20 000 candidates of a group of eight in 380 us (logits of two views and eight heads, 128 bytes each, and then every
// level of the descent over scores that do not fit its shared memory), while most of the chip has no unit at all.  Here the CLUSTER blocks of
// a cluster share one: each takes a part of the pages for the softmax (its normalisers are merged over the cluster), the scores go to the
// pool's scratch in the order of the tokens, and each takes a part of that order into its shared memory for the descents, whose bins are added
// up over the cluster at every level.  Counts and fixed-point masses are integers, so the result is that of one block over the same scores.
// What bounds it: the logits' bytes, then a chain of a dozen cluster barriers.  Two requests of 20 000, us a step: one layer, groups of eight
// 101.6 / 79.7, of four 76.3 / 65.0; four layers 184.9 / 161.2 and 147.1 / 138.3.
constexpr int CLUSTER = 8;
constexpr int SPLIT_ROUNDS = 2;             // units a cluster takes one after the other at most
constexpr int SPLIT_FROM = GP_SHARED_FROM;  // candidates above which a unit is shared out: see split_unit
static_assert(SPLIT_FROM == 2 * SEL_CAP, "up to there the scores of a job fit one thread block's shared memory");
__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
// The wait of the cluster's barrier has no limit, unlike those for a word that another block writes.  It ends because the eight blocks run at the same
// time and reach the same barriers: what any of them branches on in between are the plan's words, the ticket, and sums that each
// takes over all eight blocks' shared memory behind a barrier, the same in every block whatever the scores are.  So a wait with a limit (unit_there) that
// gives up in one block alone changes what is in the scores and not where the blocks go.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the same place in the shared memory of another block of the cluster
template <typename T>
__device__ __forceinline__ T* of_block(T* ptr, unsigned rank) {
  T* q;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(ptr), "r"(rank));
  return q;
}

// Scores of the pages [t_lo, t_hi) into aS, aL (global, in the order of the tokens), normalised over all of the unit's.  Ends with a
// barrier of the cluster, behind which all scores and the blocks' ranges of high words are there.
template <int GG>
__device__ __forceinline__ void split_softmax(const SelSmem& S, const double* __restrict__ x, size_t view_stride, const double* __restrict__ zs,
                                              double* aS, double* aL, int t_lo, int t_hi, int n, const UnitOrder& ord) {
  constexpr int NC = 2 * GG, U = GG >= 4 ? 2 : 4, FT = SEL_F / NC, TSTEP = SEL_T / NC;
  SelMisc& m = *S.m;
  const int tid = threadIdx.x, myc = tid % NC, t0 = tid / NC;
  double mx = -INFINITY;
#pragma unroll 4
  for (int t = t_lo + t0; t < t_hi; t += TSTEP) mx = fmax(mx, __ldcg(zs + ((size_t)t * NC + myc) * 2));
  column_reduce<true>(mx, NC, m.red, m.sM);
  double acc = 0.0;
#pragma unroll 2
  for (int t = t_lo + t0; t < t_hi; t += TSTEP) {
    const double2 ms = __ldcg(reinterpret_cast<const double2*>(zs + ((size_t)t * NC + myc) * 2));
    acc += ms.y * exp(ms.x - m.sM[myc]);
  }
  column_reduce<false>(acc, NC, m.red, m.sZ);
  // the places of this block's candidates in the order, ahead of their scores (in the place the scores take later)
  int* const at = reinterpret_cast<int*>(S.sS);
#pragma unroll 8
  for (int i = tid; i < (t_hi - t_lo) * GP_PAGE; i += SEL_T)
    at[i] = min(max(__ldcg(ord.rank + (size_t)__ldg(ord.table + t_lo + i / GP_PAGE) * ord.page_stride + i % GP_PAGE), 0), n - 1);  // (in bounds whatever a wait that gave up left behind)
  cluster_sync();
  if (tid < NC) {
    double M = -INFINITY, Z = 0.0;
#pragma unroll
    for (int r = 0; r < CLUSTER; ++r) M = fmax(M, of_block(m.sM, r)[tid]);
#pragma unroll 1
    for (int r = 0; r < CLUSTER; ++r) {
      const double zr = of_block(m.sZ, r)[tid], mr = of_block(m.sM, r)[tid];
      Z += zr == 0.0 ? 0.0 : zr * exp(mr - M);            // (a block without pages: 0; what is no number stays none)
    }
    m.gM[tid] = M; m.gR[tid] = 1.0 / ((double)GG * Z);
  }
  unsigned lo_w[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi_w[3] = {0u, 0u, 0u};
#pragma unroll 1
  for (int tb = t_lo; tb < t_hi; tb += FT) {
    const int te = min(t_hi, tb + FT), k_end = te * GP_PAGE;
    __syncthreads();
#pragma unroll 2
    for (int t = tb + t0; t < te; t += TSTEP) m.F[(t - tb) * NC + myc] = exp(__ldcg(zs + ((size_t)t * NC + myc) * 2) - m.gM[myc]) * m.gR[myc];
    __syncthreads();
#pragma unroll 1
    for (int k0 = tb * GP_PAGE; k0 < k_end; k0 += U * SEL_T) {
      double xv[U][2][GG];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tok = k0 + tid + u * SEL_T;
        if (tok < k_end) {
          ld_early_row<GG>(x + (size_t)tok * GG, xv[u][0]);
          ld_early_row<GG>(x + view_stride + (size_t)tok * GG, xv[u][1]);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tok = k0 + tid + u * SEL_T;
        if (tok < k_end) {
          const double* f = m.F + (tok / GP_PAGE - tb) * NC;
          double a[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            a[q] = xv[u][q][0] * f[q * GG];
#pragma unroll
            for (int g = 1; g < GG; ++g) a[q] += xv[u][q][g] * f[q * GG + g];
          }
          const int i = at[tok - t_lo * GP_PAGE];
          __stcg(aS + i, a[0]); __stcg(aL + i, a[1]);
          const unsigned w0 = (unsigned)__double2hiint(a[0]), w1 = (unsigned)__double2hiint(a[1]), w2 = max(w0, w1);
          lo_w[0] = min(lo_w[0], w0); lo_w[1] = min(lo_w[1], w1); lo_w[2] = min(lo_w[2], w2);
          hi_w[0] = max(hi_w[0], w0); hi_w[1] = max(hi_w[1], w1); hi_w[2] = max(hi_w[2], w2);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const unsigned a = __reduce_min_sync(0xffffffffu, lo_w[q]), b = __reduce_max_sync(0xffffffffu, hi_w[q]);
    if ((tid & 31) == 0) { atomicMin(&m.rng[q][0], a); atomicMax(&m.rng[q][1], b); }
  }
  cluster_sync();
}

// The tasks of unit_select over this block's part of the order, candidates [i_lo, i_lo + nl) of the unit's n, in S.sS and S.sL.  All blocks
// of the cluster take the same decisions from the same sums; lists are gathered in the first one, which writes the results.
__device__ __forceinline__ void split_select(const GpDev& p, const SelSmem& S, const double* gS, const double* gL, int i_lo, int nl, int per, int n,
                                             int tasks, int ne, int kq, int* Kout, int* acc, int* evout) {
  SelMisc& m = *S.m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned me = cluster_rank();
  const int task = warp < 2 ? 0 : (warp < 4 ? 1 : 2), T = task == 2 ? 128 : 64, gt = task == 2 ? tid - 128 : tid & 63;
  const double* a = task == 1 ? S.sL : S.sS;
  const bool lead = gt < 32, mine = (tasks >> task) & 1;
  bool run = mine;
  unsigned* bcnt = m.bins[task][0]; unsigned* blo = m.bins[task][1]; unsigned* bhi = m.bins[task][2];
  unsigned* const ccnt = reinterpret_cast<unsigned*>(m.F);                                     // [3][BIN_STRIDE] members, the cluster's
  unsigned long long* const cmass = reinterpret_cast<unsigned long long*>(ccnt + 3 * BIN_STRIDE + (3 * BIN_STRIDE & 1));      // [2][BIN_STRIDE]
#pragma unroll 1
  for (int i = tid; i < 3 * 3 * BIN_STRIDE; i += SEL_T) (&m.bins[0][0][0])[i] = 0;
  if (tid < 4) m.cnt[tid] = 0;
  if (tid < 3) {
    unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll 1
    for (int r = 0; r < CLUSTER; ++r) { lo = min(lo, of_block(&m.rng[tid][0], r)[0]); hi = max(hi, of_block(&m.rng[tid][0], r)[1]); }
    m.grng[tid][0] = lo; m.grng[tid][1] = hi;
  }
  __syncthreads();
  if (tasks & 4) {
    if (kq > 0) mark_local(S.sS, S.sL, nl, p.blk, kq, S.loc, warp, SEL_NW);
    else for (int i = tid; i < (nl + 31) / 32; i += SEL_T) S.loc[i] = 0;
  }
  auto key2 = [&](int i) { return max(key_of(S.sS[i]), key_of(S.sL[i])); };
  auto eligible = [&](int i) { return !((S.loc[i >> 5] >> (i & 31)) & 1u); };
  const unsigned h0 = m.grng[task][0], h1 = m.grng[task][1];
  int shift = h0 == h1 ? 24 : max(0, 32 + (31 - __clz((int)(h0 ^ h1))) - 7);
  int width = 8;
  unsigned long long prefix = ((unsigned long long)h1 << 32) >> (shift + 8);
  unsigned before = 0, in_bin = 0;
  unsigned long long mass = 0;
  int K = -1;
  bool ties = false, whole = false;
  __syncthreads();
  for (;;) {
    const unsigned mask = (1u << width) - 1u;
    if (run) {
#pragma unroll 1
      for (int i0 = gt; i0 < nl; i0 += 4 * T) {            // four at a time: their loads, then their adds, in flight together
        unsigned long long f[4]; bool on[4]; int b[4]; unsigned old[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = i0 + e * T, j = i < nl ? i : gt;
          const double v = a[j];
          const unsigned long long k = (task != 2 ? key_of(v) : key2(j)) >> shift;
          on[e] = i < nl && (k >> width) == prefix && (task != 2 || eligible(j));
          b[e] = BIDX((int)((unsigned)k & mask));
          f[e] = to_fix(v);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          old[e] = 0u;
          if (on[e]) { atomicAdd(&bcnt[b[e]], 1u); if (task != 2) old[e] = atomicAdd(&blo[b[e]], (unsigned)f[e]); }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {                      // the carry travels with the high word's add
          const unsigned up = (unsigned)(f[e] >> 32) + (old[e] + (unsigned)f[e] < old[e] ? 1u : 0u);
          if (on[e] && task != 2 && up) atomicAdd(&bhi[b[e]], up);
        }
      }
    }
    cluster_sync();
    {                                                      // the cluster's bins, a bin of each task per thread
      const int b = BIDX(tid);
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        unsigned c = 0; unsigned long long s = 0;
#pragma unroll
        for (int r = 0; r < CLUSTER; ++r) {
          const unsigned* q = of_block(&m.bins[t][0][b], r);
          c += q[0];
          if (t < 2) s += ((unsigned long long)q[2 * BIN_STRIDE] << 32) + q[BIN_STRIDE];
        }
        ccnt[t * BIN_STRIDE + b] = c;
        if (t < 2) cmass[t * BIN_STRIDE + b] = s;
      }
    }
    cluster_sync();                                        // (every block has read every block's: they may be cleared)
    if (run && lead) {                                     // lane owns bins [8 lane, 8 lane + 8)
      unsigned c8[8]; unsigned long long m8[8];
      unsigned c = 0; unsigned long long s = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int b = lane * 9 + j;                        // BIDX(8 lane + j)
        c8[j] = ccnt[task * BIN_STRIDE + b];
        m8[j] = task != 2 ? cmass[task * BIN_STRIDE + b] : 0ull;
        c += c8[j]; s += m8[j];
      }
      unsigned ic = c; unsigned long long is = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned td = __shfl_down_sync(0xffffffffu, ic, o), tu = __shfl_up_sync(0xffffffffu, ic, o);
        const unsigned long long ts = __shfl_down_sync(0xffffffffu, is, o);
        if (task != 2) { if (lane + o < 32) { ic += td; is += ts; } }         // largest scores first
        else if (lane >= o) ic += tu;                                          // lowest scores first
      }
      unsigned rc = before + ic - c; unsigned long long rs = mass + is - s;
      int bin = -1;
      unsigned bin_rc = 0, bin_c = 0; unsigned long long bin_rs = 0;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int j = task != 2 ? 7 - jj : jj;
        const bool here = task != 2 ? rs < p.p_fix && rs + m8[j] >= p.p_fix : rc < (unsigned)ne && rc + c8[j] >= (unsigned)ne;
        if (here) { bin = lane * 8 + j; bin_rc = rc; bin_rs = rs; bin_c = c8[j]; }
        rc += c8[j]; rs += m8[j];
      }
      // (sums of scores that a wait that gave up left behind can wrap, and more than one lane find a crossing: one of them, the same in every block)
      const unsigned found = __ballot_sync(0xffffffffu, bin >= 0);
      if (lane == (found ? __ffs((int)found) - 1 : 0)) {
        m.res[task][0] = bin; m.res[task][1] = bin_rc; m.res[task][2] = (long long)bin_rs; m.res[task][3] = bin_c;
      }
    }
    __syncthreads();
    if (run) {
      const int bin = (int)m.res[task][0];
      if (bin < 0) {
        K = n; run = false;                                // rounding kept the total below p: everything
        if (task == 2 && me == 0) {                        // (scores that are not numbers: some list within bounds, and the error bit)
          for (int t = gt; t < ne; t += T) m.ev[t] = t;
          if (gt == 0) atomicOr(p.err, GP_E_BOUNDS);
        }
      } else {
        before = (unsigned)m.res[task][1]; mass = (unsigned long long)m.res[task][2]; in_bin = (unsigned)m.res[task][3];
        prefix = (prefix << width) | (unsigned long long)bin;
        if (task != 2 && in_bin == 1) { K = (int)before + 1; run = false; }
        else if (task == 2 && before + in_bin == (unsigned)ne) { whole = true; run = false; }       // the bin goes as a whole
        else if (in_bin <= 32) run = false;
        else if (shift == 0) { ties = true; run = false; }              // copies of one value
        else { width = min(8, shift); shift -= width; }
        for (int i = gt; i < BIN_STRIDE; i += T) { bcnt[i] = 0; blo[i] = 0; bhi[i] = 0; }
      }
    }
    if (!__syncthreads_or(run)) break;                     // (the same in every block of the cluster)
  }
  // ---- the members of the crossing bin and the evicted candidates, gathered in the first block ------------------------
  SelMisc* const m0 = of_block(S.m, 0);
  const bool listed = mine && K < 0 && !ties && !whole;
  if (mine && K < 0) {
#pragma unroll 4
    for (int i = gt; i < nl; i += T) {
      if (task != 2) {
        const double v = a[i];
        if (listed && (key_of(v) >> shift) == prefix) {
          const int at = atomicAdd(&m0->cnt[1 + task], 1);
          if (at < 32) { m0->list[task][at] = key_of(v); m0->list_fix[task][at] = to_fix(v); }
        }
      } else {
        const unsigned long long full = key2(i), k = full >> shift;
        if (k <= prefix && eligible(i)) {
          if (k < prefix || whole) { const int at = atomicAdd(&m0->cnt[0], 1); if (at < ne) m0->ev[at] = i_lo + i; }
          else if (listed) { const int at = atomicAdd(&m0->cnt[3], 1); if (at < 32) { m0->list[2][at] = full; m0->list_slot[at] = i_lo + i; } }
        }
      }
    }
  }
  const bool evict_ties = __syncthreads_or(task == 2 && ties);
  cluster_sync();
  if (me == 0) {
    if (mine && lead) {
      if (task != 2) {
        if (listed) {
          const unsigned long long v = m.list[task][lane];
          int rank = 0;
          unsigned long long inc = 0;
#pragma unroll 1
          for (int j = 0; j < (int)in_bin; ++j) {
            const unsigned long long t = m.list[task][j];
            const bool first = t > v || (t == v && j <= lane);
            rank += first;
            inc += first ? m.list_fix[task][j] : 0ull;
          }
          K = (int)before + (int)__reduce_min_sync(0xffffffffu, lane < (int)in_bin && mass + inc >= p.p_fix ? (unsigned)rank : in_bin);
        } else if (ties) {
          const unsigned long long f = to_fix(__longlong_as_double((long long)prefix));
          unsigned long long j = f ? (p.p_fix - mass + f - 1) / f : 1ull;
          if (j < 1) j = 1;
          if (j > in_bin) j = in_bin;
          K = (int)before + (int)j;
        }
        if (lane == 0) { Kout[task] = K; atomicAdd(acc + task, K); }
      } else if (listed) {                                 // the lowest scores of the bin, later slots first among equals
        const unsigned long long v = m.list[2][lane];
        const int slot = m.list_slot[lane];
        int rank = 0;
#pragma unroll 1
        for (int j = 0; j < (int)in_bin; ++j) {
          const unsigned long long t = m.list[2][j];
          rank += t < v || (t == v && m.list_slot[j] > slot);
        }
        if (lane < (int)in_bin && rank < ne - (int)before) m.ev[before + rank] = slot;
      } else if (ties && lane == 0) {                      // rare: older (lower) slots win ties
        int at = (int)before;
        for (int i = n - 1; i >= 0 && at < ne; --i) {
          const unsigned r = (unsigned)(i / per);
          const int j = i - (int)r * per;
          if (max(key_of(__ldcg(gS + i)), key_of(__ldcg(gL + i))) == prefix && !((of_block(S.loc, r)[j >> 5] >> (j & 31)) & 1u)) m.ev[at++] = i;
        }
      }
    }
    if (tasks & 4) {
      __syncthreads();
#pragma unroll 1
      for (int t = tid; t < ne; t += SEL_T) {              // the evicted places in ascending order, by rank
        const int slot = m.ev[t];
        int rank = 0;
#pragma unroll 8
        for (int j = 0; j < ne; ++j) rank += (m.ev[j] < slot);
        evout[rank] = slot;
      }
    }
  }
  if (evict_ties) cluster_sync();                          // (the first block has read the others' bits)
}

// candidates a block of the cluster holds for the descents: whole blocks of Eq. 10, whole words of the bitmap
__device__ __forceinline__ int split_part(const GpDev& p, int n) {
  const int align = p.blk > 32 ? p.blk : 32;
  return ((n + CLUSTER - 1) / CLUSTER + align - 1) / align * align;
}
// Whether the units of a boundary request with `Pr` pages are shared out, in a step with `units` of all its boundary requests, on a grid of `clusters`.  The line: up to 10 240
// candidates the scores of a job fit one block's shared memory, and three blocks by themselves take no longer than the cluster's chain of
// barriers (two requests of 7000, one layer, groups of four / eight, us a step, by themselves 36.6 / 49.9, shared 36.4 / 45.5; of 4500 33.1 / 43.2 and
// 34.3 / 42.6; four layers of 7000 64.3 / 67.5), of 12 000 57.5 / 52.1 and 79.2 / 66.4; and a cluster takes its units one after the other, so that with
// three for each (12 layers of 12 000: 220 / 227, of 20 000 344 / 344) nothing is left of it.  Two units one after the other have to be of more than 20 480.
// The upper end: a block's part of the scores has to fit its shared memory, an eighth of 40 960 candidates (us of a step with
// a boundary at 40 960 / 40 976 / 60 000, one layer of 8 KV heads, groups of four 196 / 374 / 532, of eight 286 / 601 / 871).  A unit above that, and every unit of the
// entropy metric (a sum of logarithms in a fixed order), of Shrink (two eviction lists) and of the kernels launched one after the other, is one block's, or
// three blocks'.
__device__ __forceinline__ bool split_unit(const GpDev& p, const SelSmem& S, int Pr, long long units, int clusters) {
  const long long rounds = (units + clusters - 1) / clusters;
  const int n = (Pr - 1) * GP_PAGE;
  return rounds <= SPLIT_ROUNDS && n > SPLIT_FROM * rounds && split_part(p, n) <= S.n_cap && ((n / GP_PAGE + CLUSTER - 1) / CLUSTER + 1) * GP_PAGE <= 2 * S.n_cap &&
         p.metric != GP_METRIC_ENTROPY && p.policy != GP_POLICY_SHRINK;
}

// the k-th of the n boundary requests whose bit is `set` (or not)
__device__ __forceinline__ int nth_request(const unsigned* bits, int n, int k, bool set) {
#pragma unroll 1
  for (int w = 0; w * 32 < n; ++w) {
    unsigned v = set ? bits[w] : ~bits[w];
    if (n - w * 32 < 32) v &= (1u << (n - w * 32)) - 1u;
    const int c = __popc(v);
    if (k < c) {
#pragma unroll 1
      for (; k > 0; --k) v &= v - 1u;
      return w * 32 + __ffs((int)v) - 1;
    }
    k -= c;
  }
  return 0;                                                // (there are as many)
}

template <int GG>
__device__ __forceinline__ void sel_split(const GpDev& p, const SelSmem& S, int bidx, int lh, const int4 inf, const int4 inf2) {
  SelMisc& m = *S.m;
  const int LH = p.L * p.Hkv, r = inf.y, Pr = inf.z, me = (int)cluster_rank();
  const long long off = (long long)(unsigned)inf2.x | ((long long)inf2.y << 32);
  int* Kout = p.Kx + ((size_t)r * LH + lh) * 2;
  const size_t view_stride = (size_t)p.z_stride * GG;
  const double* z = p.zbuf + (size_t)lh * 2 * view_stride + (size_t)off * GG;
  const double* zs = p.zstat + ((size_t)lh * (p.max_boundary_tokens / GP_PAGE) + off / GP_PAGE) * 2 * GG * 2;
  double* aS = p.scores + (size_t)lh * p.max_boundary_tokens + off;
  double* aL = aS + (size_t)LH * p.max_boundary_tokens;
  const UnitOrder ord = {p.page_table + (size_t)r * p.cap, p.rank + gp_tok_off(p, lh / p.Hkv, 0, lh % p.Hkv), (size_t)p.Hkv * GP_PAGE};
  const bool one_support = p.sub == 1;
#pragma unroll 1
  for (int pass = 0; pass < (one_support ? 1 : 2); ++pass) {          // the two supports: see sel_unit
    const int ntile = pass == 0 ? Pr - p.sub : Pr - 1, n = ntile * GP_PAGE;
    const int tasks = one_support ? 7 : pass == 0 ? 3 : 4;
    __syncthreads();
    if (threadIdx.x < 3) { m.rng[threadIdx.x][0] = 0xffffffffu; m.rng[threadIdx.x][1] = 0u; }
    const int tpb = (ntile + CLUSTER - 1) / CLUSTER, t_lo = min(ntile, me * tpb), t_hi = min(ntile, t_lo + tpb);
    split_softmax<GG>(S, z, view_stride, zs, aS, aL, t_lo, t_hi, n, ord);
    const int per = split_part(p, n), i_lo = min(n, me * per), nl = min(n, i_lo + per) - i_lo;
#pragma unroll 4
    for (int i = threadIdx.x; i < nl; i += SEL_T) { S.sS[i] = __ldcg(aS + i_lo + i); S.sL[i] = __ldcg(aL + i_lo + i); }
    const int nblk = (n + p.blk - 1) / p.blk;
    split_select(p, S, aS, aL, i_lo, nl, per, n, tasks, p.blk, min(p.k_loc, (n - p.blk) / nblk), Kout, p.bnd_acc + 4 * bidx,
                 p.evict + ((size_t)bidx * LH + lh) * p.blk);
  }
}

// Rarely taken tails of the selection kernel's last thread block, kept out of line so that they do not weigh on the
// register allocation of the jobs.
// Layer-by-layer step: the requests' counters move on at the end of the step (a whole-step launch does it where
// the attention kernel appends the token): one token further, the summary buffers swapped.  The first work item of
// a request names it once.
__device__ __noinline__ void advance_counters(const GpDev& p, int n_rc) {
  for (int idx = threadIdx.x; idx < n_rc; idx += blockDim.x) {
    const int* d = p.rcx + (size_t)idx * GP_DESC_INTS;
    if (d[4] == 0) {
      const int r = d[1];
      p.n[r] += 1; p.pos[r] += 1; p.started[r] = 1; p.sum_par[r] ^= 1;
    }
  }
  __syncthreads();
}
// A pool that holds a part of the model's KV heads: its sums of K^S and K^L per boundary request, zero past them
__device__ __noinline__ void publish_shard_sums(const GpDev& p, int n_bnd) {
  for (int e = threadIdx.x; e < p.M; e += blockDim.x) {
    p.shard_sums[2 * e] = e < n_bnd ? __ldcg(p.bnd_acc + 4 * e) : 0;
    p.shard_sums[2 * e + 1] = e < n_bnd ? __ldcg(p.bnd_acc + 4 * e + 1) : 0;
  }
}

// Thread blocks per unit: one that runs the three tasks side by side over one softmax pass, or, while the grid has
// three for every unit, one per task, each with all its warps.  Measured on units of 730 candidates, groups of 4: a task's
// block 6.6 us, a whole unit's 10.7 us (32 units on 296 blocks take the former); on 4608 units of 640 candidates the three
// passes over the logits that blocks per task take cost 150 us per step more.
__device__ __forceinline__ int jobs_per_unit(long long units, int grid) { return units * 3 <= grid ? 3 : 1; }

// pages of C that other requests share: each needs a copy-on-write target if boundary request e compresses
__device__ __forceinline__ void count_shared(const GpDev& p, int e) {
  if (threadIdx.x >= 32) return;
  const int4 inf = p.bnd_info[2 * e];
  const int* table = p.page_table + (size_t)inf.y * p.cap;
  int ksh = 0;
#pragma unroll 4
  for (int j = threadIdx.x; j < inf.z - p.sub; j += 32) ksh += (p.refcount[table[j]] > 1);
#pragma unroll
  for (int o2 = 16; o2 > 0; o2 >>= 1) ksh += __shfl_xor_sync(0xffffffffu, ksh, o2);
  if (threadIdx.x == 0) p.bnd_acc[4 * e + 2] = ksh;
}

// Whether the calling thread block finished the step's last job: only the blocks that had one are counted, the first of the
// grid where there is none.  (All blocks of the grid counted themselves and waited for the decisions, in steps without a boundary
// as well: 16 steps of four requests 346 us, now 317.)
__device__ __forceinline__ bool last_of_the_jobs(const GpDev& p, long long jobs, int* s_i) {
  if ((long long)blockIdx.x >= (jobs > 0 ? jobs : 1)) return false;
  const int blocks = jobs < (long long)gridDim.x ? (int)jobs : (int)gridDim.x;
  if (blocks <= 1) { __syncthreads(); return true; }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const int prev = atomicAdd(&p.hdr[HDR_DONE_SEL], 1);
    s_i[2] = (prev == blocks - 1);
    if (prev == blocks - 1) p.hdr[HDR_DONE_SEL] = 0;
  }
  __syncthreads();
  return s_i[2] != 0;
}

// The selection as a kernel of its own.  Two thread blocks to an SM at 128 registers; three at 80 spill and are slower
// (20 000 cycles per unit become 36 000).  Groups of eight spill at 128 as well (236 bytes a thread here, 268 in gp_chain_kernel, 244 in its form in clusters:
// the values of a token, eight per view, are loaded two tokens ahead), the smaller groups by 8 to 16 here, not at all in gp_chain_kernel (12 for
// groups of two in clusters).
template <int GG>
__global__ void __launch_bounds__(SEL_T, 2)
gp_bsel_kernel(const __grid_constant__ GpDev p, const int* __restrict__ req_ids, int n_req, int* __restrict__ actions,
               int by_layer, int serial, int decide) {
  // decide == 0: the step of a pool that holds a part of the model's KV heads: the last thread block only hands
  // out the sums of K^S and K^L per boundary request; the decisions follow in a kernel of their own once the
  // sums of all parts are added up
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((256u - (smem_u32(smem_raw) & 255u)) & 255u);
  const SelSmem S = sel_smem_at(smem, p.cap);
  int* s_i = S.m->s_i;

  const int LH = p.L * p.Hkv;
  // What the plan kernel wrote (counts, boundary records) is read before the wait for the attention kernel: the
  // plan kernel had completed before any CTA of the attention kernel let this grid be scheduled, and the
  // attention kernel does not touch these words; the loads go to the L2 (an L1 line could date from the step
  // before).  The first unit's record is fetched before the number of units is known (same round trip); slots
  // of bnd_info past the count hold stale but readable data that is then not used.
  int4 inf_first = make_int4(0, 0, 0, 0), inf2_first = inf_first;
  {
    const int b0 = (int)(blockIdx.x / LH);               // (one thread block per unit; with three they are fetched again)
    if (b0 < p.M) { inf_first = __ldcg(p.bnd_info + 2 * b0); inf2_first = __ldcg(p.bnd_info + 2 * b0 + 1); }
  }
  const int n_bnd = __ldcg(p.hdr + HDR_N_BND);
  const int n_rc = __ldcg(p.hdr + HDR_N_RC);
  const int NJ = jobs_per_unit((long long)n_bnd * LH, gridDim.x);
  const long long items = (long long)n_bnd * LH * NJ;
  gp_pdl_wait();
  gp_pdl_launch_dependents();

  for (long long item = blockIdx.x; item < items + n_bnd; item += gridDim.x) {
    if (item >= items) { count_shared(p, (int)(item - items)); continue; }
    const int u = (int)(item / NJ), bidx = u / LH, lh = u % LH;
    const bool is_first = NJ == 1 && item == (long long)blockIdx.x;
    sel_unit<GG>(p, S, bidx, lh, is_first ? inf_first : p.bnd_info[2 * bidx],          // {slot in the batch, request, P}
                  is_first ? inf2_first : p.bnd_info[2 * bidx + 1],                     // {offset into the logit scratch}
                  NJ == 1 ? 7 : 1 << (int)(item % NJ));
  }

  // ---- the last CTA takes the decisions ----------------------------------------------------------------------
  if (last_of_the_jobs(p, items + n_bnd, s_i)) {
    __threadfence();
    if (by_layer) advance_counters(p, n_rc);
    if (decide) decide_and_allocate(p, req_ids, n_req, n_bnd, actions, reinterpret_cast<int*>(S.loc), serial);
    else publish_shard_sums(p, n_bnd);
  }
}

// ------------------------------------------------------------------------------------------------------
// compaction
// ------------------------------------------------------------------------------------------------------
// shared memory of the compaction
struct CmpSmem {
  int4* s_info;      // [GP_MAX_REQ + 1] compressing requests: {request, P, boundary index, first part}
  int* ev;           // [CMP_EV] the order indices that the unit's compression (or Shrink) evicts, ascending
  int* ev_slot;      // [CMP_EV] where they lie: slot and page (its copy-on-write target, where it has one) of each
  int* ev_page;
  int* mv_page;      // [CMP_EV] slots from the unit's new end on: page, and new order index (-1: evicted)
  int* mv_rank;
  int* hole;         // [CMP_EV] evicted slots below the new end, as entries of `ev`
  int* mover;        // [CMP_EV] retained slots from the new end on, as entries of mv_page
  int* s_i;          // [8]
  int* order;        // [GP_MAX_REQ + 1] last CTA: pages each request gives back
};
constexpr int CMP_EV = 2 * GP_MAX_BLK;
constexpr size_t CMP_SMEM_BYTES = (GP_MAX_REQ + 1) * 16 + (7 * CMP_EV + 8 + GP_MAX_REQ + 1) * 4;
__device__ __forceinline__ CmpSmem cmp_smem_at(uint8_t* base) {       // base: 16-byte aligned, CMP_SMEM_BYTES
  CmpSmem C;
  C.s_info = reinterpret_cast<int4*>(base);
  C.ev = reinterpret_cast<int*>(base + (GP_MAX_REQ + 1) * 16);
  C.ev_slot = C.ev + CMP_EV;
  C.ev_page = C.ev_slot + CMP_EV;
  C.mv_page = C.ev_page + CMP_EV;
  C.mv_rank = C.mv_page + CMP_EV;
  C.hole = C.mv_rank + CMP_EV;
  C.mover = C.hole + CMP_EV;
  C.s_i = C.mover + CMP_EV;
  C.order = C.s_i + 8;
  return C;
}

// After the step's compactions: swaps in the copy-on-write targets, drops the references to the replaced pages, and those to
// the last page of every request that shrank.  A page whose last reference goes is pushed where the last of its droppers
// stands (requests in order, pages in table order), so that the free list does not depend on timing.  By one thread block,
// a warp per request, in four passes: drop; mark a page without references with the highest dropper (below zero); count
// each request's pushes; push.  (One warp that took the requests one after the other needed 1.5 ms for 256 requests of 128
// shared pages.)  `order`: GP_MAX_REQ + 1 ints of shared memory.
__device__ __noinline__ void swap_pages(const GpDev& p, const int4* s_info, int n_cmp, int* order) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int pass = 0; pass < 4; ++pass) {
    for (int ci = warp; ci < n_cmp; ci += nw) {
      const int r = s_info[ci].x, Pr = s_info[ci].y;
      const int keep = (s_info[ci].z & CMP_SHRINK) ? Pr - p.sub : Pr;        // pages from here on go back
      int* table = p.page_table + (size_t)r * p.cap;
      int* shadow = p.shadow + (size_t)r * p.cap;
      int n_push = pass == 3 ? *p.free_top + order[ci] : 0;
#pragma unroll 4
      for (int j0 = 0; j0 < Pr; j0 += 32) {
        const int j = j0 + lane;
        // the page that loses a reference: between the passes its number stands in the shadow entry as -2 - page
        int old = -1;
        if (j < Pr) {
          const int sh = shadow[j];
          if (pass == 0) {
            if (sh >= 0 || j >= keep) {
              old = table[j];
              if (sh >= 0) table[j] = sh;
              shadow[j] = -2 - old;
            }
          } else if (sh <= -2) {
            old = -2 - sh;
          }
        }
        if (pass == 0) {
          if (old >= 0) atomicSub(&p.refcount[old], 1);
        } else if (pass == 1) {
          if (old >= 0 && __ldcg(p.refcount + old) <= 0) atomicMin(&p.refcount[old], -(ci + 1));
        } else {
          const bool push = old >= 0 && __ldcg(p.refcount + old) == -(ci + 1);
          const unsigned mask = __ballot_sync(0xffffffffu, push);
          if (pass == 3) {
            if (push) { p.free_stack[n_push + __popc(mask & ((1u << lane) - 1u))] = old; p.refcount[old] = 0; }
            if (old >= 0) shadow[j] = -1;
          }
          n_push += __popc(mask);
        }
      }
      if (pass == 2 && lane == 0) order[ci] = n_push;
    }
    __syncthreads();
    if (pass == 2 && warp == 0) {                           // where each request's pushes start
      int carry = 0;
      for (int c0 = 0; c0 < n_cmp; c0 += 32) {
        const int v = c0 + lane < n_cmp ? order[c0 + lane] : 0;
        int inc = v;
#pragma unroll
        for (int o2 = 1; o2 < 32; o2 <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o2); if (lane >= o2) inc += t; }
        if (c0 + lane < n_cmp) order[c0 + lane] = carry + inc - v;
        carry += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (lane == 0) order[n_cmp] = carry;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *p.free_top += order[n_cmp];
}

// entries [0, n) whose flag is set, in ascending order into `out`, by one warp; returns their number
template <typename F>
__device__ __forceinline__ int warp_pack(int n, int* out, F flag) {
  const int lane = threadIdx.x & 31;
  int at = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 32) {
    const bool f = i0 + lane < n && flag(i0 + lane);
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (f) out[at + __popc(m & ((1u << lane) - 1u))] = i0 + lane;
    at += __popc(m);
  }
  return at;
}

// The compaction of a step, run by every CTA of the calling grid (CT threads).  Per compressing (request, layer, KV head)
// unit the `ne` evicted slots are closed by the retained rows that lie behind the unit's new end, which is all that
// moves: `ne` rows at most (16 of 700 at a page of 16).  The order of the tokens is not in the places of the rows but in a word per
// slot, its index in that order, and the stable compaction (retained history in order, then the protected window) is the
// subtraction of the evicted indices below it.  What bounds it: four dependent round trips per unit (list and page table, order indices,
// rows, stores), three thread blocks to an SM.  Every row behind the first evicted slot moved down (in 64-slot chunks that waited for one
// another where units were few): 467 us at 36 layers x 256 requests, now 73; 53, now 12, at 36 x 16; 187, now 26, at 64 x 32; the
// one-layer step of 64 requests 74.8 us, now 70.1.
// A ticket is a unit, or, where a unit has more than 4096 slots or is copied with few others, a part of one: a part tells where its
// evicted slots lie, and the unit's last part, which waits for that word of the others, moves the rows.  Tickets come from a counter, in
// order, so that those of a unit's other parts are with CTAs that run or have ended; only where every unit is one ticket, and none waits,
// a CTA's first is its number, which saves a round trip.
template <int D>
__device__ __forceinline__ void compact_body(const GpDev& p, const CmpSmem& C, int serial) {
  constexpr int CH = D / 8;
  constexpr int ROW_BYTES = D * 2;
  constexpr int PPS = 2 * CH;                            // 16-byte pieces of a slot, keys then values
  int4* s_info = C.s_info;
  int* ev = C.ev;
  int* s_i = C.s_i;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int LH = p.L * p.Hkv;
  // the first round trip fetches everything at once: the header and the list of compressing requests (its first
  // CT entries before their count is known; entries past the count are never looked at)
  if (tid == 0) s_i[3] = 0;
  if (tid <= p.M) s_info[tid] = p.cmp_info[tid];
  const int n_cmp = p.hdr[HDR_N_CMP];
  const int n_items = p.hdr[HDR_N_CITEM];
  const int n_cow = p.hdr[HDR_N_COW];
  // unique per decode step of the pool (the part flags are never cleared): the host's step count in the
  // asynchronous mode, where the two scratch sets count on their own; otherwise the counter the plan kernel keeps
  // on the device, so that a step replayed from a CUDA graph gets a stamp of its own
  const int stamp = p.async ? serial + 1 : p.hdr[HDR_STEP];
#pragma unroll 1
  for (int i = tid + CT; i <= n_cmp; i += CT) s_info[i] = p.cmp_info[i];
  int moved = 0;

  const bool own_first = n_items == n_cmp * LH;          // (every unit is one ticket)
  int item = blockIdx.x;
  for (bool first = own_first;; first = false) {
    __syncthreads();
    if (!first) {
      if (tid == 0) s_i[0] = (own_first ? (int)gridDim.x : 0) + atomicAdd(&p.hdr[HDR_WORK_CMP], 1);
      __syncthreads();
      item = s_i[0];
    }
    if (item >= n_items) break;
    // ticket -> (compressing request, layer/head, part); the parts of a unit are consecutive
    int lo = 0, hi = n_cmp;
#pragma unroll 1
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (LH * s_info[mid].w <= item) lo = mid; else hi = mid; }
    const int n_part = s_info[lo + 1].w - s_info[lo].w;
    const int rem = item - LH * s_info[lo].w;
    int lh = rem, part = 0;
    if (n_part > 1) { lh = rem / n_part; part = rem - lh * n_part; }
    const int4 inf = s_info[lo];
    const int l = lh / p.Hkv, h = lh % p.Hkv;
    const int Pr = inf.y;
    const int* table = p.page_table + (size_t)inf.x * p.cap;
    const int* shadow = p.shadow + (size_t)inf.x * p.cap;
    const bool shrink = (inf.z & CMP_SHRINK) != 0;
    const int e_bnd = inf.z & ((1 << CMP_LOG) - 1), log = (inf.z & (CMP_SHRINK - 1)) >> CMP_LOG;
    const int ne = shrink ? 2 * p.blk : p.blk;             // slots freed: one page of the method, two at a Shrink
    const int n_src = Pr * GP_PAGE, n_end = n_src - ne;    // the unit's slots, and those that stay in use
    const int c0 = part << log, c1 = part == n_part - 1 ? n_src : c0 + (1 << log);
    // order indices of a page's slots, and its rows: the unit's place in a page
    const size_t tok_stride = (size_t)p.Hkv * GP_PAGE, tok_base = gp_tok_off(p, l, 0, h);
    const size_t page_stride = (size_t)p.Hkv * 2 * GP_PAGE * ROW_BYTES;
    uint8_t* const unit_base = reinterpret_cast<uint8_t*>(p.kv + gp_tile_off(p, l, 0, h));

#pragma unroll 1
    for (int t = tid; t < ne; t += CT) {
      ev[t] = shrink ? p.evict2[((size_t)e_bnd * LH + lh) * 2 * p.blk + t] : p.evict[((size_t)e_bnd * LH + lh) * p.blk + t];
      C.ev_slot[t] = -1;
      C.mv_rank[t] = -1;
    }
    // pages that others share: copied whole, the evicted slots are closed in the copy (below)
    if (n_cow) {
      constexpr int TB = 2 * GP_PAGE * ROW_BYTES / 16;     // 16-byte pieces of a tile
      constexpr int U = 4;                                 // tiles in flight
      const int pg_end = min(c1, n_end) / GP_PAGE;
#pragma unroll 1
      for (int pg0 = c0 / GP_PAGE; pg0 < pg_end; pg0 += U) {
        uint4 val[U][TB / CT];
        int to[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int pg = pg0 + u;
          to[u] = pg < pg_end && pg < Pr - 1 ? shadow[pg] : -1;
          const uint4* src = reinterpret_cast<const uint4*>(unit_base + (size_t)(to[u] >= 0 ? table[pg] : 0) * page_stride);
#pragma unroll
          for (int e = 0; e < TB / CT; ++e) if (to[u] >= 0) val[u][e] = __ldcg(src + tid + e * CT);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          uint4* dst = reinterpret_cast<uint4*>(unit_base + (size_t)(to[u] >= 0 ? to[u] : 0) * page_stride);
#pragma unroll
          for (int e = 0; e < TB / CT; ++e) if (to[u] >= 0) dst[tid + e * CT] = val[u][e];
        }
      }
    }
    // the slots' new order indices, a slot per thread, SU of them in flight
    constexpr int SU = 4;
    bool listed = false;
#pragma unroll 1
    for (int i0 = c0; i0 < c1; i0 += SU * CT) {
      int from[SU], to[SU], rk[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int i = i0 + u * CT + tid, pg = i / GP_PAGE;
        from[u] = i < c1 ? table[pg] : 0;
        to[u] = i < c1 && n_cow && pg < Pr - 1 ? shadow[pg] : -1;
      }
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int i = i0 + u * CT + tid;
        rk[u] = i < c1 ? __ldcg(p.rank + tok_base + (size_t)from[u] * tok_stride + i % GP_PAGE) : -1;
      }
      if (!listed) { __syncthreads(); listed = true; }     // the list of evicted indices is there
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int i = i0 + u * CT + tid;
        if (i >= c1) continue;
        int below = 0;                                     // evicted indices before this slot's
        bool gone = false;
        if (ne == GP_PAGE) {
#pragma unroll
          for (int e = 0; e < GP_PAGE; ++e) { const int x = ev[e]; below += x < rk[u]; gone |= x == rk[u]; }
        } else {
          int hi2 = ne;
#pragma unroll 1
          while (below < hi2) { const int mid = (below + hi2) >> 1; if (ev[mid] < rk[u]) below = mid + 1; else hi2 = mid; }
          gone = below < ne && ev[below] == rk[u];
        }
        if (gone) {
          C.ev_slot[below] = i;
          C.ev_page[below] = to[u] >= 0 ? to[u] : from[u];
          continue;
        }
        moved += below > 0 || to[u] >= 0;
        if (i >= n_end) {
          C.mv_page[i - n_end] = from[u];
          C.mv_rank[i - n_end] = rk[u] - below;
        } else if (below > 0 || to[u] >= 0) {
          const size_t at = tok_base + i % GP_PAGE;
          p.rank[at + (size_t)(to[u] >= 0 ? to[u] : from[u]) * tok_stride] = rk[u] - below;
          if (to[u] >= 0) p.tok[at + (size_t)to[u] * tok_stride] = __ldcg(p.tok + at + (size_t)from[u] * tok_stride);
        }
      }
    }
    __syncthreads();
    if (n_part > 1) {
      // where a unit's evicted slots lie, found by its parts: in the place of its scores, which are done with (from cmp_off: with
      // early planning the next step's plan may be writing its own boundary records by now)
      int* found = reinterpret_cast<int*>(p.scores + (size_t)lh * p.max_boundary_tokens + __ldcg(p.cmp_off + e_bnd));        // [ne][2] (a unit has ne candidates at least)
      if (part < n_part - 1) {
#pragma unroll 1
        for (int t = tid; t < ne; t += CT)
          if (C.ev_slot[t] >= 0) { found[2 * t] = C.ev_slot[t]; found[2 * t + 1] = C.ev_page[t]; }
        __threadfence();
        __syncthreads();
        if (tid == 0 && !((p.withhold & GP_WITHHOLD_CHUNK) && part == 0))      // (test support: see GP_WITHHOLD_CHUNK)
          *reinterpret_cast<volatile int*>(p.cflags + item) = stamp;
        continue;
      }
      if (tid == 0) s_i[4] = 1;
      __syncthreads();
#pragma unroll 1
      for (int back = 1 + tid; back <= part; back += CT) {
        volatile int* prev = reinterpret_cast<volatile int*>(p.cflags + item - back);
        unsigned it = 0;
        while (*prev != stamp && it < p.spin_limit) ++it;
        if (it >= p.spin_limit) { atomicOr(p.err, GP_E_SPIN_CMP); s_i[4] = 0; }
      }
      __threadfence();
      __syncthreads();
      if (!s_i[4]) continue;                               // nothing is known of those slots: no row moves
#pragma unroll 1
      for (int t = tid; t < ne; t += CT)
        if (C.ev_slot[t] < 0) {
          const int2 f = __ldcg(reinterpret_cast<const int2*>(found) + t);
          if (f.x < 0 || f.x >= n_src || f.y < 0 || f.y >= p.n_pages) { atomicOr(p.err, GP_E_BOUNDS); continue; }     // that slot stays as it is
          C.ev_slot[t] = f.x; C.ev_page[t] = f.y;
        }
      __syncthreads();
    }
    // ---- the retained rows behind the new end into the evicted slots before it, each in ascending order (as many of the one
    // as of the other) ---------------------------------------------------------------------------------------------
    if (warp == 0) {
      const int n = warp_pack(ne, C.hole, [&](int e) { return C.ev_slot[e] >= 0 && C.ev_slot[e] < n_end; });
      if (lane == 0) s_i[1] = n;
    } else if (warp == 1) {
      const int n = warp_pack(ne, C.mover, [&](int e) { return C.mv_rank[e] >= 0; });
      if (lane == 0) s_i[5] = n;
    }
    __syncthreads();
    const int n_mv = min(s_i[1], s_i[5]);
#pragma unroll 1
    for (int k = tid; k < n_mv; k += CT) {
      const int hole = C.hole[k], mv = C.mover[k], ds = C.ev_slot[hole];
      const size_t at = tok_base + (size_t)C.ev_page[hole] * tok_stride + ds % GP_PAGE;
      p.rank[at] = C.mv_rank[mv];
      p.tok[at] = __ldcg(p.tok + tok_base + (size_t)C.mv_page[mv] * tok_stride + (n_end + mv) % GP_PAGE);
    }
    constexpr int MU = 2;
#pragma unroll 1
    for (int q0 = tid; q0 < n_mv * PPS; q0 += MU * CT) {
      uint4 val[MU];
#pragma unroll
      for (int u = 0; u < MU; ++u) {
        const int q = q0 + u * CT, k = q / PPS, c = q % CH, isv = q % PPS / CH;        // c: piece of the row (rows are swizzled by slot)
        if (k < n_mv) {
          const int mv = C.mover[k], s = (n_end + mv) % GP_PAGE;
          val[u] = *reinterpret_cast<const uint4*>(unit_base + (size_t)C.mv_page[mv] * page_stride + (isv * GP_PAGE + s) * ROW_BYTES + ((c ^ (s & 7)) << 4));
        }
      }
#pragma unroll
      for (int u = 0; u < MU; ++u) {
        const int q = q0 + u * CT, k = q / PPS, c = q % CH, isv = q % PPS / CH;
        if (k < n_mv) {
          const int hole = C.hole[k], s = C.ev_slot[hole] % GP_PAGE;
          *reinterpret_cast<uint4*>(unit_base + (size_t)C.ev_page[hole] * page_stride + (isv * GP_PAGE + s) * ROW_BYTES + ((c ^ (s & 7)) << 4)) = val[u];
        }
      }
    }
  }
  moved = __reduce_add_sync(0xffffffffu, moved);
  if (lane == 0 && moved) atomicAdd(&s_i[3], moved);
  __syncthreads();
  if (tid == 0 && s_i[3] > 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(p.counters + 8), (unsigned long long)s_i[3]);

  // ---- the last CTA swaps in the copy-on-write targets and drops the old references (App. D.2), and hands
  // back the last page of every request that shrank (Eq. 13) ---------------------------------------------
  if (n_cow == 0) return;                                 // nothing was shared and nobody shrank
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const int prev = atomicAdd(&p.hdr[HDR_DONE_CMP], 1);
    s_i[2] = (prev == (int)gridDim.x - 1);
    if (prev == (int)gridDim.x - 1) p.hdr[HDR_DONE_CMP] = 0;
  }
  __syncthreads();
  if (s_i[2]) {
    __threadfence();
    swap_pages(p, s_info, n_cmp, C.order);
  }
}


template <int D>
__global__ void __launch_bounds__(CT, 3)
gp_compact_kernel(const __grid_constant__ GpDev p, const int* __restrict__ req_ids, int n_req, int serial) {
  __shared__ __align__(16) uint8_t cmp_raw[CMP_SMEM_BYTES];
  gp_pdl_wait();
  gp_pdl_launch_dependents();
  compact_body<D>(p, cmp_smem_at(cmp_raw), serial);
}

// ------------------------------------------------------------------------------------------------------
// asynchronous boundary mode: the whole boundary chain of a step in one kernel, beside the next step's attention
// ------------------------------------------------------------------------------------------------------
// Launched right behind the attention kernel of step t + 1 as its programmatic dependent, this grid works on the
// boundary chain of step t: it does not wait for that attention kernel before it starts (everything it reads
// was complete before that kernel could start), runs the selection, lets the last CTA to finish it
// decide and allocate, waits inside the grid for that (a bounded wait on a flag: the grid is sized to be
// resident at once, on the room the attention kernel leaves), compacts, and only then waits for the attention
// kernel to end.  The grid therefore ends after both, and the plan of step t + 2, its programmatic dependent, finds the
// pages and counters of the requests that sat step t + 1 out in their final state.  `p`: the view of step t (its
// scratch set, the copy of the counters its decisions go to).
// LONG: launched in clusters, which share out units of many candidates (split_unit).  Synchronous mode only.
template <int D, int GG, bool LONG>
__global__ void __launch_bounds__(SEL_T, 2)
gp_chain_kernel(const __grid_constant__ GpDev p, int n_req, int serial, int has_chain, const int* __restrict__ req_ids,
                int* __restrict__ actions, int* __restrict__ actions_copy) {
  // actions_copy: where the step's actions are wanted as well once they are final (the host entry points: the
  // caller's array in page-locked host memory; writing them there from the plan kernel made that kernel wait
  // for the bus)
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((256u - (smem_u32(smem_raw) & 255u)) & 255u);
  const int tid = threadIdx.x;
  const int LH = p.L * p.Hkv;
  // Synchronous mode (same_step): the chain belongs to the step whose attention kernel runs beside this grid.
  // A selection job then waits until the consumer warps of that kernel have reported the unit's summary logits
  // complete (the items of requests at their boundary are a list of their own there, which a part of its grid draws
  // from first), the decisions are reported through `actions` as usual, and the next kernel on the stream may only be
  // scheduled once the attention kernel has ended (its early part reads counters that kernel advances).
  const bool same_step = !p.async;
  if (!same_step) gp_pdl_launch_dependents();
  if (has_chain) {
    const SelSmem S = sel_smem_at(smem, p.cap);
    int* s_i = S.m->s_i;
    const int n_bnd = __ldcg(p.hdr + HDR_N_BND);
    const int NJ = jobs_per_unit((long long)n_bnd * LH, gridDim.x);
    const long long items = (long long)n_bnd * LH * NJ;
    const long long units = (long long)n_bnd * LH;
    const int clusters = LONG ? (int)gridDim.x / CLUSTER : 0;
    // every work item of the request reports once per consumer warp for this unit (bounded wait; the
    // attention kernel's thread blocks were all resident before this grid could be scheduled)
    auto unit_there = [&](int bidx, int lh, int reports) {
      __syncthreads();
      if (tid == 0) {
        const volatile int* rdy = p.unit_ready + (size_t)bidx * LH + lh;
        unsigned it = 0;
        while (*rdy < reports && it < p.spin_limit) { ++it; __nanosleep(200); }
        if (it >= p.spin_limit) atomicOr(p.err, GP_E_SPIN_SEL);
        __threadfence();
      }
      __syncthreads();
    };
    bool last = false;                                     // this block finished the step's last job
    if (LONG && n_bnd > 0) {
      // Jobs are drawn from counters, not numbered by block, and counted as they are done: a cluster finds its place only where eight slots of
      // one GPC are free, and a block of more shared memory than an attention block left may not fit beside another until that one is gone, so no job may
      // be tied to a block that is not there yet (a grid that the occupancy query calls resident waited for its own decision that way).
      SelMisc& m = *S.m;
      if (tid < 32) {
        int cnt = 0;
        for (int b0 = 0; b0 < n_bnd; b0 += 32) {
          const unsigned bits = __ballot_sync(0xffffffffu, b0 + tid < n_bnd && split_unit(p, S, __ldcg(&p.bnd_info[2 * min(b0 + tid, n_bnd - 1)].z), units, clusters));
          if (tid == 0) m.shared_out[b0 / 32] = bits;
          cnt += __popc(bits);
        }
        if (tid == 0) m.n_shared = cnt;
      }
      __syncthreads();
      const int n_sh = m.n_shared, sh_units = n_sh * LH;
      const int nj = jobs_per_unit((long long)(n_bnd - n_sh) * LH, gridDim.x), others = (n_bnd - n_sh) * LH * nj;
      auto done = [&]() {                                  // a job is; whether it was the last of all
        __syncthreads();
        if (tid == 0) {
          __threadfence();
          const int total = sh_units + others + n_bnd;
          s_i[2] = atomicAdd(&p.hdr[HDR_DONE_SEL], 1) == total - 1;
          if (s_i[2]) p.hdr[HDR_DONE_SEL] = 0;
        }
        __syncthreads();
        last |= s_i[2] != 0;
      };
      if (n_sh > 0) {
        cluster_sync();                                    // every block of the cluster has started: another's shared memory may be written from here on
#pragma unroll 1
        for (;;) {
          if (cluster_rank() == 0 && tid == 0) {
            const int t = atomicAdd(&p.hdr[HDR_WORK_SPLIT], 1);
#pragma unroll 1
            for (int r = 0; r < CLUSTER; ++r) *of_block(&m.ticket, r) = t;
          }
          cluster_sync();
          const int u = m.ticket;
          if (u >= sh_units) break;
          const int bidx = nth_request(m.shared_out, n_bnd, u / LH, true), lh = u % LH;
          const int4 inf = p.bnd_info[2 * bidx], inf2 = p.bnd_info[2 * bidx + 1];
          unit_there(bidx, lh, inf2.z);
          sel_split<GG>(p, S, bidx, lh, inf, inf2);
          if (cluster_rank() == 0) {
            if (tid == 0) atomicAdd(reinterpret_cast<unsigned long long*>(p.counters + 11), 1ull);
            done();
          }
        }
      }
#pragma unroll 1
      for (;;) {
        __syncthreads();
        if (tid == 0) m.ticket = atomicAdd(&p.hdr[HDR_WORK_SEL], 1);
        __syncthreads();
        const int item = m.ticket;
        if (item >= others + n_bnd) break;
        if (item >= others) {
          count_shared(p, item - others);
        } else {
          const int u = item / nj, bidx = nth_request(m.shared_out, n_bnd, u / LH, false), lh = u % LH;
          const int4 inf = p.bnd_info[2 * bidx], inf2 = p.bnd_info[2 * bidx + 1];
          if (inf.z > p.sub) unit_there(bidx, lh, inf2.z);
          sel_unit<GG>(p, S, bidx, lh, inf, inf2, nj == 1 ? 7 : 1 << (item - u * nj));
        }
        done();
      }
    }
#pragma unroll 1
    for (int item = blockIdx.x; !LONG && item < (int)items + n_bnd; item += gridDim.x) {
      if (item >= (int)items) { count_shared(p, item - (int)items); continue; }
      const int u = item / NJ, bidx = u / LH, lh = u % LH;
      const int4 inf = p.bnd_info[2 * bidx];
      const int4 inf2 = p.bnd_info[2 * bidx + 1];
      if (same_step && inf.z > p.sub) unit_there(bidx, lh, inf2.z);
      sel_unit<GG>(p, S, bidx, lh, inf, inf2, NJ == 1 ? 7 : 1 << (item - u * NJ));
    }
    // ---- the last CTA to finish its jobs takes the decisions and tells the others ------------------------------
    const int stamp = same_step ? p.hdr[HDR_STEP] : serial + 1;
    if (LONG && n_bnd > 0 ? last : last_of_the_jobs(p, items + n_bnd, s_i)) {
      __threadfence();
      decide_and_allocate(p, req_ids, n_req, n_bnd, same_step ? actions : nullptr, reinterpret_cast<int*>(S.loc), serial);
      __syncthreads();
      if (tid == 0 && !(p.withhold & GP_WITHHOLD_DECIDED)) {      // (test support: see GP_WITHHOLD_DECIDED)
        __threadfence();
        *reinterpret_cast<volatile int*>(p.hdr + HDR_DECIDED) = stamp;
      }
    } else if (tid == 0 && n_bnd > 0) {
      volatile int* flag = reinterpret_cast<volatile int*>(p.hdr + HDR_DECIDED);
      unsigned it = 0;
      while (*flag != stamp && it < p.spin_limit) { ++it; __nanosleep(100); }
      if (it >= p.spin_limit) atomicOr(p.err, GP_E_SPIN_CMP);
      __threadfence();
    }
    __syncthreads();
    if (same_step) {
      // The attention kernel of this step has all but ended by now (the decisions needed its last reports).  From here on the
      // next kernel on the stream may be scheduled.  With early planning that is the next step's plan, which so runs
      // beside the compaction below: the decisions it reads are taken, the attention kernel has moved the requests on, and
      // the compaction reads nothing the plan writes.
      gp_pdl_wait();
      if (actions_copy && blockIdx.x == gridDim.x - 1)
        for (int i = tid; i < n_req; i += SEL_T) actions_copy[i] = __ldcg(actions + i);
      gp_pdl_launch_dependents();
    }
    // ---- compaction: its arrays take the place of the selection's (no request at its boundary: nothing was decided) --------
    if (n_bnd > 0) compact_body<D>(p, cmp_smem_at(smem), serial);
  }
  if (same_step) return;
  gp_pdl_wait();              // the attention kernel beside which this grid ran has ended
}

// the decisions of a step whose sums of K^S and K^L were completed outside (KV heads spread over several pools)
__global__ void __launch_bounds__(SEL_T)
gp_decide_kernel(const __grid_constant__ GpDev p, const int* __restrict__ req_ids, int n_req, int* __restrict__ actions,
                 int serial) {
  __shared__ int s_arr[8 * GP_MAX_REQ];
  decide_and_allocate(p, req_ids, n_req, __ldcg(p.hdr + HDR_N_BND), actions, s_arr, serial, true);
}

}  // namespace

// the kernels of a pool: head dimension and query heads per KV head
static auto compact_kernel_of(const GpDev& p) -> void (*)(const GpDev, const int*, int, int) {
  return p.d == 128 ? gp_compact_kernel<128> : gp_compact_kernel<64>;
}
typedef void (*SelKernel)(const GpDev, const int*, int, int*, int, int, int);
static SelKernel sel_kernel_of(const GpDev& p) {
  return p.G == 1 ? gp_bsel_kernel<1> : p.G == 2 ? gp_bsel_kernel<2> : p.G == 4 ? gp_bsel_kernel<4> : gp_bsel_kernel<8>;
}
typedef void (*ChainKernel)(const GpDev, int, int, int, const int*, int*, int*);
template <int D, bool LONG> static ChainKernel chain_kernel_d(const GpDev& p) {
  return p.G == 1 ? gp_chain_kernel<D, 1, LONG> : p.G == 2 ? gp_chain_kernel<D, 2, LONG> : p.G == 4 ? gp_chain_kernel<D, 4, LONG> : gp_chain_kernel<D, 8, LONG>;
}
static ChainKernel chain_kernel_of(const GpDev& p, bool clusters) {
  if (clusters) return p.d == 128 ? chain_kernel_d<128, true>(p) : chain_kernel_d<64, true>(p);
  return p.d == 128 ? chain_kernel_d<128, false>(p) : chain_kernel_d<64, false>(p);
}

// shared memory of the selection for a per-request page cap
static size_t gp_sel_smem(const GpDev& p) {
  const size_t tail = sel_loc_bytes(p.cap) + 2 * (size_t)sel_n_cap(p.cap) * sizeof(double);
  return (sizeof(SelMisc) + 15) / 16 * 16 + (tail > DECIDE_SMEM ? tail : DECIDE_SMEM) + 256;
}
static_assert((sizeof(SelMisc) + 15) / 16 * 16 + ((GP_MAX_TILES_PER_REQ / 2 + 2) * 4 + 15) / 16 * 16 + 2 * SEL_CAP * sizeof(double) + 256 <= GP_MAX_DYN_SMEM,
              "the largest page cap fits");
static_assert(CMP_SMEM_BYTES <= sizeof(SelMisc) + DECIDE_SMEM, "the compaction's arrays take the selection's place");

// one-time setup for a pool: opts the selection kernels into their shared memory and sizes the grids to at most one
// resident wave, so that no CTA waits for another to leave before it can start
void gp_boundary_setup(const GpDev& p, int num_sms, int* grid_sel, int* grid_compact, int* grid_chain, int* grid_long) {
  const size_t sel_sm = gp_sel_smem(p);
  auto blocks = [&](auto kern, int threads, size_t smem, int most) {
    if (smem) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    return num_sms * (occ > most ? most : occ > 0 ? occ : 1);
  };
  *grid_sel = blocks(sel_kernel_of(p), SEL_T, sel_sm, 32);
  *grid_chain = blocks(chain_kernel_of(p, false), SEL_T, sel_sm, 2);
  // in clusters, where a request of this pool can have a unit that they share out: as many as are resident at once
  *grid_long = 0;
  if ((long long)p.cap * GP_PAGE > SPLIT_FROM && p.metric != GP_METRIC_ENTROPY && p.policy != GP_POLICY_SHRINK) {
    const ChainKernel kern = chain_kernel_of(p, true);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CLUSTER; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(num_sms * 2 / CLUSTER * CLUSTER)); cfg.blockDim = dim3(SEL_T); cfg.dynamicSmemBytes = sel_sm;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sel_sm) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0)
      *grid_long = (n * CLUSTER < num_sms * 2 ? n : num_sms * 2 / CLUSTER) * CLUSTER;
    else
      (void)cudaGetLastError();
    // (one request alone must not have more units than the clusters may take; see split_unit)
    if ((long long)p.L * p.Hkv > (long long)SPLIT_ROUNDS * (*grid_long / CLUSTER)) *grid_long = 0;
  }
  *grid_compact = blocks(compact_kernel_of(p), CT, 0, 32);
}

// the boundary chain of the step whose view is `p` (asynchronous mode: none when !has_chain)
void gp_launch_chain(const GpDev& p, int n_req, int serial, int has_chain, int grid, cudaStream_t s, bool pdl, const int* req_ids,
                     int* actions, int* actions_copy, bool clusters) {
  gp_launch_clusters(clusters ? CLUSTER : 1, chain_kernel_of(p, clusters), grid, SEL_T, gp_sel_smem(p), s, pdl, p, n_req, serial, has_chain, req_ids,
                     actions, actions_copy);
}

void gp_launch_select_only(const GpDev& p, const int* req_ids, int n_req, int* actions, int grid_sel, cudaStream_t s, bool pdl,
                           int serial) {
  gp_launch(sel_kernel_of(p), grid_sel, SEL_T, gp_sel_smem(p), s, pdl, p, req_ids, n_req, actions, 0, serial, 0);
}

// plain launches: what comes before them on the stream (the caller's reduction of the sums) is not this library's
void gp_launch_decide_compact(const GpDev& p, const int* req_ids, int n_req, int* actions, int grid_compact, cudaStream_t s,
                              int serial) {
  gp_launch(gp_decide_kernel, 1, SEL_T, 0, s, false, p, req_ids, n_req, actions, serial);
  gp_launch(compact_kernel_of(p), grid_compact, CT, 0, s, true, p, req_ids, n_req, serial);
}

void gp_launch_boundary(const GpDev& p, const int* req_ids, int n_req, int* actions, bool by_layer, int grid_sel,
                        int grid_compact, cudaStream_t s, cudaEvent_t ev, bool pdl, int serial) {
  // asynchronous mode: the kernel before this one on its stream belongs to another step (an event wait lies in
  // between): plain launch; the compaction kernel follows as a programmatic dependent as usual
  gp_launch(sel_kernel_of(p), grid_sel, SEL_T, gp_sel_smem(p), s, pdl && !p.async, p, req_ids, n_req, actions, by_layer ? 1 : 0, serial, 1);
  if (ev) cudaEventRecord(ev, s);
  gp_launch(compact_kernel_of(p), grid_compact, CT, 0, s, pdl, p, req_ids, n_req, serial);
}
