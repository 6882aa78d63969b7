// Fused append + GQA paged decode attention (Sec. 4.1) with the update of the two query summaries (Eq. 6, App. D.1),
// plus, for requests that reach their capacity boundary with this step, the logits of the two calibrated summaries
// (Eq. 12) against every candidate key while the key tile is in shared memory.
//
// Work decomposition.  The plan kernel cuts every stepped request into chunks of `chunk_pages` pages and
// writes one descriptor per chunk, those of requests at their boundary first, each part sorted by descending cost; a work item is
// (chunk, layer, KV head).  The CTAs of a persistent grid (two per SM) draw them in that order.  Each CTA is warp-specialised:
//
//   warp 0      producer: draws the CTA's items and publishes each in a ring of item slots: descriptor, query rows
//               (and the new key/value row, and the position's cosines and sines) by bulk copy, page ids.
//   warps 1, 3  summaries: the first item of a request's unit carries its summaries one step on (read from one of the
//               request's two buffers, written to the other); every item with candidate pages of a request at its
//               boundary gets the calibrated, rotated summaries q~ in the CTA's single q~ buffer, each item's CTA from
//               the old buffer for itself.  (They were CTAs of the plan kernel: 8 us before the first key could be
//               asked for in a layer-by-layer launch, 300 us of the step at 36 layers x 256 requests, and q~ went through
//               global memory.)
//   warps 4..7  consumers: take the tiles of an item round-robin (tile j, at d = 64 pair j of tiles, belongs to warp (j - its item's number) mod 4,
//               so the odd tiles of successive items fall on different warps).  Each warp
//               fetches its own K|V tiles (one contiguous 8 KB per (layer, page, head)) with 16-byte
//               asynchronous copies into a private ring of stages, running ahead across item boundaries, so
//               the ring never drains between items.  The G query heads of the group are rows 0..G-1 of an
//               m16n8k16 bf16 MMA; S = Q K^T and O += P V run on the tensor cores with fp32 accumulation.
//               Rows 8..15 of the A operand carry the bf16 rounding residual of rows 0..7 (of the rotated
//               query when RoPE is on, of P always), which costs nothing and gives ~16 mantissa bits.  For
//               boundary units the summary logits of a candidate page are an fp64 tensor-core contraction
//               (m8n8k4 DMMA: 8 tokens x (2 views x G heads) x d).  With NORM the query rows and the new key row arrive
//               raw: the summary warps normalise the queries in the slot (RMS over the head dimension, a learned weight
//               per element), the warp that appends the key normalises that.
//   warp 2      merger: combines the four consumers' partial (max, sum, O) of an item and writes the output
//               or, for requests split over several items, the partial; the merger whose partial is a unit's last merges
//               them all, in the order of the chunks.
//               Consumers hand over through a double buffer and go straight on to the next item.
//
// The two warp groups re-split the register file (setmaxnreg; 256 registers for a thread of each as launched): see SERVICE_REGS.
// All waits are bounded; a wait that gives up sets an error bit (with a code for which wait it was) and an
// abort flag that drains the CTA.  No wait of an item depends on a later item being published.
#include "gp_dev.cuh"

namespace {

constexpr int NI = 4;                      // item slots per CTA
constexpr int NSW = 2;                     // tile stages per consumer warp (at most 3: see the wait in the tile loop)
constexpr int NCW = 4;                     // consumer warps
constexpr int NTHREADS = 256;              // warp group 0: producer, summaries, merger, summaries; warp group 1: consumers
constexpr int NSUM = 2;                    // summary warps
constexpr int MERGE_FAN = 8;               // partial outputs merged at a time
constexpr double QT_SCALE = 0x1p880;       // of the q~ buffer: see bf16_lo_scaled
constexpr double Z_SCALE = 0x1p16;         // of the logits made from it
constexpr int SLOT_UNIT = 20;              // of an item's slot: offset of the unit's tile of page 0 (two words)
constexpr int QT_PAD = 8;                  // doubles of padding per q~ row: rows alternate bank halves

template <int D>
struct Geo {
  static constexpr int ROW_BYTES = D * 2;
  static constexpr int TILE_BYTES = 2 * GP_PAGE * ROW_BYTES;
  // Tiles a consumer warp takes at a time: two of 4 KB at d = 64, where one cost nearly the instructions (softmax, its shuffles, the ring) of
  // one of 8 KB (64 layers x 32 requests of 200 to 1800 tokens, groups of 4: 772 us one by one, 5.6 TB/s; now 690, 6.3 TB/s)
  static constexpr int PAIR = 128 / D;
  static constexpr int STAGE_BYTES = PAIR * TILE_BYTES;                // 8 KB
  // The weights are carried as two bf16 terms, 2^-17 of each, where two tiles share a running maximum as three: the weight at a new maximum
  // is one and carries no rounding, and tile by tile there are more of those (error of the outputs against 64 bits, 48 requests of 64 to 240
  // tokens in groups of 1 to 8: tile by tile 1.61e-6 to 1.66e-6, in pairs with two terms 1.71e-6 to 1.78e-6, now 1.6e-7, groups of eight
  // 1.22e-6).  For groups of up to four the third stands in rows of the product that no head has: lanes 16 to 31 repeat the heads of lanes
  // 0 to 15.  Groups of eight take another product, for the first tile of a pair only (for both: 6.5 % of a step).  us of this kernel at
  // 64 layers x 32 requests of 200 to 1800 tokens, none / two of them at a boundary: groups of four one by one 772 / 877, in pairs
  // 673 / 775, with the third term 690 / 803; groups of eight 821 / 1029, 741 / 1044, 757 / 1086.
  static constexpr bool THREE = PAIR > 1;
  static constexpr int KSTEPS = D / 16;
  static constexpr int DTILES = D / 8;
  static constexpr int SLOT_DESC = 384;                                // 96 ints: descriptor (32), then up to 64 page ids
  static constexpr int SLOT_PAGES = 32;                                // first page id (int index)
  static constexpr int SLOT_ROPE = SLOT_DESC + 10 * ROW_BYTES;         // cosine and sine of the position, D / 2 pairs of floats
  static constexpr int SLOT_BYTES = (SLOT_ROPE + D / 2 * 8 + 127) / 128 * 128;
};

struct Lay {            // shared-memory layout, depends on the group size
  int ncomb, off_slots, off_qt, off_comb, comb_warp, off_bars, off_misc, total;
};
constexpr int SMEM_ALIGN = 256;          // the kernel rounds the start of its shared memory up to this
template <int D>
__host__ __device__ constexpr Lay make_lay(int G) {
  using GEO = Geo<D>;
  Lay L = {};
  L.ncomb = (D == 128 && G == 8) ? 1 : 2;
  L.off_slots = NCW * NSW * GEO::STAGE_BYTES;
  L.off_qt = L.off_slots + NI * GEO::SLOT_BYTES;
  const int nrows = 2 * G < 8 ? 8 : 2 * G;
  L.off_comb = L.off_qt + nrows * (D + QT_PAD) * 8;
  L.comb_warp = (16 + (GEO::THREE && G < 8 ? 2 : 1) * G * D) * 4;     // maxima and sums, then rows (and the third terms' part of them)
  L.off_bars = L.off_comb + L.ncomb * NCW * L.comb_warp;
  L.off_misc = L.off_bars + (4 * NI + 2 + 4) * 8;
  L.total = L.off_misc + 128 + SMEM_ALIGN;   // abort flag and code; room for the rounding
  return L;
}
// two thread blocks to an SM, each with the 1 KB the system takes of its own
static_assert(2 * (make_lay<128>(8).total + 1024) <= 228 * 1024 && 2 * (make_lay<128>(4).total + 1024) <= 228 * 1024 &&
              2 * (make_lay<64>(8).total + 1024) <= 228 * 1024, "shared memory of two thread blocks");

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// bounded, abort-aware wait
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int where, uint32_t limit) {
  for (uint32_t it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 63u && *abort_flag) return false;
  }
  if (*abort_flag == 0) abort_flag[1] = where;      // which wait gave up first (reported with the error bit)
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void dmma(double& d0, double& d1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(d0), "+d"(d1)
               : "d"(a), "d"(b));
}

// double -> float -> bf16, each round-to-nearest-even (the order a host library takes)
__device__ __forceinline__ __nv_bfloat16 to_bf16(double x) { return __float2bfloat16_rn((float)x); }
__device__ __forceinline__ uint32_t pack_bf16_d(double lo, double hi) { return pack_bf16((float)lo, (float)hi); }

// Partial outputs [n][G][D + 2] at `first`, `stride` floats apart (unnormalised output, running maximum in the log2 domain, sum
// of exponentials), merged by one warp in ascending order, so that the result does not depend on who merges: into output
// rows, or, with `into`, into a partial output again (the first one's place: a row is read before it is written).
template <int D>
__device__ __forceinline__ void merge_unit(float* first, size_t stride, int n, int G, float* __restrict__ orow, bool into) {
  constexpr int PER2 = D / 64;                           // float2 pieces of a row per lane
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int g0 = 0; g0 < G; g0 += 4) {                    // four heads at a time
    const int g = g0 + (lane & 3);                       // lane: head g0 + lane % 4, partials lane / 4, + 8, ...
    const float* ml = first + (g < G ? g : 0) * (D + 2) + D;
    float M = -INFINITY, ls = 0.f;
#pragma unroll 1
    for (int c = lane >> 2; c < n; c += 8) {
      const float2 v = __ldcg(reinterpret_cast<const float2*>(ml + c * stride));
      const float Mn = fmaxf(M, v.x);
      ls = ls * exp2f(M - Mn) + exp2f(v.x - Mn) * v.y;
      M = Mn;
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {                   // (a lane without a partial: M is -inf, weight 0)
      const float Mo = __shfl_xor_sync(0xffffffffu, M, o), lo = __shfl_xor_sync(0xffffffffu, ls, o);
      const float Mn = fmaxf(M, Mo);
      ls = (M == -INFINITY ? 0.f : ls * exp2f(M - Mn)) + (Mo == -INFINITY ? 0.f : lo * exp2f(Mo - Mn));
      M = Mn;
    }
    float2 acc[4][PER2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int e = 0; e < PER2; ++e) acc[q][e] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int c0 = 0; c0 < n; c0 += 2) {                  // two partials' values in flight
      float2 vv[2][4][PER2];
      float mv[2][4];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const bool here = c0 + k < n;                  // (past the last one: weight 0 and values 0, whatever that one holds)
          const float* pr = first + (c0 + k) * stride + (g0 + q < G ? g0 + q : 0) * (D + 2);
          mv[k][q] = here ? __ldcg(pr + D) : -INFINITY;
#pragma unroll
          for (int e = 0; e < PER2; ++e) vv[k][q][e] = here ? __ldcg(reinterpret_cast<const float2*>(pr) + lane + 32 * e) : make_float2(0.f, 0.f);
        }
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float wgt = exp2f(mv[k][q] - __shfl_sync(0xffffffffu, M, q));
#pragma unroll
          for (int e = 0; e < PER2; ++e) { acc[q][e].x += wgt * vv[k][q][e].x; acc[q][e].y += wgt * vv[k][q][e].y; }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float tot = __shfl_sync(0xffffffffu, ls, q), Mq = __shfl_sync(0xffffffffu, M, q);
      if (g0 + q < G) {
        const float inv = into ? 1.f : 1.f / tot;
        float2* dst = reinterpret_cast<float2*>(into ? first + (g0 + q) * (D + 2) : orow + (g0 + q) * D);
#pragma unroll
        for (int e = 0; e < PER2; ++e) dst[lane + 32 * e] = make_float2(acc[q][e].x * inv, acc[q][e].y * inv);
        if (into && lane == 0) { first[(g0 + q) * (D + 2) + D] = Mq; first[(g0 + q) * (D + 2) + D + 1] = tot; }
      }
    }
  }
}

// The summaries of one unit, the heads g = w, w + NSUM, ... by the calling warp (w): Eq. 6 on the un-rotated query from the
// request's current buffer to the other one (`owner`), and, with `qt`, the calibrated (Eq. 12) and rotated summaries q~ into
// the q~ buffer (times QT_SCALE), all in fp64.  What bounds it is the round trip for the old rows: two heads' (both views)
// are in flight together, and the first ones' are asked for before anything else, the wait for the query rows (`rows_there`; false: it gave
// up) included.  With NORM the warp first normalises its
// heads' query rows in the slot and reports them on `norm_bar`: the consumers wait for that.
template <int D, bool ROPE, bool NORM, typename Rows>
__device__ __forceinline__ bool summary_rows(const GpDev& p, const GpNorm& nm, uint8_t* qrows, Rows rows_there, uint64_t* norm_bar, int w, int G,
                                             int l, int h, int r, int bi, int par, bool started, bool owner, double* qt) {
  constexpr int PER = D / 32;
  const int lane = threadIdx.x & 31;
  __nv_bfloat16* q0 = reinterpret_cast<__nv_bfloat16*>(qrows);
  double ov[2][2][PER];                                   // [head of the pair][view]
  auto load_old = [&](int g0) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (g0 + NSUM * k < G) {
          const double* o0 = p.summ + gp_summ_off(p, l, r, par, x, h * G + g0 + NSUM * k);
#pragma unroll
          for (int e = 0; e < PER; ++e) ov[k][x][e] = __ldcg(o0 + lane + 32 * e);
        }
  };
  if (owner || qt) load_old(w);
  if (!rows_there()) return false;
  if (NORM) {                    // the summaries follow the query after its normalisation and before its rotation (Sec. 3.2)
    for (int g = w; g < G; g += NSUM) {
      float qf[PER];
      double ssq = 0.0;
#pragma unroll
      for (int e = 0; e < PER; ++e) { qf[e] = __bfloat162float(q0[g * D + lane + 32 * e]); ssq += (double)qf[e] * (double)qf[e]; }
#pragma unroll
      for (int o2 = 16; o2 > 0; o2 >>= 1) ssq += __shfl_xor_sync(0xffffffffu, ssq, o2);
      const double scale = 1.0 / sqrt(ssq / (double)D + nm.eps);
#pragma unroll
      for (int e = 0; e < PER; ++e) q0[g * D + lane + 32 * e] = to_bf16((double)qf[e] * scale * (double)__ldg(nm.wq + lane + 32 * e));
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(norm_bar);
  }
  if (!owner && !qt) return true;
#pragma unroll 1
  for (int g0 = w; g0 < G; g0 += 2 * NSUM) {
    if (g0 != w) load_old(g0);
    double ss[2][2], sq[2];                                // sums of squares: new summaries, query
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int g = g0 + NSUM * k;
      ss[k][0] = ss[k][1] = sq[k] = 0.0;
      if (g < G) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const double qv = (double)__bfloat162float(q0[g * D + lane + 32 * e]);
          sq[k] += qv * qv;
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const double beta = x ? p.beta_l : p.beta_s;
            const double nv = started ? beta * ov[k][x][e] + (1.0 - beta) * qv : qv;             // Eq. 6
            ov[k][x][e] = nv;
            ss[k][x] += nv * nv;
          }
        }
        if (owner) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            double* newp = p.summ + gp_summ_off(p, l, r, par ^ 1, x, h * G + g);
#pragma unroll
            for (int e = 0; e < PER; ++e) newp[lane + 32 * e] = ov[k][x][e];
          }
        }
      }
    }
    if (!qt) continue;
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        sq[k] += __shfl_xor_sync(0xffffffffu, sq[k], o2);
        ss[k][0] += __shfl_xor_sync(0xffffffffu, ss[k][0], o2);
        ss[k][1] += __shfl_xor_sync(0xffffffffu, ss[k][1], o2);
      }
    }
    // Eq. 12: lane 2k + x works out its gamma (roots and quotients once for the four rows)
    const double my_ss = lane & 2 ? (lane & 1 ? ss[1][1] : ss[1][0]) : (lane & 1 ? ss[0][1] : ss[0][0]);
    const double my_sq = lane & 2 ? sq[1] : sq[0];
    const double gam = (my_ss > 0.0 ? sqrt(my_sq / (double)D) / sqrt(my_ss / (double)D) : 1.0) * QT_SCALE;
    double2 cs[PER / 2];
#pragma unroll
    for (int e = 0; e < PER / 2; ++e)
      if (ROPE) cs[e] = *reinterpret_cast<const double2*>(p.rope_cs + ((size_t)bi * (D / 2) + lane + 32 * e) * 2);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const double gamma = __shfl_sync(0xffffffffu, gam, 2 * k + x);
        if (g0 + NSUM * k < G) {
          double* dst = qt + (size_t)(x * G + g0 + NSUM * k) * (D + QT_PAD);
#pragma unroll
          for (int e = 0; e < PER / 2; ++e) {
            const int j = lane + 32 * e;
            const double x1 = gamma * ov[k][x][e], x2 = gamma * ov[k][x][e + PER / 2];
            dst[j] = ROPE ? x1 * cs[e].x - x2 * cs[e].y : x1;
            dst[j + D / 2] = ROPE ? x2 * cs[e].x + x1 * cs[e].y : x2;
          }
        }
      }
  }
  return true;
}

__device__ __forceinline__ float upper_half(float x, uint32_t mask) { return __uint_as_float(__float_as_uint(x) & mask); }

// bf16 -> double by its bits, scaled by 2^-896 (an 8-bit exponent read as an 11-bit one): exact for every finite number, and
// cheaper than the conversion unit.  The q~ buffer holds the summaries times 2^880, the logits are scaled by the remaining 2^16:
// all powers of two, so that the logits are what they were.  (The calibrated summary of a query whose elements are near the
// largest bf16, 2^128, can be sqrt(d) times as large and twice that after its rotation: 2^133 at most, and 2^896 times that is
// past the largest double.)
__device__ __forceinline__ double bf16_lo_scaled(uint32_t w) { return __hiloint2double((int)((uint32_t)((int)(w << 16) >> 3) & 0x8fffffffu), 0); }
__device__ __forceinline__ double bf16_hi_scaled(uint32_t w) { return __hiloint2double((int)((uint32_t)((int)(w & 0xffff0000u) >> 3) & 0x8fffffffu), 0); }

// fp64 logits of a boundary unit's calibrated summaries against the 16 keys of a candidate page, by one warp:
// Z[token][n] = sum_d K[token][d] q~[n][d], n = view * G + head.  One m8n8k4 DMMA covers 8 tokens,
// 8 columns and 4 values of d; inside a 16-byte chunk of a key row lane t of a quad takes the
// bf16 pair at byte 4t, whose low and high element feed two successive k-steps (q~ is read with
// the same mapping, so the contraction is over the same d on both sides).  One block of eight columns at a time (nt of them: a
// group of eight heads has two).  What bounds it: the fp64 pipe and four chains of dependent DMMAs; the registers it takes are
// the consumers' (two blocks together spilled: 84.0 ms against 80.0 on 36 layers x 256 requests).  Stores the exponentials
// per token and the page's softmax partials per column.  Keys that are infinite or not numbers, which their bits read as a
// double's are not, are looked for on the way and put in afterwards.
template <int D>
__device__ __forceinline__ void summary_logits(const GpDev& p, const uint8_t* tile, const double* qt, int G, int lh, long long zoff,
                                               int tok0, int nt) {
  constexpr int CH = D / 8, ROW_BYTES = D * 2;
  const int lane = threadIdx.x & 31, grp = lane >> 2, t4 = lane & 3;
  double z[2][2][2];                                      // [even / odd chunks][token half][column pair]
#pragma unroll
  for (int i = 0; i < 8; ++i) (&z[0][0][0])[i] = 0.0;
  const int n = nt * 8 + grp;                             // B column held by this lane's group (past 2G: another one's, not stored)
  const double* qrow = qt + (size_t)(n < 2 * G ? n : 0) * (D + QT_PAD) + 2 * t4;
  const uint8_t* krow0 = tile + grp * ROW_BYTES + 4 * t4;
  const uint8_t* krow1 = tile + (8 + grp) * ROW_BYTES + 4 * t4;
  uint32_t most = 0;                                      // the largest magnitudes among the keys' low and high halves, as bits
#pragma unroll 4
  for (int c = 0; c < CH; c += 2) {
#pragma unroll
    for (int odd = 0; odd < 2; ++odd) {
      const uint32_t ka = *reinterpret_cast<const uint32_t*>(krow0 + (((c + odd) ^ grp) << 4));   // grp == token & 7
      const uint32_t kb = *reinterpret_cast<const uint32_t*>(krow1 + (((c + odd) ^ grp) << 4));
      const double2 qq = *reinterpret_cast<const double2*>(qrow + (c + odd) * 8);
      most = __vmaxu2(most, __vmaxu2(ka & 0x7fff7fffu, kb & 0x7fff7fffu));
      dmma(z[odd][0][0], z[odd][0][1], bf16_lo_scaled(ka), qq.x);
      dmma(z[odd][1][0], z[odd][1][1], bf16_lo_scaled(kb), qq.x);
      dmma(z[odd][0][0], z[odd][0][1], bf16_hi_scaled(ka), qq.y);
      dmma(z[odd][1][0], z[odd][1][1], bf16_hi_scaled(kb), qq.y);
    }
  }
  const double inv_sqrt_d = Z_SCALE / sqrt((double)D);
  // D fragment: row = grp (token), columns 2*t4, 2*t4 + 1
  const int col = nt * 8 + 2 * t4;
  double z00 = (z[0][0][0] + z[1][0][0]) * inv_sqrt_d, z01 = (z[0][0][1] + z[1][0][1]) * inv_sqrt_d;
  double z10 = (z[0][1][0] + z[1][1][0]) * inv_sqrt_d, z11 = (z[0][1][1] + z[1][1][1]) * inv_sqrt_d;
  if (__any_sync(0xffffffffu, (most & 0xffffu) >= 0x7f80u || most >= 0x7f800000u)) {       // such a key adds infinity, or no number
#pragma unroll 1
    for (int j = 0; j < D; ++j) {
      const double* qj = qt + (size_t)(col < 2 * G ? col : 0) * (D + QT_PAD) + j;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const uint32_t kw = *reinterpret_cast<const uint16_t*>(tile + (half * 8 + grp) * ROW_BYTES + (((j >> 3) ^ grp) << 4) + (j & 7) * 2);
        if ((kw & 0x7f80u) == 0x7f80u) {
          (half ? z10 : z00) += (double)bf16_lo_f(kw) * qj[0];
          (half ? z11 : z01) += (double)bf16_lo_f(kw) * qj[D + QT_PAD];
        }
      }
    }
  }
  // the page's softmax partials per column: max and sum of exponentials over its 16 tokens; the
  // exponentials themselves are what is stored per token
  double m0 = fmax(z00, z10), m1 = fmax(z01, z11);
#pragma unroll
  for (int o2 = 4; o2 < 32; o2 <<= 1) {
    m0 = fmax(m0, __shfl_xor_sync(0xffffffffu, m0, o2));
    m1 = fmax(m1, __shfl_xor_sync(0xffffffffu, m1, o2));
  }
  z00 = exp(z00 - m0); z10 = exp(z10 - m0); z01 = exp(z01 - m1); z11 = exp(z11 - m1);
  double e0 = z00 + z10, e1 = z01 + z11;
#pragma unroll
  for (int o2 = 4; o2 < 32; o2 <<= 1) {
    e0 += __shfl_xor_sync(0xffffffffu, e0, o2);
    e1 += __shfl_xor_sync(0xffffffffu, e1, o2);
  }
  if (col < 2 * G) {
    // view = col / G (short or long summary); a view's values of one unit are contiguous [token][G]
    const size_t tokrow = (size_t)(zoff + tok0 + grp);
    if (G >= 2) {
      const int lg = 31 - __clz(G);                       // (a power of two)
      double* z0 = p.zbuf + (((((size_t)lh * 2 + (col >> lg)) * p.z_stride + tokrow) << lg) + (col & (G - 1)));
      *reinterpret_cast<double2*>(z0) = make_double2(z00, z01);
      *reinterpret_cast<double2*>(z0 + (size_t)8 * G) = make_double2(z10, z11);
    } else {
      double* zS = p.zbuf + ((size_t)lh * 2 * p.z_stride + tokrow);
      double* zL = zS + p.z_stride;
      zS[0] = z00; zS[8] = z10; zL[0] = z01; zL[8] = z11;
    }
    if (grp == 0) {
      double* st2 = p.zstat + (((size_t)lh * ((unsigned long long)p.max_boundary_tokens / GP_PAGE) + (unsigned long long)(zoff + tok0) / GP_PAGE) * (2 * G) + col) * 2;
      *reinterpret_cast<double2*>(st2) = make_double2(m0, e0);
      *reinterpret_cast<double2*>(st2 + 2) = make_double2(m1, e1);
    }
  }
}

// WIDE: groups of eight query heads.  MODE: a whole step, a layer of one, or a layer with raw queries and keys.
enum { WHOLE_STEP, ONE_LAYER, ONE_LAYER_NORM };
template <int D, bool ROPE, int MODE, bool WIDE>
__global__ void __launch_bounds__(NTHREADS, 2)
gp_attn_kernel(const __grid_constant__ GpDev p, int n_req, const __nv_bfloat16* __restrict__ q,
               const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, float* __restrict__ out, int lh0,
               int lh_n, int adv_lh, int planned, const GpNorm nm) {
  // lh0, lh_n: the (layer, KV head) units this launch covers, [lh0, lh0 + lh_n): all of them, or one layer's
  // adv_lh: the unit whose append also moves the request's counters on by one token (-1: none; the layer-by-layer
  // step does that at its end)
  // planned (a layer's launch): the step's plan had completed before this grid could start.  It follows another layer's launch on
  // its stream, and that one waited for the plan before it let this one be scheduled.  Then only the caller's tensors depend on the
  // kernel before this one: descriptor, page ids, the first tiles and the old summaries are asked for while that kernel drains, and
  // the producer waits before it asks for the first rows.  Whatever is written follows those rows.  (36 layers x 16 requests of 400 to 1000
  // tokens, layer by layer: 864 us per step with every launch waiting at its top, now 760; with an ordinary kernel of 3 us before each
  // layer 999, now 925.  In the whole step's kernel the rows share the descriptor's barrier: two barriers there cost 1 to 2 %.)
  constexpr bool LAYER = MODE != WHOLE_STEP, NORM = MODE == ONE_LAYER_NORM;
  // Registers of a service thread; the consumers, which hold the output accumulators, get the rest of 256.  At 80 it is the merge and the summaries that
  // spill at d = 128 (140 bytes a thread for whole steps of groups of eight with rotary embeddings), at 88 52 to 96 bytes in a layer's launches, at 96 0 to 16
  // in a whole step's, at 104 the consumers again; nothing at d = 64.  us of a step at 72 / 80 / 88 / 96 / 104 for all launches:
  // one layer x 64 requests 63.1 / 62.7 / 62.4 / 62.3 / 64.7, 150 of 100 to 500 tokens 65.0 / 64.4 / 63.5 / 63.1 / 67.3, d = 64 52.0 / 51.1 / 51.0 / 51.2 / 51.1;
  // a layer by itself (4 steps x 36) 3089 / 3025 / 2964 / 3005 / 3311 (groups of eight, us a layer, 28.9 at 80, 27.5 at 88); groups of eight on 8 layers x 20
  // 154.9 / 152.4 / 157 / 148.5 / 160.9.  Groups of eight with rotary embeddings at 72 / 80 / 88 / 96: 64 layers x 32 1630 / 1607 / 1611 / 1623,
  // 8 x 20 158.5 / 156.0 / 155.8 / 157.1, one layer x 64 80.2 / 79.2 / 78.8 / 79.5, 4 x 4 of 2000 to 8000 tokens 104.0 / 103.8 / 104.2 / 105.1.
  constexpr int SERVICE_REGS = D == 64 || LAYER ? 88 : WIDE && ROPE ? 80 : 96;
  using GEO = Geo<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (-smem_u32(smem_raw) & (SMEM_ALIGN - 1u));
  const int G = p.G;
  const Lay L = make_lay<D>(G);
  const uint32_t NCOMB = (uint32_t)L.ncomb;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.off_bars);
  uint64_t* slot_full = bars;                  // [NI] descriptor and page ids, and, but in a layer's launch, the rows
  uint64_t* slot_empty = slot_full + NI;       // [NI]
  uint64_t* slot_norm = slot_empty + NI;       // [NI] the slot's query rows have been normalised
  uint64_t* slot_rows = slot_norm + NI;        // [NI] a layer's launch: the slot's query, key and value rows are there
  uint64_t* qt_full = slot_rows + NI;
  uint64_t* qt_empty = qt_full + 1;
  uint64_t* comb_full = qt_empty + 1;          // [2]
  uint64_t* comb_empty = comb_full + 2;        // [2]
  volatile int* s_misc = reinterpret_cast<volatile int*>(smem + L.off_misc);   // [0] abort
  double* qt = reinterpret_cast<double*>(smem + L.off_qt);                     // [2G][D + QT_PAD]
  float* comb = reinterpret_cast<float*>(smem + L.off_comb);                   // [2][NCW][16 + G*D]
  const int comb_w = L.comb_warp / 4;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t lim = p.spin_limit;
  if (tid == 0) {
    for (int i = 0; i < NI; ++i) { mbar_init(&slot_full[i], LAYER ? 1 : 2); mbar_init(&slot_rows[i], 1); mbar_init(&slot_empty[i], NCW + 1 + NSUM); mbar_init(&slot_norm[i], NSUM); }
    mbar_init(qt_full, NSUM);
    mbar_init(qt_empty, NCW);
    for (int i = 0; i < 2; ++i) { mbar_init(&comb_full[i], NCW); mbar_init(&comb_empty[i], 1); }
    s_misc[0] = 0;
    s_misc[1] = 0;
    fence_mbar_init();
  }
  if (!LAYER || !planned) {
    gp_pdl_wait();                // everything above touched only this CTA's shared memory
    gp_pdl_launch_dependents();
  }
  __syncthreads();

  // the descriptor of the item of this CTA's own number, which its first one nearly always is, is fetched before the numbers of items
  // are known (same round trip): a slot past them holds stale but readable data that is then not used
  int hFirst = 0;
  // What runs once before the first tile is paid in instruction fetch: the numbers of items in 32 bits (their 64-bit quotients were calls of a
  // hundred instructions), a unit's layer and head worked out by the producer alone (us a pass with the tiles' addresses as they are: tiny, 16
  // steps, 286 / 279; 36 x 16 layer by layer, 4 steps, 3040 / 3000; 1 x 64, 16 steps, 1085 / 1074).
  const unsigned units = (unsigned)lh_n;
  unsigned rc = blockIdx.x / units;            // the item's descriptor
  if (warp == 0 && lane < GP_DESC_INTS && (int)rc < p.max_rc) hFirst = p.rcx[(size_t)rc * GP_DESC_INTS + lane];
  const int n_rc = __ldcg(p.hdr + HDR_N_RC), n_brc = __ldcg(p.hdr + HDR_N_BRC);
  const int LH = p.L * p.Hkv;
  // (32 bits: every item has a partial output of 264 bytes or more in the pool)
  const int total_b = n_brc * lh_n, total = n_rc * lh_n;
  const int q_bytes = G * GEO::ROW_BYTES;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SERVICE_REGS));
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(256 - SERVICE_REGS));
  }
  if (warp == 0) {
    // ================================= producer ===========================================
    // Two lists: the items of requests at their boundary, whose tiles also pay for the fp64 logits (bound by the DMMA pipe, 26 cycles
    // each, which keeps a sub-partition from much else), and the others, which are bound by memory; costliest first in each.  A part of
    // the grid draws from the former as long as there are any, the rest from the latter, so that the logits hide behind other
    // blocks' loads: half of the grid where the boundary items fit there at once (their requests' selection waits for them), else a
    // third (36 layers x 256 requests 4375 us per step with half, 4312 with a third, 4336 with a quarter).  One list, boundary
    // items first, so that all blocks were at them and the memory idle: 4478; 36 x 16: 328, now 313; 64 x 32 with groups of 8: 1813, now 1774.
    // A CTA's first item follows from its number, the others are drawn from a counter per list, and
    // only once the item before the one last published is done: a CTA holds the item it works on and the next, and what is
    // left goes to whoever is free.  (Dealt out statically by an estimate of their cost, the CTAs of a one-layer step ended
    // between 26 and 38 us; drawn as far ahead as a ring of eight slots allows, they hoarded.)  Which CTA takes an item does
    // not change its result.
    const int total_p = total - total_b, cta = blockIdx.x, grid = gridDim.x;
    const int b_ctas = total_b <= grid / 2 ? total_b : grid / 3;      // blocks that draw boundary items first
    const int first_p = min(total_p, grid - b_ctas), first_b = min(total_b, grid - first_p);
    // an item's number: of the first list, then of the second
    int item = cta < b_ctas ? cta : cta - b_ctas < first_p ? total_b + cta - b_ctas : cta - first_p < first_b ? cta - first_p : total;
    bool left[2] = {true, true};               // items of the lists this CTA still asks for
    int hdr = hFirst;                          // descriptor header, word `lane` (lanes 0..15)
    if (item != cta && item < total) {
      rc = (unsigned)item / units;
      if (lane < GP_DESC_INTS) hdr = p.rcx[(size_t)rc * GP_DESC_INTS + lane];
    }
    for (uint32_t n = 0;; ++n) {
      const int sl = n % NI;
      if (!wait_bar(&slot_empty[sl], ((n / NI) & 1u) ^ 1u, s_misc, 1, lim)) break;
      uint8_t* slot = smem + L.off_slots + sl * GEO::SLOT_BYTES;
      int* sd = reinterpret_cast<int*>(slot);
      const bool rows_later = LAYER && planned && n == 0;
      if (item >= total) {
        if (rows_later) { gp_pdl_wait(); gp_pdl_launch_dependents(); }
        if (lane == 0) sd[3] = -1;
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&slot_full[sl]);
          if (!LAYER) mbar_arrive(&slot_full[sl]);
        }
        break;
      }
      const int lh = lh0 + item - (int)(rc * units);
      const int l = (int)((unsigned)lh / (unsigned)p.Hkv), h = lh - l * p.Hkv;
      const int bi = __shfl_sync(0xffffffffu, hdr, 0);
      const int r = __shfl_sync(0xffffffffu, hdr, 1), pg0 = __shfl_sync(0xffffffffu, hdr, 2);
      const int npg = __shfl_sync(0xffffffffu, hdr, 3);
      const int chunk = __shfl_sync(0xffffffffu, hdr, 4);
      const int nchunks = __shfl_sync(0xffffffffu, hdr, 5);
      int pg = -1, pg2 = -1;                   // page ids of tiles `lane` and `lane + 32` of the item
      if (lane < npg) pg = p.page_table[(size_t)r * p.cap + pg0 + lane];
      if (lane + 32 < npg) pg2 = p.page_table[(size_t)r * p.cap + pg0 + 32 + lane];
      if (lane < 14) sd[lane] = hdr;
      if (lane == 14) sd[14] = lh;
      if (lane == 15) sd[15] = hdr;            // index among the step's boundary requests
      if (lane == 16) sd[16] = item & (NCW - 1);              // the consumer warp that takes the item's first tile
      if (lane == 17) sd[17] = l;
      if (lane == 18) sd[18] = h;
      __syncwarp();
      auto ask_rows = [&]() {
        const bool has_new = (chunk == nchunks - 1);
        uint64_t* bar = LAYER ? &slot_rows[sl] : &slot_full[sl];
        fence_proxy_async();
        mbar_expect_tx(bar, q_bytes + (has_new ? 2 * GEO::ROW_BYTES : 0) + (ROPE ? D / 2 * 8 : 0));
        bulk_g2s(slot + GEO::SLOT_DESC, q + (((size_t)l * n_req + bi) * p.Hq + h * G) * D, q_bytes, bar);
        if (ROPE) bulk_g2s(slot + GEO::SLOT_ROPE, p.rope_f + (size_t)bi * D, D / 2 * 8, bar);
        if (has_new) {
          const size_t kvo = (((size_t)l * n_req + bi) * p.Hkv + h) * D;
          bulk_g2s(slot + GEO::SLOT_DESC + 8 * GEO::ROW_BYTES, k + kvo, GEO::ROW_BYTES, bar);
          bulk_g2s(slot + GEO::SLOT_DESC + 9 * GEO::ROW_BYTES, v + kvo, GEO::ROW_BYTES, bar);
        }
      };
      if (lane == 0 && !rows_later) ask_rows();
      if (lane == 0)                                         // the unit's place in a page, in bytes from the first layer's first page
        *reinterpret_cast<unsigned long long*>(sd + SLOT_UNIT) = gp_tile_off(p, l, 0, h) * sizeof(__nv_bfloat16);
      sd[GEO::SLOT_PAGES + lane] = pg;
      sd[GEO::SLOT_PAGES + 32 + lane] = pg2;
      __syncwarp();
      // (test support: the first CTA's second item can be withheld, so that the consumers' bounded wait runs out)
      const bool withheld = (p.withhold & GP_WITHHOLD_ITEM) && blockIdx.x == 0 && n == 1;
      if (lane == 0 && !withheld) mbar_arrive(&slot_full[sl]);
      if (rows_later) {
        gp_pdl_wait();
        gp_pdl_launch_dependents();
        if (lane == 0) ask_rows();
      }
      // ---- the next item ----------------------------------------------------------------------------------
      if (n > 0 && !wait_bar(&slot_empty[(n - 1) % NI], ((n - 1) / NI) & 1u, s_misc, 2, lim)) break;
      item = total;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int list = cta < b_ctas ? k : 1 - k;
        if (item < total || !left[list]) continue;
        int t = 0;
        if (lane == 0) t = atomicAdd(p.tickets + 2 * (lh0 / p.Hkv) + list, 1);
        const int at = (list ? first_p : first_b) + __shfl_sync(0xffffffffu, t, 0);
        left[list] = at < (list ? total_p : total_b);
        if (left[list]) item = list ? total_b + at : at;
      }
      hdr = 0;
      if (item < total) {
        rc = (unsigned)item / units;
        if (lane < GP_DESC_INTS) hdr = p.rcx[(size_t)rc * GP_DESC_INTS + lane];
      }
    }
  } else if (warp >= 4) {
    // ================================= consumers ==========================================
    const int cw = warp - 4;
    const float sc = 1.4426950408889634f * rsqrtf((float)D);
    constexpr bool REPEAT = GEO::THREE && !WIDE;
    const int row = lane >> 2;
    const bool third = REPEAT && row >= 4;                 // this lane has the third terms of head row - 4
    const int head = third ? row - 4 : row;
    const uint32_t keep = third ? 0u : 0xffffffffu, cut = third || WIDE ? 0xffff0000u : 0u;
    const int qc = (lane & 3) * 2;
    uint32_t qt_uses = 0, my_tiles = 0;
    // Each consumer warp fetches its own tiles (tile j of an item belongs to warp j mod 4) into its private
    // ring of NSW stages: as soon as it is done with a stage it issues the copy of its next tile but NSW - 1,
    // which may belong to a later item (the fetch position runs ahead of the compute position, across item
    // boundaries, but never further than the ring of item slots allows).  No other warp touches the ring, so
    // program order plus a proxy fence orders the reads of a stage before the copy that overwrites it.
    const uint64_t kv_policy = l2_policy_evict_first();    // the K/V stream is read once per step: first out of the L2
    constexpr int PAIR = GEO::PAIR;
    uint32_t my_fetch = 0, f_it = 0;
    int f_pgl = 0, f_npg = 0;
    bool f_have = false, f_done = false;
    auto top_up = [&](uint32_t it_now) -> bool {           // false: a wait gave up
      while (!f_done && my_fetch - my_tiles < (uint32_t)NSW) {
        const int* fsd = reinterpret_cast<const int*>(smem + L.off_slots + (f_it % NI) * GEO::SLOT_BYTES);
        if (!f_have) {
          if (f_it + 1 >= it_now + NI) break;              // that slot may still hold an item this warp has not finished
          // an item ahead of the one being computed is fetched from only if its slot is already there:
          // nothing the current item needs may wait for a later item to be published
          if (f_it > it_now) {
            if (!mbar_test_wait(&slot_full[f_it % NI], (f_it / NI) & 1u)) break;
          } else if (!wait_bar(&slot_full[f_it % NI], (f_it / NI) & 1u, s_misc, 3, lim)) {
            return false;
          }
          f_npg = fsd[3];
          if (f_npg < 0) { f_done = true; break; }
          f_pgl = (cw + fsd[16]) % NCW;                   // in units of PAIR tiles; the first goes to another warp from item to item
          f_have = true;
        }
        if (f_pgl * PAIR >= f_npg) { ++f_it; f_have = false; continue; }
        const uint32_t fst = cw * NSW + (my_fetch % NSW);
#pragma unroll
        for (int sub = 0; sub < PAIR; ++sub) {
          if (sub && f_pgl * PAIR + sub >= f_npg) break;
          const int page = fsd[GEO::SLOT_PAGES + f_pgl * PAIR + sub];
          // 16-byte asynchronous copies through the load/store path, 512 contiguous bytes per warp instruction:
          // the bulk-copy engine takes several hundred cycles to accept an 8 KB copy, which paced the kernel
          // A fetch is a third of what a tile costs a consumer warp (cycles, one request alone: fetch 530, S 290, softmax 300, weights and
          // P V 310, the rest 250), so the unit's place is in the slot: with the unit's layer and head taken apart here by divisions, per
          // fetch, it was that; now 390, and no register more is held through the loop and the logits (kept in registers it cost
          // groups of eight 5 % of a step in spills).  us of this kernel before / now: 64 layers x 32 requests, groups of eight, none and two at a
          // boundary 1345 / 1328 and 1741 / 1659; 36 x 256, 16 at a boundary 3941 / 3763; 36 x 16, two 285 / 280.
          const uint8_t* src = reinterpret_cast<const uint8_t*>(p.kv) + *reinterpret_cast<const unsigned long long*>(fsd + SLOT_UNIT) +
                               (uint64_t)(uint32_t)page * ((uint32_t)p.Hkv * GEO::TILE_BYTES) + lane * 16;
          const uint32_t dst = smem_u32(smem + fst * GEO::STAGE_BYTES + sub * GEO::TILE_BYTES) + lane * 16;
#pragma unroll
          for (int c = 0; c < GEO::TILE_BYTES / 512; ++c) cp_async16_hint(dst + c * 512, src + c * 512, kv_policy);
        }
        cp_async_commit();
        ++my_fetch;
        f_pgl += NCW;
      }
      return true;
    };
    for (uint32_t it = 0;; ++it) {
      const int sl = it % NI;
      if (!top_up(it)) break;
      if (!wait_bar(&slot_full[sl], (it / NI) & 1u, s_misc, 4, lim)) break;
      const uint8_t* slot = smem + L.off_slots + sl * GEO::SLOT_BYTES;
      const int* sd = reinterpret_cast<const int*>(slot);
      const int npg = sd[3];
      if (npg < 0) break;
      const int bi = sd[0], pg0 = sd[2], chunk = sd[4], nchunks = sd[5], n_old = sd[6];
      const int flags = sd[8], Pr = sd[9], lh = sd[14];
      const int n_new = n_old + 1;
      const bool need_qt = (flags & 1) && (pg0 < Pr - 1);

      if (LAYER && !wait_bar(NORM ? &slot_norm[sl] : &slot_rows[sl], (it / NI) & 1u, s_misc, NORM ? 11 : 12, lim)) break;
      // ---- query fragments (A operand), rotated when RoPE is on ----------------------------------
      uint32_t qa[GEO::KSTEPS][2];
      uint32_t ql[GEO::KSTEPS][2];
      {
        const bool valid = head < G;
        const uint8_t* qrow = slot + GEO::SLOT_DESC + (valid ? head : 0) * GEO::ROW_BYTES;
#pragma unroll
        for (int kk = 0; kk < GEO::KSTEPS; ++kk)
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            qa[kk][half] = valid ? *reinterpret_cast<const uint32_t*>(qrow + (kk * 16 + half * 8 + qc) * 2) : 0u;
            ql[kk][half] = 0u;
          }
        if (ROPE) {                                        // column col pairs with col + D / 2: the fragment KSTEPS / 2 on
#pragma unroll
          for (int kk = 0; kk < GEO::KSTEPS / 2; ++kk)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              const int j = kk * 16 + half * 8 + qc;
              const uint32_t w1 = qa[kk][half], w2 = qa[kk + GEO::KSTEPS / 2][half];
              const float4 cs = *reinterpret_cast<const float4*>(slot + GEO::SLOT_ROPE + j * 8);     // (j is even)
              const float c0 = cs.x, s0 = cs.y, c1 = cs.z, s1 = cs.w;
              const float a0 = bf16_lo_f(w1) * c0 - bf16_lo_f(w2) * s0, a1 = bf16_hi_f(w1) * c1 - bf16_hi_f(w2) * s1;
              const float b0 = bf16_lo_f(w2) * c0 + bf16_lo_f(w1) * s0, b1 = bf16_hi_f(w2) * c1 + bf16_hi_f(w1) * s1;
              const uint32_t ha = pack_bf16(a0, a1), hb = pack_bf16(b0, b1);
              qa[kk][half] = ha;
              ql[kk][half] = pack_bf16(a0 - bf16_lo_f(ha), a1 - bf16_hi_f(ha));
              qa[kk + GEO::KSTEPS / 2][half] = hb;
              ql[kk + GEO::KSTEPS / 2][half] = pack_bf16(b0 - bf16_lo_f(hb), b1 - bf16_hi_f(hb));
            }
        }
      }
      bool qt_here = false;                                // the item's q~ is in the buffer

      const bool last_chunk = (chunk == nchunks - 1);
      float o[GEO::DTILES][4];
#pragma unroll
      for (int i = 0; i < GEO::DTILES; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
      float m_run = -INFINITY, l_run = 0.f;
      bool ok = true;

      for (int pgl = (cw + sd[16]) % NCW * PAIR; pgl < npg; pgl += NCW * PAIR) {
        const uint32_t st = cw * NSW + (my_tiles % NSW);
        {
          // one copy group per tile, in fetch order: all but the groups younger than this tile's must be done
          const uint32_t younger = my_fetch - my_tiles - 1;
          if (younger == 0) cp_async_wait<0>(); else if (younger == 1) cp_async_wait<1>(); else cp_async_wait<2>();
          __syncwarp();
        }
        ++my_tiles;
        uint8_t* stage = smem + st * GEO::STAGE_BYTES;
        const int tok0 = (pg0 + pgl) * GP_PAGE;
        const int nsub = PAIR == 1 ? 1 : min(PAIR, npg - pgl);         // tiles of the stage
        const bool has_new = last_chunk && (pgl + PAIR >= npg);        // the last of them is the request's
        if (has_new) {
          uint8_t* tile = stage + (nsub - 1) * GEO::TILE_BYTES;
          // append: slot n_old of this page receives k_t, v_t; patch the staged copy too
          const int s = n_old - tok0 - (nsub - 1) * GP_PAGE;
          const int page = sd[GEO::SLOT_PAGES + npg - 1], l = sd[17], h = sd[18];
          constexpr int CH = D / 8;
          uint4 k_new = make_uint4(0, 0, 0, 0);
          if (NORM) {
            // the raw key row (a chunk of eight elements per lane, CH lanes): normalised per head, rotated to the token's
            // position, its cache form
            const int c = lane % CH;
            const uint4 raw = *reinterpret_cast<const uint4*>(slot + GEO::SLOT_DESC + 8 * GEO::ROW_BYTES + c * 16);
            const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
            double e[8];
            double ss = 0.0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              e[2 * i] = bf16_lo_f(w[i]); e[2 * i + 1] = bf16_hi_f(w[i]);
              ss += e[2 * i] * e[2 * i] + e[2 * i + 1] * e[2 * i + 1];
            }
#pragma unroll
            for (int o2 = 1; o2 < CH; o2 <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o2);
            const double ks = 1.0 / sqrt(ss / (double)D + nm.eps);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              e[i] = e[i] * ks * (double)__ldg(nm.wk + c * 8 + i);
              if (ROPE) {
                const double other = __shfl_xor_sync(0xffffffffu, e[i], CH / 2);     // element j + D / 2 of j, and back
                const double* cs = p.rope_cs + ((size_t)bi * (D / 2) + (c % (CH / 2)) * 8 + i) * 2;
                e[i] = c < CH / 2 ? e[i] * cs[0] - other * cs[1] : e[i] * cs[0] + other * cs[1];
              }
            }
            k_new = make_uint4(pack_bf16_d(e[0], e[1]), pack_bf16_d(e[2], e[3]), pack_bf16_d(e[4], e[5]), pack_bf16_d(e[6], e[7]));
          }
          if (lane < 2 * CH) {
            const int isv = lane / CH, c = lane % CH;
            const uint4 val = NORM && !isv ? k_new
                                           : *reinterpret_cast<const uint4*>(slot + GEO::SLOT_DESC + (8 + isv) * GEO::ROW_BYTES + c * 16);
            const int off = isv * GP_PAGE * GEO::ROW_BYTES + s * GEO::ROW_BYTES + ((c ^ (s & 7)) << 4);
            *reinterpret_cast<uint4*>(tile + off) = val;
            uint8_t* g = reinterpret_cast<uint8_t*>(p.kv + gp_tile_off(p, l, page, h)) + off;
            *reinterpret_cast<uint4*>(g) = val;
            fence_proxy_async();
          }
          if (lane == 0) {
            const size_t at = gp_tok_off(p, l, page, h) + s;
            p.tok[at] = sd[7];
            p.rank[at] = n_old;                            // the newest token: last in the order
          }
          if (lane == 1 && lh == adv_lh) {
            // the request is one token further, its summaries in the other buffer (nothing in this kernel looks at these
            // words: what it needs is in the descriptors)
            const int r = sd[1];
            p.n[r] = n_new; p.pos[r] = (long long)sd[7] + 1; p.started[r] = 1; p.sum_par[r] = sd[12] ^ 1;
          }
          __syncwarp();
        }
        // S = Q K^T for the 16 tokens of each page
        float s_acc[PAIR][2][4];
#pragma unroll
        for (int i = 0; i < PAIR * 8; ++i) (&s_acc[0][0][0])[i] = 0.f;
#pragma unroll
        for (int sub = 0; sub < PAIR; ++sub) {
          if (sub && sub >= nsub) break;
          const int token = (lane & 7) + ((lane >> 4) << 3);
          const int csel = (lane >> 3) & 1;
          const uint32_t rowaddr = smem_u32(stage) + sub * GEO::TILE_BYTES + token * GEO::ROW_BYTES;
#pragma unroll
          for (int kk = 0; kk < GEO::KSTEPS; ++kk) {
            uint32_t b00, b01, b10, b11;
            ldsm_x4(rowaddr + ((((2 * kk + csel) ^ (token & 7))) << 4), b00, b01, b10, b11);
            mma_bf16(s_acc[sub][0], qa[kk][0], ql[kk][0], qa[kk][1], ql[kk][1], b00, b01);
            mma_bf16(s_acc[sub][1], qa[kk][0], ql[kk][0], qa[kk][1], ql[kk][1], b10, b11);
          }
        }
        // online softmax in the log2 domain
        float sv[PAIR][2][2];
        const int n_valid = has_new ? (n_new - tok0) : nsub * GP_PAGE;
        float mx = -INFINITY;
#pragma unroll
        for (int sub = 0; sub < PAIR; ++sub)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            float x = s_acc[sub][nt][j];
            if (ROPE) x += s_acc[sub][nt][j + 2];
            x *= sc;
            if (sub * GP_PAGE + nt * 8 + qc + j >= n_valid) x = -INFINITY;
            sv[sub][nt][j] = x;
            mx = fmaxf(mx, x);
          }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);
        const float corr = exp2f(m_run - m_new);
        if (__any_sync(0xffffffffu, corr != 1.f)) {
          l_run *= corr;
#pragma unroll
          for (int i = 0; i < GEO::DTILES; ++i) {
            o[i][0] *= corr; o[i][1] *= corr; o[i][2] *= corr; o[i][3] *= corr;
          }
        }
        m_run = m_new;
#pragma unroll
        for (int sub = 0; sub < PAIR; ++sub) {
          if (sub && sub >= nsub) break;
          const bool three = REPEAT || (GEO::THREE && sub == 0);
          uint32_t pa[4], pc[2];
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            const float p0 = exp2f(sv[sub][nt][0] - m_new), p1 = exp2f(sv[sub][nt][1] - m_new);
            l_run += p0 + p1;
            const uint32_t hi = pack_bf16(p0, p1);
            const float r0 = p0 - bf16_lo_f(hi), r1 = p1 - bf16_hi_f(hi);
            if (!three) {
              pa[nt * 2] = hi;
              pa[nt * 2 + 1] = pack_bf16(r0, r1);
            } else {
              // the residual has 16 bits at most: the second term is the upper eight, cut off, the third the others
              const float c0 = r0 - upper_half(r0, cut), c1 = r1 - upper_half(r1, cut);
              pa[nt * 2] = REPEAT ? hi & keep : hi;
              pa[nt * 2 + 1] = __byte_perm(__float_as_uint(REPEAT ? c0 : r0), __float_as_uint(REPEAT ? c1 : r1), 0x7632);
              if (WIDE) pc[nt] = __byte_perm(__float_as_uint(c0), __float_as_uint(c1), 0x7632);
            }
          }
          // O += P V
          const int token = (lane & 7) + (((lane >> 3) & 1) << 3);
          const int csel = lane >> 4;
          const uint32_t rowaddr = smem_u32(stage) + sub * GEO::TILE_BYTES + GP_PAGE * GEO::ROW_BYTES + token * GEO::ROW_BYTES;
#pragma unroll
          for (int jd = 0; jd < GEO::DTILES; jd += 2) {
            uint32_t v0, v1, v2, v3;
            ldsm_x4_t(rowaddr + (((jd + csel) ^ (token & 7)) << 4), v0, v1, v2, v3);
            mma_bf16(o[jd], pa[0], pa[1], pa[2], pa[3], v0, v1);
            mma_bf16(o[jd + 1], pa[0], pa[1], pa[2], pa[3], v2, v3);
            if (WIDE && three) {
              mma_bf16(o[jd], pc[0], 0u, pc[1], 0u, v0, v1);
              mma_bf16(o[jd + 1], pc[0], 0u, pc[1], 0u, v2, v3);
            }
          }
        }
        // Boundary unit: fp64 logits of the calibrated summaries against the 16 keys of a candidate page
        if (need_qt && (pg0 + pgl) < Pr - 1) {
          if (!qt_here) {
            if (!wait_bar(qt_full, qt_uses & 1u, s_misc, 5, lim)) { ok = false; break; }
            qt_here = true;
          }
          const long long zoff = ((long long)(unsigned)sd[10]) | ((long long)sd[11] << 32);
#pragma unroll 1
          for (int sub = 0; sub < PAIR; ++sub) {
            if (sub && (sub >= nsub || pg0 + pgl + sub >= Pr - 1)) break;
#pragma unroll
            for (int nt = 0; nt < (WIDE ? 2 : 1); ++nt)
              summary_logits<D>(p, stage + sub * GEO::TILE_BYTES, qt, G, lh, zoff, tok0 + sub * GP_PAGE, nt);
          }
        }
        __syncwarp();
        if (!top_up(it)) { ok = false; break; }            // the stage is free: fetch the next tile into it
      }
      if (!ok) break;
      // (a warp without a candidate tile waits all the same: its next wait is for the phase after this one)
      if (need_qt && !qt_here && !wait_bar(qt_full, qt_uses & 1u, s_misc, 5, lim)) break;

      // ---- a request at its boundary: this warp's share of the unit's summary logits (and the appended row, and the
      // request's counters) is written; the boundary work that may run beside this kernel counts the reports
      if ((flags & 1) && p.report_units) {
        __threadfence();
        __syncwarp();
        if (lane == 0 && !(p.withhold & GP_WITHHOLD_READY)) atomicAdd(p.unit_ready + (size_t)sd[15] * LH + lh, 1);
      }
      // ---- hand the partial result to the merger warp ---------------------------------------------
      l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
      l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
      const int cb = it % NCOMB;
      if (!wait_bar(&comb_empty[cb], ((it / NCOMB) & 1u) ^ 1u, s_misc, 6, lim)) break;
      float* my_comb = comb + (cb * NCW + cw) * comb_w;
      if (head < G) {
        if ((lane & 3) == 0 && !third) { my_comb[row] = m_run; my_comb[8 + row] = l_run; }
        float* my_row = my_comb + 16 + (head + (third ? G : 0)) * D + qc;
#pragma unroll
        for (int jd = 0; jd < GEO::DTILES; ++jd) {
          *reinterpret_cast<float2*>(my_row + jd * 8) =
              make_float2(o[jd][0] + o[jd][2], o[jd][1] + o[jd][3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&comb_full[cb]);
      if (need_qt) {
        ++qt_uses;
        if (lane == 0) mbar_arrive(qt_empty);
      }
      if (lane == 0) mbar_arrive(&slot_empty[sl]);
    }
    cp_async_wait<0>();                  // after an abort copies may still be in flight: let them land
  } else if (warp == 2) {
    // ================================= merger =============================================
    for (uint32_t it = 0;; ++it) {
      const int sl = it % NI;
      if (!wait_bar(&slot_full[sl], (it / NI) & 1u, s_misc, 7, lim)) break;
      const uint8_t* slot = smem + L.off_slots + sl * GEO::SLOT_BYTES;
      const int* sd = reinterpret_cast<const int*>(slot);
      const int npg = sd[3];
      if (npg < 0) break;
      const int bi = sd[0], chunk = sd[4], nchunks = sd[5], rc_i = sd[13], lh = sd[14];
      const int l = sd[17], h = sd[18];
      const int cb = it % NCOMB;
      if (!wait_bar(&comb_full[cb], (it / NCOMB) & 1u, s_misc, 8, lim)) break;
      const float* cbuf = comb + (size_t)cb * NCW * comb_w;
      const size_t out_row0 = (((size_t)l * n_req + bi) * p.Hq + h * G) * D;
      const int PSTRIDE = G * (D + 2);
      float* part = p.partials + ((size_t)lh * n_rc + rc_i) * PSTRIDE;
      // weights of the four warps' rows, lane = 4 head + warp; then a row at a time, a lane owning D / 32 columns of it
      static_assert(NCW == 4, "a quad of lanes per head");
      const int mg = lane >> 2;
      const float mw = mg < G ? cbuf[(lane & 3) * comb_w + mg] : 0.f;
      float M = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, 1));
      M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 2));
      const float wgt = exp2f(mw - M);
      float ls = mg < G ? wgt * cbuf[(lane & 3) * comb_w + 8 + mg] : 1.f;
      ls += __shfl_xor_sync(0xffffffffu, ls, 1);
      ls += __shfl_xor_sync(0xffffffffu, ls, 2);
      if (nchunks > 1 && mg < G && (lane & 3) == 0) { part[mg * (D + 2) + D] = M; part[mg * (D + 2) + D + 1] = ls; }
      const float inv = nchunks == 1 ? 1.f / ls : 1.f;
      constexpr int PER2 = D / 64;                        // float2 pieces of a row per lane
#pragma unroll 2
      for (int g = 0; g < G; ++g) {
        float2 acc[PER2];
#pragma unroll
        for (int e = 0; e < PER2; ++e) acc[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < NCW; ++w) {
          const float ww = __shfl_sync(0xffffffffu, wgt, g * 4 + w);
#pragma unroll
          for (int e = 0; e < PER2; ++e) {
            float2 x = *reinterpret_cast<const float2*>(cbuf + w * comb_w + 16 + g * D + 2 * lane + 64 * e);
            if (GEO::THREE && !WIDE) {
              const float2 y = *reinterpret_cast<const float2*>(cbuf + w * comb_w + 16 + (g + G) * D + 2 * lane + 64 * e);
              x.x += y.x; x.y += y.y;
            }
            acc[e].x += ww * x.x; acc[e].y += ww * x.y;
          }
        }
        const float sc2 = __shfl_sync(0xffffffffu, inv, g * 4);
        float* dst = nchunks == 1 ? out + out_row0 + g * D : part + g * (D + 2);
#pragma unroll
        for (int e = 0; e < PER2; ++e) *reinterpret_cast<float2*>(dst + 2 * lane + 64 * e) = make_float2(acc[e].x * sc2, acc[e].y * sc2);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&comb_empty[cb]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&slot_empty[sl]);
      if (nchunks > 1) {
        // A split unit: whoever adds the last partial of a group of MERGE_FAN chunks merges the group, and whoever adds the
        // last group's the groups (a tree of two levels, whatever the order of arrival).  The counters go back to zero
        // for the next step.
        const int n_grp = (nchunks + MERGE_FAN - 1) / MERGE_FAN, c_grp = chunk / MERGE_FAN * MERGE_FAN;
        const int in_grp = min(MERGE_FAN, nchunks - c_grp);
        float* unit = p.partials + ((size_t)lh * n_rc + rc_i - chunk) * PSTRIDE;
        auto last_of = [&](int* cnt, int n) {
          __threadfence();
          __syncwarp();
          int last = 0;
          if (lane == 0 && atomicAdd(cnt, 1) == n - 1) { *cnt = 0; last = 1; }
          last = __shfl_sync(0xffffffffu, last, 0);
          __threadfence();
          return last != 0;
        };
        int* cnt = p.merge_cnt + ((size_t)rc_i - chunk) * LH + (size_t)lh * nchunks;       // the unit's: one per chunk
        const bool tree = n_grp > 1;
        bool go = last_of(cnt + c_grp, in_grp), into = tree;
#pragma unroll 1
        while (go) {
          // One call of the merge: three copies, unrolled, were 37 KB of the kernel's 130, and these kernels' few units wait for instructions
          // (gp_attn_kernel<128, true, WHOLE_STEP, false> 102 KB now; us a pass: four requests, 16 steps, 259 / 256; one layer x 64, 16 steps,
          // 1039 / 1026; long contexts, 16 steps, 5080 / 5039).  Its first rows asked for before the maxima: spills at 80 registers, 4 % of a layer.
          const bool groups = tree && !into;
          const int n = groups ? n_grp : tree ? in_grp : nchunks;
          if (!into || n > 1)
            merge_unit<D>(unit + (into ? (size_t)c_grp * PSTRIDE : 0), groups ? (size_t)MERGE_FAN * PSTRIDE : PSTRIDE, n, G, out + out_row0, into);
          go = into && last_of(cnt + 1, n_grp);
          into = false;
        }
      }
    }
  } else {
    // ================================= summaries ==========================================
    const int w = warp >> 1;
    uint32_t qt_uses = 0;
    for (uint32_t it = 0;; ++it) {
      const int sl = it % NI;
      if (!wait_bar(&slot_full[sl], (it / NI) & 1u, s_misc, 9, lim)) break;
      uint8_t* slot = smem + L.off_slots + sl * GEO::SLOT_BYTES;
      const int* sd = reinterpret_cast<const int*>(slot);
      if (sd[3] < 0) break;
      const int bi = sd[0], r = sd[1], flags = sd[8], par = sd[12];
      const bool owner = sd[4] == 0;                       // this item writes the unit's new summaries
      const bool need_qt = (flags & 1) && sd[2] < sd[9] - 1;
      if (NORM || owner || need_qt) {
        if (need_qt && !wait_bar(qt_empty, (qt_uses & 1u) ^ 1u, s_misc, 10, lim)) break;
        const int l = sd[17], h = sd[18];
        auto rows_there = [&]() { return !LAYER || wait_bar(&slot_rows[sl], (it / NI) & 1u, s_misc, 13, lim); };
        if (!summary_rows<D, ROPE, NORM>(p, nm, slot + GEO::SLOT_DESC, rows_there, &slot_norm[sl], w, G, l, h, r, bi, par, (flags & 2) != 0, owner,
                                         need_qt ? qt : nullptr)) break;
        __syncwarp();
        if (need_qt) {
          ++qt_uses;
          if (lane == 0) mbar_arrive(qt_full);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&slot_empty[sl]);
    }
  }
  __syncthreads();
  // a wait of this CTA gave up (whichever warp it was, and however late): say so, with the code of the wait
  if (tid == 0 && s_misc[0]) atomicOr(p.err, GP_E_SPIN | (1 << (7 + s_misc[1])));
}

}  // namespace

size_t gp_attention_smem(int d, int G) { return d == 128 ? make_lay<128>(G).total : make_lay<64>(G).total; }
int gp_attention_ctas_per_sm(int d) { (void)d; return 2; }

typedef void (*AttnKernel)(const GpDev, int, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, float*, int, int, int, int,
                           const GpNorm);
template <int D, bool WIDE> static AttnKernel attn_kernel_d(bool rope, int mode) {
  return mode == WHOLE_STEP ? (rope ? gp_attn_kernel<D, true, WHOLE_STEP, WIDE> : gp_attn_kernel<D, false, WHOLE_STEP, WIDE>)
         : mode == ONE_LAYER ? (rope ? gp_attn_kernel<D, true, ONE_LAYER, WIDE> : gp_attn_kernel<D, false, ONE_LAYER, WIDE>)
                             : (rope ? gp_attn_kernel<D, true, ONE_LAYER_NORM, WIDE> : gp_attn_kernel<D, false, ONE_LAYER_NORM, WIDE>);
}
static AttnKernel attn_kernel_of(const GpDev& p, int mode) {
  const bool rope = p.rope_theta != 0.0;
  if (p.d == 128) return p.G == 8 ? attn_kernel_d<128, true>(rope, mode) : attn_kernel_d<128, false>(rope, mode);
  return p.G == 8 ? attn_kernel_d<64, true>(rope, mode) : attn_kernel_d<64, false>(rope, mode);
}

void gp_attention_setup(const GpDev& p) {           // once per pool: opt into the kernels' shared memory
  for (int mode = WHOLE_STEP; mode <= ONE_LAYER_NORM; ++mode)
    cudaFuncSetAttribute(attn_kernel_of(p, mode), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gp_attention_smem(p.d, p.G));
}

void gp_launch_attention(const GpDev& p, int n_req, const void* q, const void* k, const void* v, float* out, int grid, cudaStream_t s,
                         bool pdl, int lh0, int lh_n, int adv_lh, bool layer, bool planned, const GpNorm& nm) {
  const int mode = !layer ? WHOLE_STEP : nm.wq ? ONE_LAYER_NORM : ONE_LAYER;
  gp_launch(attn_kernel_of(p, mode), grid, NTHREADS, gp_attention_smem(p.d, p.G), s, pdl, p, n_req,
            static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v), out, lh0,
            lh_n, adv_lh, planned ? 1 : 0, nm);
}
