// gp_attention_noalloc: GQA decode attention over plain (un-paged) K/V that needs no memory beyond what the
// caller passes in.  The split-KV partial results, which the pool's attention kernel keeps in the pool blob,
// live here in a fixed array inside the library image.
//
// Who needs this: callers that are not allowed to allocate device memory when they call us.  Examples are a
// serving process that commits all of the GPU's memory to its KV pool at start-up (a later cudaMalloc would
// fail, and even a successful one synchronises the device in the middle of a decode loop), and hosts that run
// this library as a plug-in under a rule that library code never calls the allocator.  Such a caller can hand
// us inputs and outputs it already owns, but has nowhere to get scratch from.
//
// The price: every GPU whose context loads this library carries the array (8.5 MB) until the process exits,
// the problem size is capped (GP_NOALLOC_MAX_ROWS query-head rows), and all calls share the one array, so two
// calls that overlap on the GPU (different streams) corrupt each other's partial results.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/growpage.h"
#include "gp_dev.cuh"

namespace {

constexpr int NA_MAX_ROWS = GP_NOALLOC_MAX_ROWS;
constexpr int NA_MAX_D = 128;
constexpr int NA_STRIDE = NA_MAX_D + 2;        // accumulator row, then running max and sum
constexpr int NA_MAX_DEVICES = 64;
constexpr int NA_ROOM = NA_MAX_ROWS * GP_NOALLOC_SPLITS;      // partial rows the array holds
constexpr int NA_WARPS = 4;
constexpr int NA_THREADS = NA_WARPS * 32;
constexpr int NA_STAGES = 2;                   // tiles a warp has in flight
constexpr int NA_TILE_BYTES = 8192;            // K and V of a tile: 16 tokens of 128 elements, 32 of 64
constexpr int NA_SMEM = NA_WARPS * NA_STAGES * NA_TILE_BYTES + 128;
constexpr int NA_CTAS = 888;                   // thread blocks a launch is cut into where there is that much work
constexpr int NA_MIN_SPLIT = 256;              // tokens of the longest request below which splits are not cut further

// Scratch of the entry point.  In host code this name is only a handle for the runtime's symbol calls; the
// device address is fetched once per device with cudaGetSymbolAddress (below) and passed to the kernels.
static __device__ __align__(256) float gp_noalloc_scratch[(size_t)NA_ROOM * NA_STRIDE];

static float* g_scratch_addr[NA_MAX_DEVICES];  // device address of the array, per device, once known

// 16-byte asynchronous copy that reads `bytes` (0 or 16) and fills the rest with zeros
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst_smem, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src), "r"(bytes) : "memory");
}
// transpose of an 8 x 8 matrix of 16-bit elements spread over the warp (row lane / 4, columns 2 (lane % 4), + 1)
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
  uint32_t y;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// The tokens [t0, t1) of one (request, KV head) with plain loads of single elements and fp32 arithmetic throughout.
// Writes the split's partial results.  `smem`: NA_PLAIN_FLOATS floats.  Bound by the latency of a warp's chain of loads, sums over
// the warp and exponentials, so by the warps an SM holds.  AHEAD: the next token's elements are on their way while one is worked on,
// which pays where they are few (twelve in the tensor-core kernel: 507 us for 64 requests of 60 to 4000 tokens, groups of 4, d = 128,
// against 805) and costs where they are many (twenty-four in the plain kernel: 664 us against 507, both with the width a variable).
constexpr int NA_PLAIN_FLOATS = 8 * NA_MAX_D + NA_WARPS * 8 * NA_STRIDE;
template <int D, bool AHEAD>
__device__ __forceinline__ void na_plain_tokens(const __nv_bfloat16* __restrict__ qrow0, const __nv_bfloat16* __restrict__ kbase,
                                                const __nv_bfloat16* __restrict__ vbase, int G, int t0, int t1, float* smem,
                                                float* __restrict__ part, size_t row_stride) {
  constexpr int PER = D / 32;                                              // elements of a row per lane
  float* s_q = smem;                                                       // [8][NA_MAX_D]
  float (*s_part)[8][NA_STRIDE] = reinterpret_cast<float (*)[8][NA_STRIDE]>(smem + 8 * NA_MAX_D);     // [warps]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  __syncthreads();                                                         // whatever the memory held before is done with
  for (int i = tid; i < G * D; i += NA_THREADS) s_q[(i / D) * NA_MAX_D + i % D] = __bfloat162float(qrow0[i]);
  __syncthreads();
  const float scale = 1.4426950408889634f * rsqrtf((float)D);
  float m[8], l[8], acc[8][PER];
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    m[g] = -INFINITY; l[g] = 0.f;
#pragma unroll
    for (int e = 0; e < PER; ++e) acc[g][e] = 0.f;
  }
  __nv_bfloat16 kn[PER], vn[PER];                         // AHEAD: as loaded, converted where they are used, so that nothing waits for them before
  auto load = [&](int t) {
#pragma unroll
    for (int e = 0; e < PER; ++e) { kn[e] = kbase[(size_t)t * D + lane + 32 * e]; vn[e] = vbase[(size_t)t * D + lane + 32 * e]; }
  };
  if (AHEAD && t0 + warp < t1) load(t0 + warp);
  for (int t = t0 + warp; t < t1; t += NA_WARPS) {
    if (!AHEAD) load(t);
    float kv[PER], vv[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) { kv[e] = __bfloat162float(kn[e]); vv[e] = __bfloat162float(vn[e]); }
    if (AHEAD) load(min(t + NA_WARPS, t1 - 1));
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      if (g < G) {
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < PER; ++e) s += s_q[g * NA_MAX_D + lane + 32 * e] * kv[e];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s *= scale;
        const float mn = fmaxf(m[g], s);
        const float corr = exp2f(m[g] - mn), p = exp2f(s - mn);
        l[g] = l[g] * corr + p;
#pragma unroll
        for (int e = 0; e < PER; ++e) acc[g][e] = acc[g][e] * corr + p * vv[e];
        m[g] = mn;
      }
    }
  }
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    if (g < G) {
#pragma unroll
      for (int e = 0; e < PER; ++e) s_part[warp][g][lane + 32 * e] = acc[g][e];
      if (lane == 0) { s_part[warp][g][NA_MAX_D] = m[g]; s_part[warp][g][NA_MAX_D + 1] = l[g]; }
    }
  }
  __syncthreads();
  for (int i = tid; i < G * D; i += NA_THREADS) {
    const int g = i / D, c = i % D;
    float M = -INFINITY;
    for (int w = 0; w < NA_WARPS; ++w) M = fmaxf(M, s_part[w][g][NA_MAX_D]);
    float a = 0.f, ls = 0.f;
    for (int w = 0; w < NA_WARPS; ++w) {
      const float wt = (M == -INFINITY) ? 0.f : exp2f(s_part[w][g][NA_MAX_D] - M);
      a += wt * s_part[w][g][c];
      ls += wt * s_part[w][g][NA_MAX_D + 1];
    }
    float* dst = part + g * row_stride;
    dst[c] = a;
    if (c == 0) { dst[NA_MAX_D] = M; dst[NA_MAX_D + 1] = ls; }
  }
}
// out of line, for a split whose tensor-core result is not finite (below)
template <int D>
__device__ __noinline__ void na_split_plain(const __nv_bfloat16* qrow0, const __nv_bfloat16* kbase, const __nv_bfloat16* vbase, int G,
                                            int t0, int t1, float* smem, float* part, size_t row_stride) {
  na_plain_tokens<D, true>(qrow0, kbase, vbase, G, t0, t1, smem, part, row_stride);
}

// Keys or values whose addresses are not 16-byte aligned.  A kernel of its own: it needs a third of the tensor-core kernel's shared
// memory, so that an SM holds twice the warps (inside that kernel: 1120 us for 64 requests of 60 to 4000 tokens, 8 KV heads, groups
// of 4, d = 128, against 466).
template <int D>
__global__ void __launch_bounds__(NA_THREADS)
na_plain_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                const int* __restrict__ lens, int Hq, int Hkv, int max_len, float* __restrict__ scratch) {
  __shared__ float smem[NA_PLAIN_FLOATS];
  const int split = blockIdx.x, n_split = gridDim.x, unit = blockIdx.y;
  const int req = unit / Hkv, h = unit % Hkv, G = Hq / Hkv;
  gp_pdl_launch_dependents();                           // the merge waits for this grid's end before it reads
  const int len = max(0, min(lens[req], max_len));
  const int chunk = (int)(((long long)len + n_split - 1) / n_split);
  const int t0 = min(len, split * chunk), t1 = min(len, t0 + chunk);
  const size_t at = ((size_t)req * Hkv + h) * (size_t)max_len * D;
  na_plain_tokens<D, false>(q + ((size_t)req * Hq + h * G) * D, k + at, v + at, G, t0, t1, smem,
                            scratch + (((size_t)req * Hq + h * G) * n_split + split) * NA_STRIDE, (size_t)n_split * NA_STRIDE);
}

// One thread block per (split, request, KV head): the split's share of the tokens, all G query heads of the group.
//
// What bounds it: HBM, once the contractions run on the tensor cores.  Each warp takes every NA_WARPS-th tile of the
// split and fetches its own tiles with 16-byte asynchronous copies into a private ring, so nothing in the loop waits for
// another warp.  The tokens are the rows of the MMAs, so the eight columns of an m16n8k16 hold the (up to eight) query
// heads of the group and nothing is spent on padding a group to sixteen rows:
//   S^T [16 tokens x 8 heads] = K (A operand, ldmatrix) x Q^T (B operand, in registers for the whole split)
//   O^T [16 of d x 8 heads]  += V^T (A operand, ldmatrix.trans) x P^T (B operand: S^T's fragments, transposed 8 x 8)
// Queries, keys and values are bf16 as the caller gave them, so their products are exact.  The weights p are fp32 and
// are carried as three bf16 terms, p = hi + mid + lo, which hold all their 24 bits; and no sum grows inside the tensor
// core over a long chain: the logits are added up in fp32 registers from MMAs of 16 products each, and so is O from
// one tile to the next.
// An infinite value would meet a zero mid or lo term (inf x 0), so a split whose result is not finite is done over
// in plain arithmetic (an infinite value in every split, on the sizes below: 507 us; 491 before there was a first pass).
// Measured, both kernels: 64 requests of 60 to 4000 tokens, 8 KV heads, groups of 4, d = 128 (532 MB): 464 us before (one
// element per load, fp32 FMAs and shuffles), 96 us now, 5.6 TB/s; 32 requests of 8 to 1678, 4 KV heads, groups of 8: 114 us
// before, 25 now.  Error against 64 bits 1.3e-7 to 1.9e-7 (before: 1.4e-7 to 2.0e-7 on the same inputs).  Four warps
// with two stages, three thread blocks to an SM; three stages and two blocks: 109 us, two warps: 99 to 114 us.
template <int D>
__global__ void __launch_bounds__(NA_THREADS)
na_partial_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                  const __nv_bfloat16* __restrict__ v, const int* __restrict__ lens, int Hq, int Hkv, int max_len,
                  float* __restrict__ scratch) {
  constexpr int ROW = D * 2;                            // bytes of a token's key or value
  constexpr int CH = D / 8;                             // 16-byte pieces of one
  constexpr int NT = NA_TILE_BYTES / (2 * 16 * ROW);    // groups of 16 tokens in a tile
  constexpr int TOK = NT * 16;
  constexpr int KSTEPS = D / 16;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int split = blockIdx.x, n_split = gridDim.x, unit = blockIdx.y;
  const int req = unit / Hkv, h = unit % Hkv, G = Hq / Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  gp_pdl_launch_dependents();                           // the merge waits for this grid's end before it reads
  const int len = max(0, min(lens[req], max_len));
  const int chunk = ((len + n_split - 1) / n_split + 15) / 16 * 16;
  const int t0 = min(len, split * chunk), t1 = min(len, t0 + chunk);
  const __nv_bfloat16* qrow0 = q + ((size_t)req * Hq + h * G) * D;
  const __nv_bfloat16* kbase = k + ((size_t)req * Hkv + h) * (size_t)max_len * D;
  const __nv_bfloat16* vbase = v + ((size_t)req * Hkv + h) * (size_t)max_len * D;
  const size_t row_stride = (size_t)n_split * NA_STRIDE;
  float* part = scratch + (((size_t)req * Hq + h * G) * n_split + split) * NA_STRIDE;      // row g: + g * row_stride

  const int n_tiles = (t1 - t0 + TOK - 1) / TOK;
  uint8_t* ring = smem + warp * NA_STAGES * NA_TILE_BYTES;
  auto fetch = [&](int i) {                             // this warp's i-th tile, tile warp + i NA_WARPS of the split
    const int tile = warp + i * NA_WARPS;
    if (tile < n_tiles) {
      const uint32_t dst = smem_u32(ring + (i % NA_STAGES) * NA_TILE_BYTES);
      const int tb = t0 + tile * TOK;
#pragma unroll
      for (int c = 0; c < NA_TILE_BYTES / 512; ++c) {
        const int piece = (c * 32 + lane) % (TOK * CH);
        const bool isv = c * 32 >= TOK * CH;
        const int t = piece / CH, pc = piece % CH;
        const int tt = min(tb + t, t1 - 1);             // rows past the split's end are zeros; their address stays inside
        cp_async16_or_zero(dst + (isv ? TOK * ROW : 0) + t * ROW + ((pc ^ (t & 7)) << 4),
                           reinterpret_cast<const uint8_t*>((isv ? vbase : kbase) + (size_t)tt * D) + pc * 16, tb + t < t1 ? 16 : 0);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < NA_STAGES - 1; ++i) fetch(i);

  // B fragments of Q^T: column n = lane / 4 is head n of the group, rows 2 (lane % 4), + 1 (and + 8)
  uint32_t qb[KSTEPS][2];
  {
    const int g = lane >> 2;
    const unsigned short* qr = reinterpret_cast<const unsigned short*>(qrow0 + (g < G ? g : 0) * D);
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int c = kk * 16 + half * 8 + (lane & 3) * 2;
        qb[kk][half] = g < G ? (uint32_t)qr[c] | ((uint32_t)qr[c + 1] << 16) : 0u;
      }
  }
  const float scale = 1.4426950408889634f * rsqrtf((float)D);
  float o[KSTEPS][4];                                   // O^T: rows lane / 4 (+ 8) of block jd of d, heads 2 (lane % 4), + 1
#pragma unroll
  for (int i = 0; i < KSTEPS; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;

  const int mi = lane >> 3, mr = lane & 7;              // ldmatrix: matrix and row this lane addresses
  for (int i = 0; warp + i * NA_WARPS < n_tiles; ++i) {
    fetch(i + NA_STAGES - 1);
    cp_async_wait<NA_STAGES - 1>();
    __syncwarp();
    const uint32_t kt = smem_u32(ring + (i % NA_STAGES) * NA_TILE_BYTES), vt = kt + TOK * ROW;
    const int left = t1 - (t0 + (warp + i * NA_WARPS) * TOK);       // valid tokens of the tile (TOK or more: all)
    float s[NT][4];
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
      const int t = nt * 16 + mr + (mi & 1) * 8;
      const uint32_t row = kt + t * ROW;
#pragma unroll
      for (int kk = 0; kk < KSTEPS; ++kk) {
        uint32_t a0, a1, a2, a3;
        ldsm_x4(row + (((2 * kk + (mi >> 1)) ^ (t & 7)) << 4), a0, a1, a2, a3);
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(c, a0, a1, a2, a3, qb[kk][0], qb[kk][1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) s[nt][e] += c[e];
      }
      const int tr = nt * 16 + (lane >> 2);
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nt][e] = tr + (e >> 1) * 8 < left ? s[nt][e] * scale : -INFINITY;
      mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][2]));
      mx1 = fmaxf(mx1, fmaxf(s[nt][1], s[nt][3]));
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
    }
    mx0 = fmaxf(m0, mx0); mx1 = fmaxf(m1, mx1);
    const float c0 = exp2f(m0 - mx0), c1 = exp2f(m1 - mx1);
    m0 = mx0; m1 = mx1;
    if (__any_sync(0xffffffffu, c0 != 1.f || c1 != 1.f)) {
      l0 *= c0; l1 *= c1;
#pragma unroll
      for (int jd = 0; jd < KSTEPS; ++jd) { o[jd][0] *= c0; o[jd][1] *= c1; o[jd][2] *= c0; o[jd][3] *= c1; }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      uint32_t hi[2], mid[2], lo[2];                    // B fragments of P^T: tokens 0..7 and 8..15 of the group
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const float p0 = exp2f(s[nt][2 * half] - m0), p1 = exp2f(s[nt][2 * half + 1] - m1);
        l0 += p0; l1 += p1;
        const uint32_t w0 = pack_bf16(p0, p1);
        const float r0 = p0 - bf16_lo_f(w0), r1 = p1 - bf16_hi_f(w0);
        const uint32_t w1 = pack_bf16(r0, r1);
        const uint32_t w2 = pack_bf16(r0 - bf16_lo_f(w1), r1 - bf16_hi_f(w1));
        hi[half] = transpose8x8(w0); mid[half] = transpose8x8(w1); lo[half] = transpose8x8(w2);
      }
      const int t = nt * 16 + mr + (mi >> 1) * 8;
      const uint32_t row = vt + t * ROW;
#pragma unroll
      for (int jd = 0; jd < KSTEPS; ++jd) {
        uint32_t a0, a1, a2, a3;
        ldsm_x4_t(row + (((2 * jd + (mi & 1)) ^ (t & 7)) << 4), a0, a1, a2, a3);
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(c, a0, a1, a2, a3, lo[0], lo[1]);
        mma_bf16(c, a0, a1, a2, a3, mid[0], mid[1]);
        mma_bf16(c, a0, a1, a2, a3, hi[0], hi[1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[jd][e] += c[e];
      }
    }
    __syncwarp();                                       // the tile has been read: its stage may be fetched into
  }
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    l0 += __shfl_xor_sync(0xffffffffu, l0, off);
    l1 += __shfl_xor_sync(0xffffffffu, l1, off);
  }
  bool bad = false;
#pragma unroll
  for (int jd = 0; jd < KSTEPS; ++jd)
#pragma unroll
    for (int e = 0; e < 4; ++e) bad |= !(fabsf(o[jd][e]) < INFINITY) && (lane & 3) * 2 + (e & 1) < G;
  cp_async_wait<0>();
  if (__syncthreads_or(bad)) {
    na_split_plain<D>(qrow0, kbase, vbase, G, t0, t1, reinterpret_cast<float*>(smem), part, row_stride);
    return;
  }
  // merge the warps; every slot of this (row, split) is rewritten on every call, so nothing stale survives
  float (*s_part)[8][NA_STRIDE] = reinterpret_cast<float (*)[8][NA_STRIDE]>(smem);
  {
    const int g0 = (lane & 3) * 2, r0 = lane >> 2;
#pragma unroll
    for (int jd = 0; jd < KSTEPS; ++jd)
#pragma unroll
      for (int e = 0; e < 4; ++e) s_part[warp][g0 + (e & 1)][jd * 16 + r0 + (e >> 1) * 8] = o[jd][e];
    if (r0 == 0) {
      s_part[warp][g0][NA_MAX_D] = m0; s_part[warp][g0][NA_MAX_D + 1] = l0;
      s_part[warp][g0 + 1][NA_MAX_D] = m1; s_part[warp][g0 + 1][NA_MAX_D + 1] = l1;
    }
  }
  __syncthreads();
  for (int i = tid; i < G * D; i += NA_THREADS) {
    const int g = i / D, c = i % D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < NA_WARPS; ++w) M = fmaxf(M, s_part[w][g][NA_MAX_D]);
    float a = 0.f, ls = 0.f;
#pragma unroll
    for (int w = 0; w < NA_WARPS; ++w) {
      const float wt = (M == -INFINITY) ? 0.f : exp2f(s_part[w][g][NA_MAX_D] - M);
      a += wt * s_part[w][g][c];
      ls += wt * s_part[w][g][NA_MAX_D + 1];
    }
    float* dst = part + g * row_stride;
    dst[c] = a;
    if (c == 0) { dst[NA_MAX_D] = M; dst[NA_MAX_D + 1] = ls; }
  }
}

// One thread block per query-head row: merge the splits.  The weights of up to 256 splits at a time are computed once
// per block and shared; a thread owns a column.
__global__ void __launch_bounds__(NA_MAX_D)
na_merge_kernel(const float* __restrict__ scratch, int n_split, float* __restrict__ out) {
  __shared__ float s_w[256], s_l[256], s_red[NA_MAX_D / 32];
  const int row = blockIdx.x, d = blockDim.x, c = threadIdx.x;
  const float* base = scratch + (size_t)row * n_split * NA_STRIDE;
  gp_pdl_wait();
  float M = -INFINITY;
  for (int s = c; s < n_split; s += d) M = fmaxf(M, __ldcg(base + (size_t)s * NA_STRIDE + NA_MAX_D));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
  if ((c & 31) == 0) s_red[c >> 5] = M;
  __syncthreads();
  for (int w = 0; w < d / 32; ++w) M = fmaxf(M, s_red[w]);
  float a = 0.f, ls = 0.f;
  for (int s0 = 0; s0 < n_split; s0 += 256) {
    const int n = min(256, n_split - s0);
    __syncthreads();
    for (int s = c; s < n; s += d) {
      const float2 ml = __ldcg(reinterpret_cast<const float2*>(base + (size_t)(s0 + s) * NA_STRIDE + NA_MAX_D));
      s_w[s] = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - M);
      s_l[s] = ml.y;
    }
    __syncthreads();
#pragma unroll 8
    for (int s = 0; s < n; ++s) {
      a += s_w[s] * __ldcg(base + (size_t)(s0 + s) * NA_STRIDE + c);
      ls += s_w[s] * s_l[s];
    }
  }
  out[(size_t)row * d + c] = ls > 0.f ? a / ls : 0.f;       // a request without tokens: a row of zeros
}

}  // namespace

extern "C" int gp_attention_noalloc(const void* q, const void* k, const void* v, const int32_t* lens, int32_t n_req,
                                    int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim, int32_t max_len,
                                    void* out, void* stream) {
  if (!q || !k || !v || !lens || !out) return GP_ERR_INVALID;
  if (n_req < 1 || n_q_heads < 1 || n_kv_heads < 1 || max_len < 1) return GP_ERR_INVALID;
  if (n_q_heads % n_kv_heads) return GP_ERR_INVALID;
  const int G = n_q_heads / n_kv_heads;
  if (G > 8 || (head_dim != 64 && head_dim != 128)) return GP_ERR_INVALID;
  if ((long long)n_req * n_q_heads > NA_MAX_ROWS) return GP_ERR_TOO_LARGE;   // the fixed array has no room
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return GP_ERR_CUDA;
  auto partial = head_dim == 128 ? na_partial_kernel<128> : na_partial_kernel<64>;
  if (!g_scratch_addr[dev]) {
    // First call on this device: ask the runtime where the array lives here, and opt the kernels into their shared
    // memory.  No allocation happens; the array came with the library image.
    float* ptr = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), gp_noalloc_scratch) != cudaSuccess || !ptr) return GP_ERR_CUDA;
    if (cudaFuncSetAttribute(na_partial_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, NA_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(na_partial_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, NA_SMEM) != cudaSuccess)
      return GP_ERR_CUDA;
    g_scratch_addr[dev] = ptr;
  }
  float* scratch = g_scratch_addr[dev];
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // Splits per (request, KV head): enough for NA_CTAS thread blocks, two rounds of what fits the GPU, no shorter than
  // NA_MIN_SPLIT tokens of the longest request, and no more than the array holds.  (More and shorter ones cost a thread
  // block's start-up each and more rows to merge: with 4096 blocks or splits of 64 tokens 25 requests of 4 to 479 tokens take
  // 21 us against 16, while 64 requests of up to 4000 tokens, which need no splitting, lie between 94 and 98 either way.)
  const int units = n_req * n_kv_heads;
  long long splits = (NA_CTAS + units - 1) / units;
  const long long most = ((long long)max_len + NA_MIN_SPLIT - 1) / NA_MIN_SPLIT, room = NA_ROOM / (n_req * n_q_heads);
  if (splits > most) splits = most;
  if (splits > room) splits = room;
  const __nv_bfloat16 *qp = static_cast<const __nv_bfloat16*>(q), *kp = static_cast<const __nv_bfloat16*>(k),
                      *vp = static_cast<const __nv_bfloat16*>(v);
  if ((((uintptr_t)k | (uintptr_t)v) & 15) == 0) {                    // the tiles' copies move 16 bytes
    partial<<<dim3((unsigned)splits, (unsigned)units), NA_THREADS, NA_SMEM, s>>>(qp, kp, vp, lens, n_q_heads, n_kv_heads, max_len, scratch);
  } else {
    // a token costs a warp here what a tile of 16 costs there, so short splits pay: no fewer than the array holds at any size (with the
    // rule above 128 requests, one of 16 000 tokens and the others of 200, 8 KV heads, groups of 2: 3860 us; now 477)
    if (splits < GP_NOALLOC_SPLITS) splits = GP_NOALLOC_SPLITS;
    auto plain = head_dim == 128 ? na_plain_kernel<128> : na_plain_kernel<64>;
    plain<<<dim3((unsigned)splits, (unsigned)units), NA_THREADS, 0, s>>>(qp, kp, vp, lens, n_q_heads, n_kv_heads, max_len, scratch);
  }
  if (cudaGetLastError() != cudaSuccess) return GP_ERR_CUDA;
  return gp_launch(na_merge_kernel, n_req * n_q_heads, head_dim, 0, s, true, static_cast<const float*>(scratch), (int)splits,
                   static_cast<float*>(out)) == cudaSuccess ? GP_OK : GP_ERR_CUDA;
}
