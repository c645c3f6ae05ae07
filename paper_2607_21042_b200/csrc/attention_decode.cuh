// Decode attention of middle batches (two to ten (row, head) pairs per SM): work split by 32-token units over one CTA per
// SM, Q K^T and P V on the warp-level tensor pipe (Section I: the decode engine's attention kernels).
//
// What bounds the kernels it replaces there: instructions and waves, not HBM.  Folding a page of 64 tokens on the CUDA
// cores takes a warp about 750 instructions (half of them unpack bf16), straight-line code of 11 KB that is fetched cold
// in every launch, and one CTA per pair leaves a nearly empty last wave (320 pairs on 296 resident CTAs: 15 us at 16
// rows of 530 tokens where the bytes need 7).
//
// Here a unit of 32 tokens takes about 110 instructions in one rolled loop.  The query is the 8-wide operand of the MMA:
// its 64 fp32 values are split into three bf16 parts (24 bits, nothing lost) in columns 0-2, so that K, the 16-row
// operand, is multiplied by q exactly as in fp32; P is split the same way for P V, whose 16-row operand is V transposed
// on the way out of shared memory (ldmatrix).  K and V rows come in as 4 KB tensor copies with the 128-byte swizzle,
// two units ahead per warp.
//
// Work split.  The pairs are dealt to the CTAs (longest rows first), the units of a CTA's pairs laid end to end and cut
// into one contiguous range per warp: ranges are equal to within a unit whatever the context lengths are.  A pair that
// lies inside one range is finished by that warp; the parts of a pair cut over several warps meet in shared memory, in
// unit order.  No global scratch, no atomics; the result does not depend on timing.  Clusters of 2, 4 or 8 CTAs dealing
// with a pair together balance better but lose 3 to 5 us to the barrier and the remote reads at the end.
// Measured per step: 16 rows at 530 tokens 0.951 -> 0.870 ms, at 1530 1.316 -> 1.171; 37 rows at 610 1.436 -> 1.359; 64 rows
// at 730 1.835 -> 1.792.  At 128 rows the streaming kernel's dynamic order is ahead again (2.747 against 2.792).
#pragma once
#include "attention.cuh"
#include "gemm_pw.cuh"

namespace ttsgpt {

constexpr int kAdWarps = 12;
constexpr int kAdUnit = 32;                         // tokens per unit
constexpr int kAdHalf = kAdUnit * kHeadDim * 2;     // K or V of a unit: 4 KB
constexpr int kAdStages = 2;                        // units in flight per warp
constexpr int kAdMaxPairs = 64;                     // pairs of one CTA
constexpr int kAdPitchP = 80;                       // bytes per row of a warp's P buffer (8 rows of 32 bf16): conflict-free fragment loads

struct AdArgs {
  AttnArgs at;
  int layer_row;      // first row of the layer in the pool's tensor
  int n_pair;
};

// per-CTA shared memory, behind the stages
struct AdShared {
  float q[kAdMaxPairs][kHeadDim];
  float part[kAdWarps][2][kHeadDim + 2];           // partial results of pairs cut over warps: (begun before the warp's range, going on behind it)
  unsigned char p[kAdWarps][8 * kAdPitchP];        // rows 0-2: the three parts of P, the rest stays zero
  uint64_t bar[kAdWarps][kAdStages];
  int first_unit[kAdMaxPairs + 1];                 // running unit counts of the CTA's pairs
  int row[kAdMaxPairs], n_tok[kAdMaxPairs];
  const int *pt[kAdMaxPairs];                      // the pair's page list
  int dead;                                        // some warp's wait has expired: parts are not merged
};
inline size_t attention_decode_smem_bytes() { return (size_t)kAdWarps * kAdStages * 2 * kAdHalf + sizeof(AdShared) + 1024; }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ad_copy(const CUtensorMap *map, int row, unsigned char *dst, uint64_t *bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_u32(dst)), "l"(map), "r"(0), "r"(row), "r"(smem_u32(bar)) : "memory");
}
// part k of x in three bf16 parts: bf16(x), bf16 of what that leaves, bf16 of what those leave
__device__ __forceinline__ void split3(float x, float &a, float &b, float &c) {
  a = __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);   // truncation keeps the rest exact and of the same sign
  const float r = x - a;
  b = __uint_as_float(__float_as_uint(r) & 0xFFFF0000u);
  c = r - b;
}
__device__ __forceinline__ uint32_t high_halves(float lo, float hi) { return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632); }

__global__ void __launch_bounds__(kAdWarps * 32, 1) attention_decode_kernel(const __grid_constant__ CUtensorMap kv_map, const AdArgs ad) {
  extern __shared__ __align__(16) unsigned char ad_smem_raw[];
  const AttnArgs &a = ad.at;
  unsigned char *stages = ad_smem_raw + ((1024u - (smem_u32(ad_smem_raw) & 1023u)) & 1023u);
  AdShared &sh = *reinterpret_cast<AdShared *>(stages + (size_t)kAdWarps * kAdStages * 2 * kAdHalf);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int cid = blockIdx.x, n_cta = gridDim.x;
  const int P = (ad.n_pair - cid + n_cta - 1) / n_cta;   // pair i of this CTA: cid + i * n_cta
  trace_mark(a.trace, a.trace_slot, 0);

  // ---- the CTA's unit list (row, page and order tables are final before the step's first kernel starts) ----
  if (threadIdx.x < kAdMaxPairs) {
    int n = 0;
    if ((int)threadIdx.x < P) {
      const int slot = (cid + (int)threadIdx.x * n_cta) / a.H;
      const int4 d = a.slots ? a.slots[slot] : make_int4(slot, a.row_pos[slot] + 1, a.row_stream[slot], 0);
      n = d.y;
      sh.row[threadIdx.x] = d.x;
      sh.pt[threadIdx.x] = a.slots ? a.slot_pages + (size_t)slot * a.pps : a.page_table + (size_t)d.z * a.pps;
    }
    sh.n_tok[threadIdx.x] = n;
  }
  if (lane < kAdStages) mbar_init(&sh.bar[warp][lane], 1);
  if (threadIdx.x == 0) sh.dead = 0;
  for (int i = lane; i < 8 * kAdPitchP / 4; i += 32) reinterpret_cast<uint32_t *>(sh.p[warp])[i] = 0u;
  __syncthreads();
  if (warp == 0) {   // running unit counts, two pairs per lane
    const int u0 = (sh.n_tok[2 * lane] + kAdUnit - 1) / kAdUnit, u1 = (sh.n_tok[2 * lane + 1] + kAdUnit - 1) / kAdUnit;
    int incl = u0 + u1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += n;
    }
    sh.first_unit[2 * lane] = incl - u0 - u1;
    sh.first_unit[2 * lane + 1] = incl - u1;
    if (lane == 31) sh.first_unit[kAdMaxPairs] = incl;
  }
  __syncthreads();
  const int total = sh.first_unit[kAdMaxPairs];
  const int u_begin = total * warp / kAdWarps, u_end = total * (warp + 1) / kAdWarps;

  // what a unit is: lane l holds it for unit base + l of the warp's range (page-table reads of 32 units at a time)
  int my_row_k = 0, my_pair = 0, my_left = 0;   // tensor row of its K half; pair; tokens of the pair from this unit on
  auto describe = [&](int base) {
    const int u = base + lane;
    if (u < u_end) {
      int lo = 0, hi = P - 1;                   // last pair whose first unit is <= u
      while (lo < hi) { const int m = (lo + hi + 1) >> 1; if (sh.first_unit[m] <= u) lo = m; else hi = m - 1; }
      const int k = u - sh.first_unit[lo];
      my_pair = lo;
      my_left = sh.n_tok[lo] - k * kAdUnit;
      const int h = (cid + lo * n_cta) % a.H;
      const int phys = sh.pt[lo][k >> 1];
      my_row_k = ad.layer_row + ((phys * 2) * a.H + h) * kPageTokens + (k & 1) * kAdUnit;
    }
  };
  unsigned char *stage0 = stages + (size_t)warp * kAdStages * 2 * kAdHalf;
  auto issue = [&](int idx, int s) {            // unit number idx of the described 32 into stage s
    const int row = __shfl_sync(0xFFFFFFFFu, my_row_k, idx);
    if (elect_one()) {
      unsigned char *dst = stage0 + (size_t)s * 2 * kAdHalf;
      mbar_expect_tx(&sh.bar[warp][s], 2 * kAdHalf);
      ad_copy(&kv_map, row, dst, &sh.bar[warp][s]);
      ad_copy(&kv_map, row + a.H * kPageTokens, dst + kAdHalf, &sh.bar[warp][s]);
    }
    __syncwarp();
  };
  // In a decode step only the new token's own K/V rows are written by the kernel in front: the first units are requested
  // ahead of the dependency wait and those two rows are read again afterwards.
  int base = u_begin, issued = u_begin;
  describe(base);
  if (a.old_pages_final)
    for (int s = 0; s < kAdStages && issued < u_end; ++s, ++issued) issue(issued - base, s);
  const int early_end = issued;
  pdl_launch_dependents();
  pdl_wait();
  trace_mark(a.trace, a.trace_slot, 1);
  for (int s = issued - u_begin; s < kAdStages && issued < u_end; ++s, ++issued) issue(issued - base, s);
  // Asked for here: looked up where they are needed, two round trips to L2 held up the warp (attention, us a layer: 16 rows
  // of 200 to 800 tokens 12.3 -> 11.7, 24 rows 13.4 -> 12.9, 37 rows of 50 to 1100 19.7 -> 19.5, 64 rows level).
  uint4 fresh[kAdStages];
#pragma unroll
  for (int e = 0; e < kAdStages; ++e) {
    const int row = __shfl_sync(0xFFFFFFFFu, my_row_k, e), n = __shfl_sync(0xFFFFFFFFu, my_left, e) - 1;
    if (u_begin + e < early_end && n < kAdUnit && lane < 16)   // the unit holds its pair's newest token
      fresh[e] = ld_cg_u4(a.kv_layer + (size_t)(row - ad.layer_row + (lane >> 3) * a.H * kPageTokens + n) * kHeadDim + 8 * (lane & 7));
  }
  // the queries of the CTA's pairs, in log2 units: times 1/sqrt(64) * log2(e)
  for (int i = threadIdx.x; i < P * (kHeadDim / 4); i += kAdWarps * 32) {
    const int pr = i / (kHeadDim / 4), c = i % (kHeadDim / 4), h = (cid + pr * n_cta) % a.H;
    const float qs = 0.125f * 1.4426950408889634f;
    const float4 x = *reinterpret_cast<const float4 *>(a.q + (size_t)sh.row[pr] * a.H * kHeadDim + h * kHeadDim + 4 * c);
    *reinterpret_cast<float4 *>(&sh.q[pr][4 * c]) = make_float4(x.x * qs, x.y * qs, x.z * qs, x.w * qs);
  }
  __syncthreads();

  uint32_t qb[4][2];                            // the query's operand fragments: k-step, half
  float acc[4][4];                              // O: dimensions 16 mt + g and + 8, columns 2t and 2t + 1 (the parts of P)
  float m = -INFINITY, l = 0.f;                 // running maximum (warp-uniform); this lane's share of the sum
  int pair = -1;
  bool dead = false;

  auto write_out = [&](int pr, const float (&o)[4][2], float inv) {   // lane t of a quad writes dimensions 16 t + g and + 8
    const int h = (cid + pr * n_cta) % a.H, r = sh.row[pr];
    const float x0 = (t == 0 ? o[0][0] : t == 1 ? o[1][0] : t == 2 ? o[2][0] : o[3][0]) * inv;
    const float x1 = (t == 0 ? o[0][1] : t == 1 ? o[1][1] : t == 2 ? o[2][1] : o[3][1]) * inv;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int dim = h * kHeadDim + 16 * t + g + 8 * e;
      uint16_t *out = a.out_image ? reinterpret_cast<uint16_t *>(reinterpret_cast<unsigned char *>(a.out) + act_image_offset_tiled(r, dim, a.H * kHeadDim))
                                  : a.out + (size_t)r * a.H * kHeadDim + dim;
      *out = float_to_bf16_bits(e ? x1 : x0);
    }
  };
  auto finish = [&]() {                         // the warp leaves `pair`
    float o[4][2];
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {             // columns 0-2 hold the three parts, the others zero
        float v = acc[mt][2 * e] + acc[mt][2 * e + 1];
        v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
        v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
        o[mt][e] = v;
      }
    const float L = warp_sum(l);
    const bool before = sh.first_unit[pair] < u_begin, behind = sh.first_unit[pair + 1] > u_end;
    if (!before && !behind) {
      if (!dead) write_out(pair, o, 1.0f / L);
    } else {
      float *dst = sh.part[warp][before ? 0 : 1];
      if (lane == 0) { dst[0] = m; dst[1] = L; }
      if (t == 0) {
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) { dst[2 + 16 * mt + g] = o[mt][0]; dst[2 + 16 * mt + g + 8] = o[mt][1]; }
      }
    }
  };

  uint32_t phase = 0;                           // bit s: parity stage s completes next
  int s = 0;
#pragma unroll 1
  for (int u = u_begin; u < u_end; ++u) {
    if (u - base == 32) { base = u; describe(base); }   // (units of the next 32 that were issued already are described again)
    const int pr = __shfl_sync(0xFFFFFFFFu, my_pair, u - base), left = __shfl_sync(0xFFFFFFFFu, my_left, u - base);
    if (pr != pair) {
      if (pair >= 0) finish();
      pair = pr; m = -INFINITY; l = 0.f;
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float2 x = *reinterpret_cast<const float2 *>(&sh.q[pr][16 * ks + 8 * hf + 2 * t]);
          float x0, x1, x2, y0, y1, y2;
          split3(x.x, x0, x1, x2);
          split3(x.y, y0, y1, y2);
          qb[ks][hf] = g == 0 ? high_halves(x0, y0) : g == 1 ? high_halves(x1, y1) : g == 2 ? high_halves(x2, y2) : 0u;
        }
      }
#pragma unroll
      for (int mt = 0; mt < 4; ++mt) acc[mt][0] = acc[mt][1] = acc[mt][2] = acc[mt][3] = 0.f;
    }
    unsigned char *st = stage0 + (size_t)s * 2 * kAdHalf;
    if (!dead && !mbar_wait_bounded(&sh.bar[warp][s], (phase >> s) & 1u, kAttnWaitNs)) {
      if (a.err) atomicExch(a.err, 1);
      dead = true;
    }
    dead = __any_sync(0xFFFFFFFFu, dead);
    if (dead) sh.dead = 1;
    phase ^= 1u << s;
    const bool last = left <= kAdUnit;          // the unit holds the pair's newest token
    if (last) {
      if (u < early_end && lane < 16) {         // copied before the kernel in front had written that token's rows
        const int n = left - 1, part = lane >> 3, c = lane & 7;
        static_assert(kAdStages == 2, "early units are the range's first two");
        *reinterpret_cast<uint4 *>(st + part * kAdHalf + n * 128 + ((c ^ (n & 7)) << 4)) = u == u_begin ? fresh[0] : fresh[1];
      }
      // V rows without a token may hold NaN, and 0 * NaN must not reach O
      for (int i = left * 8 + lane; i < kAdUnit * 8; i += 32) *reinterpret_cast<uint4 *>(st + kAdHalf + i * 16) = make_uint4(0, 0, 0, 0);
      __syncwarp();
    }
    // ---- S = K q: tokens are the rows, the three parts of q the columns ----
    const uint32_t k_base = smem_u32(st), v_base = k_base + kAdHalf;
    float sc[2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      sc[mt][0] = sc[mt][1] = sc[mt][2] = sc[mt][3] = 0.f;
      const int row = 16 * mt + (lane & 15);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t f[4];
        ldmatrix_x4(f, k_base + row * 128 + (((2 * ks + (lane >> 4)) ^ (row & 7)) << 4));
        mma_bf16_16816(sc[mt], f[0], f[1], f[2], f[3], qb[ks][0], qb[ks][1]);
      }
    }
    // lane = token: its score is the sum of columns 0-2 of row lane % 8 (+ 8) of tile lane / 16
    float x = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = sc[q >> 1][2 * (q & 1)] + sc[q >> 1][2 * (q & 1) + 1];
      const float w = __shfl_sync(0xFFFFFFFFu, v, 4 * (lane & 7)) + __shfl_sync(0xFFFFFFFFu, v, 4 * (lane & 7) + 1);
      if ((lane >> 3) == q) x = w;
    }
    if (lane >= left) x = -INFINITY;
    const float m_new = fmaxf(m, warp_max(x));
    const float f = exp2f(m - m_new), p = exp2f(x - m_new);   // first unit: exp2(-inf) = 0
    m = m_new;
    l = l * f + p;
    float p0, p1, p2;
    split3(p, p0, p1, p2);
    unsigned char *pb = sh.p[warp];
    *reinterpret_cast<uint16_t *>(pb + 2 * lane) = (uint16_t)(__float_as_uint(p0) >> 16);
    *reinterpret_cast<uint16_t *>(pb + kAdPitchP + 2 * lane) = (uint16_t)(__float_as_uint(p1) >> 16);
    *reinterpret_cast<uint16_t *>(pb + 2 * kAdPitchP + 2 * lane) = (uint16_t)(__float_as_uint(p2) >> 16);
    __syncwarp();
    if (f != 1.0f) {
#pragma unroll
      for (int mt = 0; mt < 4; ++mt) { acc[mt][0] *= f; acc[mt][1] *= f; acc[mt][2] *= f; acc[mt][3] *= f; }
    }
    // ---- O += V^T P: dimensions are the rows, the three parts of P the columns ----
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      const uint32_t b0 = *reinterpret_cast<const uint32_t *>(pb + g * kAdPitchP + 32 * ks + 4 * t);
      const uint32_t b1 = *reinterpret_cast<const uint32_t *>(pb + g * kAdPitchP + 32 * ks + 16 + 4 * t);
      const int row = 16 * ks + (lane & 7) + 8 * (lane >> 4);
#pragma unroll
      for (int mt = 0; mt < 4; ++mt) {
        uint32_t fr[4];
        ldmatrix_x4_trans(fr, v_base + row * 128 + (((2 * mt + ((lane >> 3) & 1)) ^ (row & 7)) << 4));
        mma_bf16_16816(acc[mt], fr[0], fr[1], fr[2], fr[3], b0, b1);
      }
    }
    // every lane has read the stage (the MMAs consumed what it loaded): refill it
    fence_proxy_async_smem();
    __syncwarp();
    if (issued < u_end && !dead) {              // (behind an expired wait the stage's barrier may still be in its old phase)
      if (issued - base < 32) {
        issue(issued - base, s);
      } else {                                  // beyond the described units: describe ahead, then return to the present ones
        describe(issued);
        issue(0, s);
        describe(base);
      }
      ++issued;
    }
    s = s + 1 == kAdStages ? 0 : s + 1;
  }
  trace_mark(a.trace, a.trace_slot, 3);
  if (pair >= 0) finish();
  __syncthreads();
  trace_mark(a.trace, a.trace_slot, 4);
  // ---- a pair that begins in this warp's range and goes on behind it: the parts in unit order, lane i on part i ----
  if (pair >= 0 && sh.first_unit[pair] >= u_begin && sh.first_unit[pair + 1] > u_end) {
    const int w = warp + lane;
    const bool mine = w < kAdWarps && total * w / kAdWarps < sh.first_unit[pair + 1] && total * (w + 1) / kAdWarps > total * w / kAdWarps;
    const float *src = sh.part[mine ? w : warp][w == warp ? 1 : 0];
    const float pm = mine ? src[0] : -INFINITY;
    const float M = warp_max(pm), fn = mine ? exp2f(pm - M) : 0.f;
    const float L = warp_sum(mine ? src[1] * fn : 0.f);
    const int n = 32 - __clz(__ballot_sync(0xFFFFFFFFu, mine));
    float O0 = 0.f, O1 = 0.f;
#pragma unroll 2
    for (int i = 0; i < n; ++i) {
      const float f = __shfl_sync(0xFFFFFFFFu, fn, i);
      if (f == 0.f) continue;                   // an empty range (or a part too small to count)
      const float *o = sh.part[warp + i][i == 0 ? 1 : 0] + 2;
      O0 = fmaf(f, o[lane], O0);
      O1 = fmaf(f, o[lane + 32], O1);
    }
    if (!sh.dead) {
      const int h = (cid + pair * n_cta) % a.H, r = sh.row[pair];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int dim = h * kHeadDim + lane + 32 * e;
        uint16_t *out = a.out_image ? reinterpret_cast<uint16_t *>(reinterpret_cast<unsigned char *>(a.out) + act_image_offset_tiled(r, dim, a.H * kHeadDim))
                                    : a.out + (size_t)r * a.H * kHeadDim + dim;
        *out = float_to_bf16_bits((e ? O1 : O0) / L);
      }
    }
  }
  if (dead) tc_linger(&sh.dead);                // copies of the warp may still be in flight
  trace_mark(a.trace, a.trace_slot, 2);
}

// (row, head) pairs for which the kernel is used: between the half-page kernel, of which up to two pairs per SM are one wave,
// and the streaming kernel.  ms per step, here / half pages / streaming, rows of one context of 100, 530 and 1400 tokens:
// 15 rows 0.901 / 0.834 / 0.861, 0.973 / 0.990 / 1.007, 1.195 / 1.268 / 1.311; 24 rows 0.853 / 0.793 / 0.894, 1.027 / 0.979 /
// 1.151, 1.425 / 1.339 / 1.741; 37 rows 0.934 / 0.912 / 0.987, 1.224 / 1.264 / 1.288, 1.777 / 1.939 / 1.965; 64 rows 1.063 / 1.081 /
// 1.194, 1.528 / 1.622 / 1.668, 2.579 / 2.664 / 2.692; 74 rows 1.133 / 1.146 / 1.280, 1.677 / 1.725 / 1.861, 2.857 / 2.846 / 3.202;
// 96 rows 1.329 / 1.278 / 1.418, 2.078 / 2.043 / 2.133, 3.613 / 3.609 / 3.819; 128 rows 1.611 / 1.469 / 1.678, 2.613 / 2.425 / 2.599,
// 4.71 / 4.48 / 4.78 (the three took turns, each with contexts up to 70 tokens longer than the one before).  For rows of
// equal length half pages are ahead where their splits fill the places (24, 48 rows) and from 80 rows on; the line at ten
// pairs per SM was drawn with the ragged batch of 128 rows (2.747 streaming, 2.792 here).
inline bool attention_use_decode(int R, int H, int n_sm) { return R * H > 2 * n_sm && R * H <= 10 * n_sm; }

// layer_row: first row of the layer in kv_map, the whole pool as rows of 64 bf16 (attention_decode_map)
inline cudaError_t launch_attention_decode(const AttnArgs &a, int R, const CUtensorMap &kv_map, int layer_row, int n_sm, cudaStream_t st, bool pdl) {
  static SmemOptIn opt_in;
  if (const cudaError_t e = opt_in(attention_decode_kernel, attention_decode_smem_bytes())) return e;
  AdArgs ad;
  ad.at = a; ad.layer_row = layer_row; ad.n_pair = R * a.H;
  const int n_cta = std::min(n_sm, ad.n_pair);
  if ((ad.n_pair + n_cta - 1) / n_cta > kAdMaxPairs) return cudaErrorInvalidConfiguration;
  return launch_kernel(attention_decode_kernel, dim3(n_cta), dim3(kAdWarps * 32), attention_decode_smem_bytes(), st, pdl, kv_map, ad);
}

// the pool (all layers) as rows of 64 bf16; a copy is 32 rows with the 128-byte swizzle
inline cudaError_t attention_decode_map(CUtensorMap *map, const void *pool, size_t rows) {
  return pw_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, pool, kHeadDim, rows, kHeadDim * 2, kHeadDim, kAdUnit, CU_TENSOR_MAP_SWIZZLE_128B);
}

}  // namespace ttsgpt
