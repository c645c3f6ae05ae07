// Linear of large prefill passes (Table I / III regime: the prefixes of many utterances): a persistent tcgen05 kernel
// over tiles of 256 rows x BN output features (BN = 128 or 256), one tile per pair of CTAs (cta_group::2).
//
// Operand images, epilogue kinds and arguments are those of gemm_tc.cuh: the activation block of a k-chunk (128 rows x
// 64 columns, 16 KB) of each CTA is its half of the M operand, BN/2 weight rows its half of the N operand.  The images
// are copied as two-dimensional tensors whose copies may complete on the barrier of the other CTA of the pair, so that
// CTA 0's issuer waits on one barrier per stage for both CTAs' copies.  A pair of CTAs walks the tiles; warp 0 of each
// keeps a ring of stages full across tile boundaries, warp 1 of CTA 0 issues the instructions, and warps 2-9 of each
// drain one of two accumulators in tensor memory while the other fills, so that the epilogue of a tile and the first
// copies of the next run under the instructions.
//
// Every wait is bounded.  A role acts only behind a wait that was satisfied; where one expires, the roles of both CTAs
// stop (going on would arrive on barriers whose phase is still open, which is a fault).  The issuer then commits
// nothing more, so that a tile is stored, by either CTA, only if every wait in front of its accumulator was satisfied.
// A pair that gave up stays until the copies it requested have landed in its shared memory.
//
// What bounds it.  One CTA per 128 x 256 tile is bound by shared memory: an instruction of K = 16 reads 12 KB of
// operands in 128 cycles and its copies write another 12 KB, 192 of 128 bytes per cycle; measured 0.40 us per k-chunk
// where the instructions alone take 0.30.  A pair reads and writes 8 KB each per CTA: 0.315 us.  A thread of the epilogue
// holds columns of one row, and rows are kilobytes apart in every destination (written row by row from the registers
// the epilogue of a tile took 13 us): a warp parks its 32 rows in shared memory and hands them to the copy engine, as
// 4 KB of the next linear's image (32 rows x 64 columns are contiguous there) or as a 32 x 32 fp32 block that the copy
// itself adds into the residual stream, so that x is never read here.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include "gemm_tc.cuh"

namespace ttsgpt {

constexpr int kPwThreads = 320;             // warp 0 producer, warp 1 issuer, warps 2-9 epilogue
constexpr int kPwMaxStages = 8;
constexpr uint32_t kPwRingBytes = 6 * 32768;             // per CTA: 6 stages at BN = 256, 8 at BN = 128
constexpr uint32_t kPwPatchBytes = 8 * 4096;             // 4 KB per epilogue warp
constexpr uint32_t kPwTokenBytes = 8192;                 // a CTA with neither rows nor weights in a tile copies one box all the same
inline size_t pw_smem_bytes() { return (size_t)kPwRingBytes + kPwPatchBytes + 1024 + 512; }
inline int pw_stages(int bn) { return std::min(kPwMaxStages, (int)(kPwRingBytes / (16384u + (uint32_t)bn * 64u))); }

struct PwTile { int row0, rows, n0, ks, kc0, n_it; };

// tile t as CTA `rank` of the pair sees it: row tiles (two per pair) run fastest, so that concurrent pairs share a few
// weight blocks; then k-ranges, then feature tiles
__device__ __forceinline__ PwTile pw_tile(const GemmTcArgs &a, int t, int n_rp, int rank, int KC) {
  PwTile p;
  const int rp = t % n_rp, u = t / n_rp;
  p.ks = u % a.ksplit;
  p.n0 = (u / a.ksplit) * a.bn;
  p.row0 = (2 * rp + rank) * kMaxRows;
  p.rows = min(kMaxRows, a.B - p.row0);   // <= 0: the last pair's second row tile does not exist
  const int per = (KC + a.ksplit - 1) / a.ksplit;
  p.kc0 = min(KC, p.ks * per);
  p.n_it = min(KC, p.kc0 + per) - p.kc0;
  return p;
}

// this CTA's half of a tile's weight rows in one k-chunk: rows n0 + rank * bn/2 .. + bn/2 - 1 (bn/2 = 64 or 128, so the
// half lies in one 128-row block of the image); a half past the last feature is not copied: its accumulator columns are
// not stored
__device__ __forceinline__ bool pw_half_exists(const GemmTcArgs &a, int n0, int rank) { return n0 + rank * (a.bn >> 1) < a.N; }
__device__ __forceinline__ uint32_t pw_pair_bytes(const GemmTcArgs &a, const PwTile &p, int t) {   // of a stage of tile t, both CTAs together; p: CTA 0's view
  const uint32_t starved = t + 1 == a.starve ? 16u : 0u;   // test aid: bytes that never arrive
  const bool half1 = pw_half_exists(a, p.n0, 1);
  return 16384u + (a.B > p.row0 + kMaxRows ? 16384u : half1 ? 0u : kPwTokenBytes) + (uint32_t)(a.bn >> 1) * 128u * (half1 ? 2u : 1u) + starved;
}
// An operand image as a two-dimensional tensor: rows of 64 bf16 (128 bytes), blocks one behind the other.  The bytes
// are already in the order the tensor core wants, so the copy itself does not swizzle.  Both CTAs of a pair complete
// on the barrier of CTA 0 (`bar`: its address in the cluster's window).
constexpr int kPwBoxRows = 64;   // rows per tensor copy
__device__ __forceinline__ void pw_copy_rows(const CUtensorMap *map, int row, unsigned char *dst, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_u32(dst)), "l"(map), "r"(0), "r"(row), "r"(bar) : "memory");
}
__device__ __forceinline__ void pw_copy_weights(const CUtensorMap *map, const GemmTcArgs &a, int n0, int rank, int kc, int KC, unsigned char *dst, uint32_t bar) {
  const int b = n0 + rank * (a.bn >> 1), row = ((b >> 7) * KC + kc) * 128 + (b & 127);
  for (int r = 0; r < (a.bn >> 1); r += kPwBoxRows) pw_copy_rows(map, row + r, dst + r * 128, bar);
}

// ---- pairs of CTAs (cta_group::2) ----
__device__ __forceinline__ void cluster_barrier() { asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory"); }
// arrives on the barrier at the same place in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ void mbar_arrive_remote(uint64_t *bar, uint32_t rank) {
  asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\tmbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t}"
               ::"r"(smem_u32(bar)), "r"(rank) : "memory");
}
// sets the flag of CTA `rank` of the pair
__device__ __forceinline__ void pw_tell(volatile int *failed, uint32_t rank) {
  asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\tst.relaxed.cluster.shared::cluster.u32 [ra], 1;\n\t}"
               ::"r"(smem_u32(const_cast<const int *>(failed))), "r"(rank) : "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// arrives on the barrier of both CTAs once every MMA issued so far by this thread has completed
__device__ __forceinline__ void tc_commit2(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tc_mma2(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0u)
      : "memory");
}

// ---- out of shared memory by the copy engine ----
__device__ __forceinline__ void bulk_store(void *dst, const unsigned char *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes) : "memory");
}
// a 32 x 32 fp32 block at (col, row), 128 bytes per row with the 128-byte swizzle; ADD: into what is there
template <bool ADD>
__device__ __forceinline__ void block_store(const CUtensorMap *map, int col, int row, const unsigned char *src) {
  if (ADD) asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(col), "r"(row), "r"(smem_u32(src)) : "memory");
  else asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(col), "r"(row), "r"(smem_u32(src)) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }   // sources may be overwritten
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }         // writes are done

// 32 lanes x 8 columns of 32-bit
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Where a group of 64 features of a warp's 32 rows goes.
enum { PW_GELU_TANH = 0, PW_GELU_ERF = 1, PW_BF16 = 2, PW_F32 = 3 };
// One group out of tensor memory, through bias (and int8 scale) and GELU, into the warp's patch: [32 rows][128 bytes],
// 16-byte unit u at u ^ (row % 8); bf16 kinds leave the 64 columns there, fp32 leaves in two blocks of 32 columns.
// The loop is kept rolled, eight columns a turn: unrolled over 32 columns this code ran at ten cycles an instruction,
// fetched from beyond the instruction cache for every block (10.7 us of epilogue for a tile of the O projection).
// bs, sc: two features per lane and register, columns 0..31 and 32..63 of the group, dealt out by shuffles.
template <int KIND>
__device__ __forceinline__ void pw_group(const GemmTcArgs &a, uint32_t t_grp, unsigned char *patch, int lane, const uint32_t (&bs)[2], const uint32_t (&sc)[2],
                                         bool empty_range, bool store, const CUtensorMap *out_map, bool add, int col, int map_row, float *plain, size_t pitch, int rows) {
#pragma unroll 1
  for (int c8 = 0; c8 < 8; ++c8) {
    float v[8];
    tmem_ld8(t_grp + 8u * c8, v);
    if (empty_range) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = 0.f;
    }
    const uint32_t b_mine = c8 < 4 ? bs[0] : bs[1];
    if (a.wfmt == WF_INT8) {
      const uint32_t s_mine = c8 < 4 ? sc[0] : sc[1];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, b_mine, 4 * (c8 & 3) + q), s = __shfl_sync(0xFFFFFFFFu, s_mine, 4 * (c8 & 3) + q);
        v[2 * q] = fmaf(v[2 * q], bf16_lo(s), bf16_lo(b));
        v[2 * q + 1] = fmaf(v[2 * q + 1], bf16_hi(s), bf16_hi(b));
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, b_mine, 4 * (c8 & 3) + q);
        v[2 * q] += bf16_lo(b);
        v[2 * q + 1] += bf16_hi(b);
      }
    }
    if (KIND == PW_GELU_TANH) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = gelu_tanh_f(v[c]);
    }
    if (KIND == PW_GELU_ERF) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = gelu_erf_f(v[c]);
    }
    if (c8 == 0 || (KIND == PW_F32 && c8 == 4)) {   // the patch is free once the copy engine has read it
      if (elect_one()) bulk_wait_read();
      __syncwarp();
    }
    if (KIND != PW_F32) {
      *reinterpret_cast<uint4 *>(patch + lane * 128 + ((c8 ^ (lane & 7)) << 4)) =
          make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
      continue;
    }
    const int u = 2 * (c8 & 3);
    *reinterpret_cast<float4 *>(patch + lane * 128 + ((u ^ (lane & 7)) << 4)) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(patch + lane * 128 + (((u + 1) ^ (lane & 7)) << 4)) = make_float4(v[4], v[5], v[6], v[7]);
    if ((c8 & 3) != 3) continue;
    const int c32 = 32 * (c8 >> 2);
    if (out_map) {
      fence_proxy_async_smem();
      __syncwarp();
      if (store && elect_one()) {
        if (add) block_store<true>(out_map, col + c32, map_row, patch);
        else block_store<false>(out_map, col + c32, map_row, patch);
        bulk_commit();
      }
      __syncwarp();
    } else {   // rows the copy engine cannot address (a caller's own array): eight lanes per row
      __syncwarp();
      for (int rr = lane >> 3; rr < rows && store; rr += 4) {
        const float4 x = *reinterpret_cast<const float4 *>(patch + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4));
        const float xs[4] = {x.x, x.y, x.z, x.w};
        float *dst = plain + (size_t)rr * pitch + c32 + 4 * (lane & 7);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (col + c32 + 4 * (lane & 7) + e < a.N) dst[e] = add ? dst[e] + xs[e] : xs[e];   // the last features may be ragged
      }
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(kPwThreads, 1) gemm_pw_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap x_map,
                                                              const __grid_constant__ CUtensorMap out_map, const GemmTcArgs a) {
  extern __shared__ __align__(16) unsigned char pw_smem_raw[];
  unsigned char *ring = pw_smem_raw + ((1024u - (smem_u32(pw_smem_raw) & 1023u)) & 1023u);
  uint64_t *full = reinterpret_cast<uint64_t *>(ring + kPwRingBytes + kPwPatchBytes);   // (CTA 0's) the copies of both CTAs into the stage have landed
  uint64_t *empty = full + kPwMaxStages;
  uint64_t *acc_full = empty + kPwMaxStages;   // [2] accumulator complete (issuer -> epilogues of both CTAs)
  uint64_t *acc_free = acc_full + 2;           // [2] (CTA 0's) accumulator read out (epilogue warps of both CTAs -> issuer)
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_free + 2);
  volatile int *failed = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, n_pair = gridDim.x >> 1;   // cluster of two along x
  const int KC = a.K / kTcKChunk, n_stage = a.stages;
  const int n_rp = (a.B + 2 * kMaxRows - 1) / (2 * kMaxRows);
  const int n_tile = n_rp * a.ksplit * ((a.N + a.bn - 1) / a.bn);
  const uint32_t stage_bytes = 16384u + (uint32_t)a.bn * 64u;
  trace_mark(a.trace, a.trace_slot, 0);
  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stage; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    for (int g = 0; g < 2; ++g) { mbar_init(acc_full + g, 1); mbar_init(acc_free + g, 16); }   // 8 epilogue warps of either CTA
    *failed = 0;
  }
  if (warp == 0) tmem_alloc2(tmem_slot, 512);
  tc_fence_before_sync();
  __syncthreads();
  cluster_barrier();   // both CTAs' barriers and tensor memory exist
  tc_fence_after_sync();
  const uint32_t tmem_d = *tmem_slot;

  // weights do not depend on the kernel in front: the first stages' are requested ahead of the dependency wait
  int pre = 0;
  uint32_t full0;   // CTA 0's full barriers
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(full0) : "r"(smem_u32(full)));
  if (warp == 0) {
    const PwTile p = pw_tile(a, pair, n_rp, rank, KC);
    pre = min(p.n_it, n_stage);
    for (int i = 0; i < pre; ++i)
      if (elect_one()) {
        if (rank == 0) mbar_expect_tx(full + i, pw_pair_bytes(a, p, pair));
        if (pw_half_exists(a, p.n0, rank)) pw_copy_weights(&w_map, a, p.n0, rank, p.kc0 + i, KC, ring + (size_t)i * stage_bytes + 16384, full0 + 8u * i);
      }
    __syncwarp();
  }
  pdl_launch_dependents();
  pdl_wait();
  trace_mark(a.trace, a.trace_slot, 1);

  if (warp == 0) {
    // A stage's release is waited for by its parity, so a producer may not fall two releases behind the issuer.  It does not
    // as long as the issuer needs something of each chunk from it: a CTA with neither rows nor weights in a tile copies a
    // box of the other's rows.  In the first lap that does not hold (its weights were requested above, and CTA 1 may have
    // no rows), so the first lap, whose stages are free, does not wait.  (A wait there for the phase before a fresh barrier's
    // first found that first phase complete in one launch in 10^6, and stood still.)
    int it = 0, s = 0;         // stages handed out so far, over all tiles; the next stage
    uint32_t parity = 1;       // of the phase that frees it
    bool go = true;
    for (int t = pair; go && t < n_tile; t += n_pair) {
      const PwTile p = pw_tile(a, t, n_rp, rank, KC);
      const uint32_t bytes = pw_pair_bytes(a, p, t);   // used by CTA 0 only
      const bool w_mine = pw_half_exists(a, p.n0, rank);
      const int n_box = p.rows > 0 ? 2 : w_mine ? 0 : 1;
      const int xrow = (((p.row0 >> 7) - (n_box == 1 ? 1 : 0)) * KC + p.kc0) * kMaxRows;
      if (a.starve < 0 && rank == 1) {                 // test aid: CTA 1's producer is late
        const unsigned long long t0 = global_timer_ns();
        while (__any_sync(0xFFFFFFFFu, global_timer_ns() - t0 <= a.issue_wait_ns)) {}
      }
      auto chunk = [&](int i) {
        unsigned char *st = ring + (size_t)s * stage_bytes;
        if (elect_one()) {
          if (it >= pre) {
            if (rank == 0) mbar_expect_tx(full + s, bytes);
            if (w_mine) pw_copy_weights(&w_map, a, p.n0, rank, p.kc0 + i, KC, st + 16384, full0 + 8u * s);
          }
          if (n_box > 0) pw_copy_rows(&x_map, xrow + i * kMaxRows, st, full0 + 8u * s);
          if (n_box > 1) pw_copy_rows(&x_map, xrow + i * kMaxRows + kPwBoxRows, st + kPwBoxRows * 128, full0 + 8u * s);
        }
        __syncwarp();
        if (++s == n_stage) { s = 0; parity ^= 1u; }   // no division by the runtime ring depth
        ++it;
      };
      int i = 0;   // two loops: one that asks in every turn whether to wait takes 0.7 us more per launch
      for (; i < p.n_it && it < n_stage; ++i) chunk(i);
      for (; i < p.n_it; ++i) {
        if (!(go = tc_wait_warp<false>(empty + s, parity, failed, a.err))) break;
        chunk(i);
      }
    }
    trace_mark(a.trace, a.trace_slot, 3);   // last copy issued
    // The issuer's releases of the last stages are arrivals in this CTA's shared memory, which is the next CTA's once this
    // one has left: they are waited for too.
    if (it < n_stage) { s = 0; parity = 0; }
    for (int i = 0; go && i < min(it, n_stage); ++i) {
      go = tc_wait_warp<false>(empty + s, parity, failed, a.err);
      if (++s == n_stage) { s = 0; parity ^= 1u; }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = tc_instr_desc(256, a.bn);
      int s = 0, k = 0;
      uint32_t parity = 0;
      bool go = true;
      for (int t = pair; go && t < n_tile; t += n_pair, ++k) {
        const PwTile p = pw_tile(a, t, n_rp, rank, KC);
        const uint32_t dst = tmem_d + 256u * (uint32_t)(k & 1);
        if (k >= 2 && !tc_wait_warp<true>(acc_free + (k & 1), (uint32_t)((k >> 1) - 1) & 1u, failed, a.err, &a)) break;
        for (int i = 0; i < p.n_it; ++i) {
          if (!(go = tc_wait_warp<true>(full + s, parity, failed, a.err, &a))) break;
          tc_fence_after_sync();
          const unsigned char *st = ring + (size_t)s * stage_bytes;
          const uint64_t da = tc_smem_desc(st), db = tc_smem_desc(st + 16384);
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < kTcKChunk / 16; ++j) tc_mma2(dst, da + 2 * j, db + 2 * j, idesc, (i == 0 && j == 0) ? 0u : 1u);
            tc_commit2(empty + s);
            if (i == p.n_it - 1) tc_commit2(acc_full + (k & 1));
          }
          __syncwarp();
          if (++s == n_stage) { s = 0; parity ^= 1u; }
        }
        if (p.n_it <= 0 && elect_one()) tc_commit2(acc_full + (k & 1));
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warp w may read accumulator lanes 32*(w%4)..+31 = rows of the tile; warps w and w+4 share a lane
    //      quarter and take alternate groups of 64 features (one head of q, K or V; one k-chunk of the next linear) ----
    const int lw = warp & 3, grp = (warp - 2) >> 2;
    unsigned char *patch = ring + kPwRingBytes + (size_t)(warp - 2) * 4096;   // [32 rows][128 bytes], 16-byte unit u at u ^ (row % 8)
    const bool partial = a.mode == EPI_RESID && a.ksplit > 1;
    const bool use_bias = a.bias && !partial, add = a.mode == EPI_RESID && !partial;
    int k = 0;
    for (int t = pair; t < n_tile; t += n_pair, ++k) {
      const PwTile p = pw_tile(a, t, n_rp, rank, KC);
      const int rows = min(32, p.rows - lw * 32);       // real rows of this warp
      const int r = p.row0 + lw * 32 + lane;            // this thread's row of the pass
      const int n_end = min(p.n0 + a.bn, a.N);
      uint16_t *kv_mine = nullptr;                      // EPI_QKV: where the K/V of the row go
      if (a.mode == EPI_QKV && p.n0 + a.bn > a.d && lane < rows) {
        if (a.kv_stage) {
          kv_mine = a.kv_stage + (size_t)r * 2 * a.d;
        } else {
          const int pos = a.row_pos[r];
          kv_mine = a.kv_layer + ((size_t)a.page_table[(size_t)a.row_stream[r] * a.pps + (pos >> 6)] * 2 * a.H) * kPageElems + (size_t)(pos & 63) * kHeadDim;
        }
      }
      // bias and scales of this warp's (up to two) groups, two features per lane and register, fetched ahead of the
      // accumulator: a load behind it takes over 1000 cycles while every SM streams operands
      uint32_t bias2[2][2], scale2[2][2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int n = p.n0 + grp * 64 + (q >> 1) * 128 + (q & 1) * 32 + 2 * (lane & 15);
        uint32_t bw = 0u, sw = 0u;
        if (n + 1 < n_end) {
          if (use_bias) bw = __ldg(reinterpret_cast<const uint32_t *>(a.bias + n));
          if (a.wfmt == WF_INT8) sw = __ldg(reinterpret_cast<const uint32_t *>(a.scales + n));
        } else if (n < n_end) {
          if (use_bias) bw = a.bias[n];
          if (a.wfmt == WF_INT8) sw = a.scales[n];
        }
        bias2[q >> 1][q & 1] = bw; scale2[q >> 1][q & 1] = sw;
      }
      if (!tc_wait_warp<false>(acc_full + (k & 1), (uint32_t)(k >> 1) & 1u, failed, a.err)) break;   // committed by CTA 0 to both CTAs
      if (k == 0) trace_mark(a.trace, a.trace_slot, 4, 64);   // first accumulator complete
      tc_fence_after_sync();
      __syncwarp();
      const uint32_t t_row = tmem_d + 256u * (uint32_t)(k & 1) + ((uint32_t)(lw * 32) << 16);
      const bool store = rows > 0;
#pragma unroll 1
      for (int n64 = p.n0 + grp * 64; n64 < n_end; n64 += 128) {
        const bool second = n64 - p.n0 >= 128;
        const uint32_t bs[2] = {second ? bias2[1][0] : bias2[0][0], second ? bias2[1][1] : bias2[0][1]};
        const uint32_t sc[2] = {second ? scale2[1][0] : scale2[0][0], second ? scale2[1][1] : scale2[0][1]};
        const uint32_t t_grp = t_row + (uint32_t)(n64 - p.n0);
        const bool to_img = a.mode == EPI_GELU || (a.mode == EPI_QKV && n64 < a.d && a.q_img);
        const bool none = p.n_it <= 0;
        if (a.mode == EPI_GELU) {
          if (a.gelu_tanh) pw_group<PW_GELU_TANH>(a, t_grp, patch, lane, bs, sc, none, store, nullptr, false, 0, 0, nullptr, 0, 0);
          else pw_group<PW_GELU_ERF>(a, t_grp, patch, lane, bs, sc, none, store, nullptr, false, 0, 0, nullptr, 0, 0);
        } else if (to_img || (a.mode == EPI_QKV && n64 >= a.d)) {
          pw_group<PW_BF16>(a, t_grp, patch, lane, bs, sc, none, store, nullptr, false, 0, 0, nullptr, 0, 0);
        } else {
          const int prow = ((p.row0 >> 7) * a.ksplit + p.ks) * kMaxRows + lw * 32;
          float *plain = partial ? a.out_f32 + (size_t)prow * a.N + n64 : a.out_f32 + (size_t)(p.row0 + lw * 32) * a.out_stride + n64;
          pw_group<PW_F32>(a, t_grp, patch, lane, bs, sc, none, store, a.out_mapped ? &out_map : nullptr, add, n64, partial ? prow : p.row0 + lw * 32, plain,
                           partial ? (size_t)a.N : (size_t)a.out_stride, rows);
          continue;
        }
        if (to_img) {   // 32 rows x 64 columns are 4 KB of the image; rows past the pass are never read
          fence_proxy_async_smem();
          __syncwarp();
          unsigned char *img = reinterpret_cast<unsigned char *>(a.mode == EPI_GELU ? a.out_img : a.q_img);
          const int cols64 = (a.mode == EPI_GELU ? a.N : a.d) >> 6;
          if (store && elect_one()) {
            bulk_store(img + ((size_t)(p.row0 >> 7) * cols64 + (n64 >> 6)) * (kMaxRows * 128) + (size_t)lw * 4096, patch, 4096);
            bulk_commit();
          }
          __syncwarp();
        } else {        // K/V rows: eight lanes write the 128 bytes of a row into its page slot or staging row
          __syncwarp();
          const int which = n64 >= 2 * a.d, col = n64 - (which ? 2 * a.d : a.d);
          const size_t kv_off = a.kv_stage ? (size_t)which * a.d + col : ((size_t)which * a.H + (col >> 6)) * kPageElems;
#pragma unroll 2
          for (int i = 0; i < 8; ++i) {
            const int rr = 4 * i + (lane >> 3);
            const uint4 y = *reinterpret_cast<const uint4 *>(patch + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4));
            uint16_t *dst = reinterpret_cast<uint16_t *>(__shfl_sync(0xFFFFFFFFu, reinterpret_cast<unsigned long long>(kv_mine), rr));
            if (rr < rows && store) *reinterpret_cast<uint4 *>(dst + kv_off + 8 * (lane & 7)) = y;
          }
          __syncwarp();
        }
      }
      // this warp has read its part of the accumulator, which may take the tile after next
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(acc_free + (k & 1), 0);
    }
    bulk_wait_all();   // (the lane that committed the copies; nothing to wait for in the others)
    trace_mark(a.trace, a.trace_slot, 6, 64);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    if (__any_sync(0xFFFFFFFFu, *failed)) pw_tell(failed, rank ^ 1);
    tc_linger(failed);
  }
  __syncwarp();
  cluster_barrier();   // neither CTA leaves, nor frees tensor memory, while the other still arrives on its barriers or computes
  trace_mark(a.trace, a.trace_slot, 2, 64);
  if (warp == 0) tmem_dealloc2(tmem_d, 512);
}

// Tile width and k-ranges of a linear on n_sm SMs: the plan with the smallest estimate.  A k-chunk takes about
// chunk_us in a full ring, a tile's epilogue epi_us, hidden behind the next tile's instructions unless it is longer.
// k-ranges (residual linears only, at least 4 k-chunks each) fill the SMs of small passes; the LayerNorm behind them
// reads one more partial row per range.
struct PwPlan { int bn, ksplit; float us; };
inline PwPlan pw_plan(int N, int K, int rows, bool resid, int n_sm, int fixed_ks = 0) {   // fixed_ks: only that many k-ranges
  const int n_rp = (rows + 2 * kMaxRows - 1) / (2 * kMaxRows), KC = K / kTcKChunk, n_pair = std::max(1, n_sm / 2);
  PwPlan best = {128, 1, 1e30f};
  for (int bn = 128; bn <= 256; bn += 128) {
    const float chunk_us = bn <= 128 ? 0.20f : 0.33f, epi_us = 1.2f * (bn / 64) / 2;
    for (int ks = 1; ks <= (resid ? kTwMaxPartials : 1); ++ks) {
      const int per = (KC + ks - 1) / ks;
      if (fixed_ks > 0 && ks != fixed_ks) continue;
      if (fixed_ks <= 0 && ks > 1 && (per < 4 || per * (ks - 1) >= KC || (rows + kMaxRows - 1) / kMaxRows * ks > 4 * kMaxSplitRows / kMaxRows)) break;
      const int tiles = n_rp * ((N + bn - 1) / bn) * ks, waves = (tiles + n_pair - 1) / n_pair;
      const float tile_us = std::max(per * chunk_us, epi_us);
      const float us = waves * tile_us + epi_us + (ks > 1 ? 0.4f + 0.0005f * rows * ks : 0.f);
      if (us < best.us) best = {bn, ks, us};
    }
  }
  return best;
}

inline cudaError_t pw_encode(CUtensorMap *map, CUtensorMapDataType type, const void *base, size_t cols, size_t rows, size_t pitch_bytes, int box_cols,
                             int box_rows, CUtensorMapSwizzle swizzle) {
  static std::atomic<PFN_cuTensorMapEncodeTiled> known{nullptr};   // the same address whoever looks it up first
  PFN_cuTensorMapEncodeTiled encode = known.load(std::memory_order_acquire);
  if (!encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
    if (e != cudaSuccess) return e;
    if (found != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = (PFN_cuTensorMapEncodeTiled)fn;
    known.store(encode, std::memory_order_release);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)pitch_bytes};
  const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows}, step[2] = {1, 1};
  return encode(map, type, 2, const_cast<void *>(base), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess : cudaErrorInvalidValue;
}
// an operand image of `blocks` blocks of 128 rows x 128 bytes, as the source of pw_copy_rows
inline cudaError_t pw_image_map(CUtensorMap *map, const void *img, size_t blocks) {
  return pw_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, img, 64, blocks * 128, 128, 64, kPwBoxRows, CU_TENSOR_MAP_SWIZZLE_NONE);
}
// fp32 rows (16-byte aligned, cols a multiple of 4), as the destination of block_store
inline cudaError_t pw_rows_map(CUtensorMap *map, const float *base, size_t cols, size_t rows) {
  return pw_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, base, cols, rows, cols * 4, 32, 32, CU_TENSOR_MAP_SWIZZLE_128B);
}

// w_map, x_map: pw_image_map of a0.w_img and a0.act_img; out_map: pw_rows_map of a0.out_f32 (null: plain stores)
inline cudaError_t launch_gemm_pw(const GemmTcArgs &a0, const CUtensorMap &w_map, const CUtensorMap &x_map, const CUtensorMap *out_map, int bn, int n_sm,
                                  cudaStream_t st, bool pdl) {
  static SmemOptIn opt_in;
  if (const cudaError_t e = opt_in(gemm_pw_kernel, pw_smem_bytes())) return e;
  GemmTcArgs a = a0;
  a.bn = bn;
  a.stages = pw_stages(bn);
  a.out_mapped = out_map != nullptr;
  const int tiles = ((a.B + 2 * kMaxRows - 1) / (2 * kMaxRows)) * a.ksplit * ((a.N + bn - 1) / bn);
  cudaLaunchConfig_t cfg;
  cfg.gridDim = dim3(2 * std::min(tiles, std::max(1, n_sm / 2))); cfg.blockDim = dim3(kPwThreads);
  cfg.dynamicSmemBytes = pw_smem_bytes(); cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_pw_kernel, w_map, x_map, out_map ? *out_map : x_map, a);
}

}  // namespace ttsgpt
