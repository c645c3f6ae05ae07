// Shared device helpers: bf16 bit handling, warp reductions, the legacy warp-level MMA wrapper.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>

namespace ttsgpt {

typedef __nv_bfloat16 bf16;

constexpr int kHeadDim = 64;
constexpr int kPageTokens = 64;
constexpr int kPageElems = kPageTokens * kHeadDim;  // one (page, head, K|V) block: 4096 bf16 = 8 KB
constexpr int kMaxRows = 128;                       // rows per decode step, and rows of one row tile of a prefill pass
constexpr int kMaxPassRows = 4096;                  // rows (streams x positions) of a prefill pass: up to 32 row tiles
constexpr int kMaxSplitRows = 1024;                 // rows up to which every pass may leave four k-range partial sums (or attend over e4m3 codes)
constexpr int kMaxOrderedRows = 2688;               // rows of a sampled pass, all of which leave up to four partial sums: 55 MB of them at width 1280

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) { return __uint_as_float(((uint32_t)b) << 16); }

__device__ __forceinline__ uint16_t float_to_bf16_bits(float f) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}

// Two fp32 operations in one instruction, each rounded as its scalar form.
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Streaming 128-bit load that does not pollute L1 (weights and KV pages are read once per step).
__device__ __forceinline__ uint4 ld_stream_u4(const void *p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// Programmatic dependent launch.  A kernel launched with the programmatic-serialization attribute
// may start while its predecessor on the stream is still running; `pdl_wait` blocks until every
// predecessor has completed and its writes are visible, `pdl_launch_dependents` lets the successor
// start early.  Before `pdl_wait` a kernel may only touch data that no kernel of the step writes
// (weights, and state written before the first kernel of the chain started).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Optional timeline trace: thread 0 of CTA 0 of a traced kernel stores the global nanosecond timer
// at entry, after the dependency wait, at its end (and at up to five inner points) into
// trace[8*slot + 0..7].
__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");   // "memory": the read stays where it is written, e.g. behind a barrier
  return t;
}
__device__ __forceinline__ void trace_mark(unsigned long long *trace, int slot, int which, int tid = 0) {
  if (trace && threadIdx.x == tid && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
    trace[8 * slot + which] = global_timer_ns();
}

// ---- bulk asynchronous copy (TMA, untiled) into shared memory, completion on an mbarrier ----
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// both addresses 16-byte aligned, size a multiple of 16
__device__ __forceinline__ void bulk_copy_g2s(void *dst_smem, const void *src_gmem, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst_smem)),
               "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for the barrier's phase, at most about `limit_ns` nanoseconds.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > limit_ns) return false;
  }
  return true;
}
// orders this thread's earlier generic-proxy accesses of shared memory before its later bulk copies
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The opt-in to more than 48 KB of dynamic shared memory, a function attribute that belongs to one device: made by every
// thread that comes before one of them has made it, so that none launches ahead of it.
struct SmemOptIn {
  std::atomic<bool> done[64] = {};
  template <typename... KArgs>
  cudaError_t operator()(void (*kernel)(KArgs...), size_t bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < 64;
    if (known && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && known) done[dev].store(true, std::memory_order_release);
    return e;
  }
};

// Launches `kernel` with or without the programmatic-serialization attribute.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 bool pdl, Args... args) {
  cudaLaunchConfig_t cfg;
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// A cluster barrier in two halves, by every thread of every CTA: arrive early, wait where the others must have arrived.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
// writes the word at `p`'s place in the shared memory of a CTA of the cluster
__device__ __forceinline__ void st_shared_of_rank(float *p, uint32_t rank, float v) {
  asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.f32 [a], %2;\n\t}" ::"r"(smem_u32(p)), "r"(rank), "f"(v) : "memory");
}

// The same with `cluster` neighbouring CTAs as a thread-block cluster (one: none).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_cluster_dims(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, dim3 cluster, cudaStream_t st, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg;
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (cluster.x * cluster.y * cluster.z > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = cluster.x; at[n].val.clusterDim.y = cluster.y; at[n].val.clusterDim.z = cluster.z;
    ++n;
  }
  if (pdl) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, int cluster, cudaStream_t st, bool pdl, Args... args) {
  return launch_kernel_cluster_dims(kernel, grid, block, 0, dim3(cluster), st, pdl, args...);
}

// 128-bit load served by L2 (never by a possibly stale L1 line).
__device__ __forceinline__ uint4 ld_cg_u4(const void *p) {
  uint4 r;
  asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Pages of a decode step's next attention, asked into L2 while the linears leave the memory idle: by one warp of every CTA.
struct KvPrefetch {
  const unsigned char *layer;   // the layer's slice of the page pool; null: nothing to ask for
  uint32_t block_bytes;         // one (page, K|V, head) block
  int blocks;                   // blocks of a page, contiguous
  const int4 *slots;            // rows by rank of length, and their pages (AttnArgs)
  const int *slot_pages;
  int pps, rows, cap;           // up to `cap` complete pages of every row
  int part, n_parts;            // this kernel's share of the blocks
};
// The blocks are numbered rank by rank, page by page; a lane takes the number it starts with and every stride-th behind it.
__host__ __device__ __forceinline__ int kv_prefetch_first(const KvPrefetch &p, int cta, int lane) { return (cta * 32 + lane) * p.n_parts + p.part; }
__host__ __device__ __forceinline__ int kv_prefetch_stride(const KvPrefetch &p, int n_cta) { return n_cta * 32 * p.n_parts; }
__host__ __device__ __forceinline__ int kv_prefetch_total(const KvPrefetch &p) { return p.rows * p.cap * p.blocks; }
// address of block number u, or null: that page is not complete
__host__ __device__ __forceinline__ const unsigned char *kv_prefetch_address(const KvPrefetch &p, int u) {
  const int t = u / p.blocks, b = u - t * p.blocks, z = t / p.cap, j = t - z * p.cap;
  const int phys = p.slot_pages[z * p.pps + j];
  if (j >= (p.slots[z].y - 1) / kPageTokens) return nullptr;
  return p.layer + ((size_t)phys * p.blocks + b) * p.block_bytes;
}
__device__ __forceinline__ void kv_prefetch(const KvPrefetch &p, int cta, int n_cta) {
  const int total = kv_prefetch_total(p), stride = kv_prefetch_stride(p, n_cta);
#pragma unroll 1
  for (int u = kv_prefetch_first(p, cta, threadIdx.x & 31); u < total; u += stride)
    if (const unsigned char *q = kv_prefetch_address(p, u)) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "r"(p.block_bytes) : "memory");
}

// D(16x8,f32) += A(16x16,bf16,row) * B(16x8,bf16,col).  Fragment layout (g = lane/4, t = lane%4):
// a0=(row g, k 2t..2t+1) a1=(row g+8, same k) a2=(row g, k 2t+8..2t+9) a3=(row g+8, same);
// b0=(k 2t..2t+1, col g) b1=(k 2t+8..2t+9, col g); c0,c1=(row g, cols 2t,2t+1) c2,c3=(row g+8).
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 0.5 x (1 + tanh(u)) = x / (1 + exp(-2u)), u = sqrt(2/pi) (x + 0.044715 x^3): the same function, written
// with one exponential and one reciprocal (about 6 instructions; the library tanhf is about 30 with
// branches, which made the GELU epilogue of the 128-row FC1 the longest part of that kernel).  The
// quotient form keeps the relative error at a few ulp in the negative tail too, where 1 + tanh cancels.
__device__ __forceinline__ float gelu_tanh_f(float x) {
  const float k0 = 0.7978845608028654f, k1 = 0.044715f;
  const float u = k0 * (x + k1 * x * x * x);
  return __fdividef(x, 1.0f + __expf(-2.0f * u));
}
__device__ __forceinline__ float gelu_erf_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.7071067811865476f)); }

}  // namespace ttsgpt
