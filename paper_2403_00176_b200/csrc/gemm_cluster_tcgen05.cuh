// The varlen GEMM for few output tiles and a long K: a thread-block cluster of S CTAs per 128 x 64 tile, K split among them.
//   out[M,N] = act2(act(A[M,K] * Wt[N,K]^T + bias[N]) (+ residual[M,N])),  bf16 in, fp32 accumulate, bf16 out.
// With a tile per CTA, 64 rows x 768 columns are 12 CTAs that each pull K x 128 columns of operands (K = 3072: 790 KB)
// through one SM's load path, 8 of the kernel's 11 us; the other 136 SMs idle.  Here each CTA of a cluster multiplies K / S
// into its own tensor memory, with every stage in flight at once, puts its fp32 tile into its shared memory, and after one
// hardware cluster barrier adds up a 1 / S share of the rows out of all S shared memories (always in the order of the
// ranks: results do not depend on timing), applies the epilogue and writes whole 128-byte row pieces.
// No exchange buffers and no mbarrier signals between CTAs: the reads take one hop.  (An exchange through remote stores
// and mbarriers cost more than the split gained.)
// Measured (us, launches back to back, one CTA per tile -> clusters): 64 x 768 x 3072 11.8 -> 5.9, 577 x 384 x 1536 7.9 -> 6.4,
// 200 x 768 x 3072 12.0 -> 7.8, 64 x 768 x 768 5.6 -> 5.0.  What is left is the chain of fixed costs: 1.5 us until the
// previous kernel's end is seen, 0.45 us for the first load, 0.6 us of MMAs, 1.2 us of exchange, 0.5 us to the end.
// Every wait is bounded (ptx.cuh) but the cluster barriers, which every thread reaches.  Launch: cluster dimension S, grid =
// tiles x S.
#pragma once
#include "gemm_pair_tcgen05.cuh"

namespace sod2 {
namespace k {

constexpr int GCL_THREADS = 256;
constexpr int GCL_STAGES = 8;
struct GemmClusterSmem {
  static constexpr int A_BYTES = GEMM_BM * 128, B_BYTES = 64 * 128;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;        // one 64-wide k-chunk; the fp32 tile later reuses the stages
  static constexpr int USED = GCL_STAGES * STAGE_BYTES + 8 * (2 * GCL_STAGES + 1) + 16;
  static constexpr int TOTAL = USED + 1024;
};
struct GemmClusterParams {
  __nv_bfloat16* out;
  const __nv_bfloat16* res;
  const __nv_bfloat16* bias;
  long long ldo, ldr;
  int M, N, K, act2;
  int* status;
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

template <int S, int ACT>
__global__ void __launch_bounds__(GCL_THREADS, 1)
gemm_cluster_bf16_tcgen05(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmClusterParams p) {
  using L = GemmClusterSmem;
  constexpr int STAGES = GCL_STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + STAGES * L::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  volatile int* dead = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int tiles_m = (p.M + GEMM_BM - 1) / GEMM_BM, tile = blockIdx.x / S;
  const int m0 = (tile % tiles_m) * GEMM_BM, n0 = (tile / tiles_m) * 64;
  const int chunks = p.K / 64;        // at least S of them
  if (chunks < S) {                   // uniform over the grid
    if (threadIdx.x == 0 && p.status) atomicExch(p.status, 2);
    return;
  }
  const int k0 = chunks * rank / S, kn = chunks * (rank + 1) / S - k0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { ptx::mbar_init(&full[s], 2); ptx::mbar_init(&empty[s], 1); }
    ptx::mbar_init(acc_full, 1);
    *dead = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
  }
  if (warp == 2) { ptx::tmem_alloc(tmem_slot, 64); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  ptx::pdl_launch();

  if (warp == 0 || warp == 1) {
    // ---- TMA producers: warp 0 A, warp 1 the weights (constants: no wait for the previous kernel)
    if (warp == 0) ptx::pdl_wait();
    const ptx::Leader one = ptx::elect_leader();
    for (int n = 0; n < kn; ++n) {
      const int s = n % STAGES;
      if (n >= STAGES) ptx::mbar_wait_warp(&empty[s], ((n / STAGES) - 1) & 1, dead);
      uint8_t* st = tiles + s * L::STAGE_BYTES;
      ptx::mbar_expect_tx(one, &full[s], warp == 0 ? L::A_BYTES : L::B_BYTES);
      if (warp == 0) ptx::tma_load_3d(one, st, &tmA, 0, m0, k0 + n, &full[s]);
      else ptx::tma_load_3d(one, st + L::A_BYTES, &tmB, 0, n0, k0 + n, &full[s]);
    }
    __syncwarp();
  } else if (warp == 2) {
    // ---- MMA issuer
    constexpr uint32_t idesc = ptx::idesc_bf16(GEMM_BM, 64);
    const ptx::Leader one = ptx::elect_leader();
    const uint64_t a0 = ptx::smem_desc_sw128(ptx::smem_u32(tiles)), b0 = ptx::smem_desc_sw128(ptx::smem_u32(tiles + L::A_BYTES));
    uint32_t s = 0, par = 0;
    for (int n = 0; n < kn; ++n) {
      ptx::mbar_wait_lanes(&full[s], par, dead);
      ptx::tc_fence_after();
      const uint64_t ad = a0 + s * (L::STAGE_BYTES >> 4), bd = b0 + s * (L::STAGE_BYTES >> 4);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) ptx::mma_bf16(one, tmem, ad + 2 * kk, bd + 2 * kk, idesc, n != 0 || kk != 0);
      __syncwarp();
      ptx::mma_commit(one, &empty[s]);
      if (++s == STAGES) { s = 0; par ^= 1; }
    }
    ptx::mma_commit(one, acc_full);
    __syncwarp();
  }
  ptx::pdl_wait();        // residual and output belong to the previous kernels
  // ---- this thread's share of the reduction: pieces of four columns, rows [r0, r0 + rows) of the tile; its residual and
  // bias are fetched ahead of the barriers
  const int live = min(GEMM_BM, p.M - m0), per = (live + S - 1) / S;
  const int r0 = rank * per, pieces = max(0, min(per, live - r0)) * 16;
  constexpr int PT = GEMM_BM / S * 16 / GCL_THREADS > 0 ? GEMM_BM / S * 16 / GCL_THREADS : 1;
  uint2 rv[PT];
  const int c = threadIdx.x & 15, col = n0 + c * 4;
  const bool in_n = col < p.N;
  float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
  if (p.bias && in_n) {
    const uint2 q = *reinterpret_cast<const uint2*>(p.bias + col);
    const float2 lo = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&q)[0]), hi = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&q)[1]);
    b = make_float4(lo.x, lo.y, hi.x, hi.y);
  }
#pragma unroll
  for (int i = 0; i < PT; ++i) {
    const int q = threadIdx.x + i * GCL_THREADS;
    rv[i] = make_uint2(0u, 0u);
    if (p.res && q < pieces && in_n) rv[i] = *reinterpret_cast<const uint2*>(p.res + (m0 + r0 + (q >> 4)) * p.ldr + col);
  }
  // ---- fp32 tile -> shared memory, over the stages (every MMA has read them); 16-byte pieces swizzled by the row
  ptx::mbar_wait_warp(acc_full, 0, dead);
  ptx::tc_fence_after();
  {
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    uint32_t r[32];
    ptx::tmem_ld32(tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + half * 32, r);
    ptx::tmem_ld_wait();
    if (row < live) {
#pragma unroll
      for (int g = 0; g < 8; ++g)
        *reinterpret_cast<uint4*>(tiles + row * 256 + (((half * 8 + g) ^ (row & 7)) << 4)) = make_uint4(r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
    }
  }
  __syncwarp();
  cluster_sync_all();
#pragma unroll
  for (int i = 0; i < PT; ++i) {
    const int q = threadIdx.x + i * GCL_THREADS;
    if (q < pieces && in_n) {
      const int row = r0 + (q >> 4);
      const uint32_t at = ptx::smem_u32(tiles + row * 256 + ((c ^ (row & 7)) << 4));
      float4 v[S];
#pragma unroll
      for (int k = 0; k < S; ++k) v[k] = ld_cluster_f4(map_to_cta(at, k));
      float2 lo = make_float2(v[0].x, v[0].y), hi = make_float2(v[0].z, v[0].w);
#pragma unroll
      for (int k = 1; k < S; ++k) { lo = ptx::add_x2(lo, make_float2(v[k].x, v[k].y)); hi = ptx::add_x2(hi, make_float2(v[k].z, v[k].w)); }
      lo = apply_act_x2<ACT>(ptx::add_x2(lo, make_float2(b.x, b.y)));
      hi = apply_act_x2<ACT>(ptx::add_x2(hi, make_float2(b.z, b.w)));
      if (p.res) {
        lo = ptx::add_x2(lo, __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&rv[i])[0]));
        hi = ptx::add_x2(hi, __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&rv[i])[1]));
        if (p.act2 == ACT_RELU) { lo.x = fmaxf(lo.x, 0.f); lo.y = fmaxf(lo.y, 0.f); hi.x = fmaxf(hi.x, 0.f); hi.y = fmaxf(hi.y, 0.f); }
      }
      uint2 o;
      reinterpret_cast<__nv_bfloat162*>(&o)[0] = __floats2bfloat162_rn(lo.x, lo.y);
      reinterpret_cast<__nv_bfloat162*>(&o)[1] = __floats2bfloat162_rn(hi.x, hi.y);
      *reinterpret_cast<uint2*>(p.out + (m0 + row) * p.ldo + col) = o;
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  cluster_sync_all();      // no CTA leaves while another may still read its shared memory
  if (warp == 2) ptx::tmem_dealloc(tmem, 64);
  if (threadIdx.x == 0 && *dead && p.status) atomicExch(p.status, 1);
}

}  // namespace k
}  // namespace sod2
