// 3x3 / stride 1 / pad 1 convolution of images narrower than the row tiles, "halo patch" form (channels-last, bf16, tcgen05).
//
// The implicit-GEMM kernel (conv_tcgen05.cuh) fetches a 128-pixel tile nine times per 64 input channels, once per tap:
// 16 KB of activations and 16 KB of weights for every 128 x 128 x 64 product, which the tensor pipe does in 290 cycles and
// L2 -> shared memory in 420.  Here one box per kernel row dy and 64 channels does for the three taps of that row: the
// TH lines of TW + 2 pixels that a patch of TW x TH output pixels needs, zero-filled outside the image (= the padding), which
// lie in shared memory as rows of 128 bytes with pitch P = TW + 2.  Row m = y * P + x of the MMA is output pixel (y, x); tap dx
// reads the same buffer dx rows further down, which is a shift of the operand descriptor's start address.  The two rows per
// patch line with x >= TW are computed and dropped.  What is left to fetch per tap is the weights and a third of the patch.
// K is summed in the order (dy, 64-channel chunk, dx, channel), as in the implicit-GEMM and row kernels: the same sums in the
// same order, so that the three forms give the same bits.
// Measured on B200, implicit GEMM -> here, 32 images of 56 x 56 to 128 channels: 64 channels 21.3 -> 17.0 us, 128 32.3 -> 25.6, 256
// 58.8 -> 47.8, 512 122 -> 99 (1200 TFLOP/s); bound by the MMAs and the 85 bytes per cycle that a stage of 64 KB takes in beside them.
// (A patch fetched once per 64 channels, K in the order (chunk, dy, dx): 24.7 us at 128 channels, 27.0 against 26.5 at 512
// channels of 14 x 14, and other bits.)
//
// Warps (384 threads, persistent, 1 CTA/SM): 0 activation TMA, 1 weight TMA (constant: starts before the previous kernel has
// ended), 3 MMA issuer, 4..11 epilogue (as in conv_tcgen05.cuh; the staging tile is packed to TW pixels per line).
// Channel tiles vary fastest, so that a CTA knows its first weights before the image count.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include "conv_tcgen05.cuh"

namespace sod2 {
namespace k {

constexpr int HALO_BN = 128;
constexpr int HALO_MAX_ROWS = 128;                    // (TW + 2) * TH: the two rows read behind them end up in dropped rows only
constexpr int HALO_A_BYTES = HALO_MAX_ROWS * 128;
constexpr int HALO_B_BYTES = 3 * HALO_BN * 128;       // the dx taps of one (dy, 64-channel chunk)
constexpr int HALO_STAGE = HALO_A_BYTES + HALO_B_BYTES;
constexpr int HALO_STAGES = 3;
constexpr int HALO_SMEM = HALO_STAGES * HALO_STAGE + 2 * CONV_STAGE_OUT + 2 * HALO_BN * 4 /*bias*/ + 8 * (2 * HALO_STAGES + 6) + 16 + 1024 /*alignment*/;
static_assert(HALO_SMEM <= 227 * 1024, "shared memory of a CTA");

// tmX: {Cin, W, H, N}, box {64, TW + 2, TH, 1};  tmW: k-chunk view {64, Cout, K/64} of the weights in (dy, chunk, dx, ci)
// order, box {64, 128, 3};  tmOut / tmRes: {Cout, W, H, N}, box {64, TW, TH, 1}.  (p.TW + 2) * p.TH <= HALO_MAX_ROWS.
template <int ACT, bool HASRES>
__global__ void __launch_bounds__(CONV_THREADS, 1)
conv3x3_halo_bf16_tcgen05(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                          const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ CUtensorMap tmRes, ConvParams p) {
  constexpr int ST = HALO_STAGES, BN = HALO_BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));   // weights, then the patch
  uint8_t* out_stage = stages + ST * HALO_STAGE;
  float* bias_s = reinterpret_cast<float*>(out_stage + 2 * CONV_STAGE_OUT);   // [2][128]
  uint64_t* full = reinterpret_cast<uint64_t*>(bias_s + 2 * BN);
  uint64_t* empty = full + ST;
  uint64_t* tmem_full = empty + ST;       // [2]
  uint64_t* tmem_empty = tmem_full + 2;   // [2]
  uint64_t* res_full = tmem_empty + 2;    // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(res_full + 2);
  volatile int* dead = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) { ptx::mbar_init(&full[s], 2); ptx::mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&tmem_full[b], 1); ptx::mbar_init(&tmem_empty[b], 8); ptx::mbar_init(&res_full[b], 1); }
    *dead = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    ptx::prefetch_tmap(&tmX);
    ptx::prefetch_tmap(&tmW);
    ptx::prefetch_tmap(&tmOut);
    if (HASRES) ptx::prefetch_tmap(&tmRes);
  }
  if (warp == 3) { ptx::tmem_alloc(tmem_slot, 2 * BN); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  ptx::pdl_launch();

  const int P = p.TW + 2;
  const int tiles_n = p.Cout / BN;
  const int cchunks = p.Cin / 64;
  const int groups = 3 * cchunks;                    // stages per tile, (dy, chunk): a multiple of three
  const int tiles_w = (p.Wo + p.TW - 1) / p.TW, tiles_h = (p.Ho + p.TH - 1) / p.TH;
  auto weight_box = [&](ptx::Leader one, int s, int n0, int g) {
    ptx::mbar_expect_tx(one, &full[s], HALO_B_BYTES);
    ptx::tma_load_3d(one, stages + s * HALO_STAGE, &tmW, 0, n0, g * 3, &full[s]);
  };
  // the first weight stages do not depend on the previous kernel
  if (warp == 1) {
    const ptx::Leader one = ptx::elect_leader();
    for (int g = 0; g < ST; ++g) weight_box(one, g, (static_cast<int>(blockIdx.x) % tiles_n) * BN, g);   // groups >= 3 = ST
  }
  ptx::pdl_wait();
  int n_img = p.n_img;
  if (p.n_img_ptr) n_img = min(p.n_img, max(0, p.cnt_a + p.cnt_b * static_cast<int>(*p.n_img_ptr)));
  const int num_tiles = tiles_n * tiles_w * tiles_h * n_img;
  auto decode = [&](int t, int* n0, int* img, int* ho0, int* wo0) {
    const int tp = t / tiles_n;
    *n0 = (t - tp * tiles_n) * BN;
    *img = tp / (tiles_w * tiles_h);
    const int r = tp - *img * (tiles_w * tiles_h);
    *ho0 = (r / tiles_w) * p.TH;
    *wo0 = (r % tiles_w) * p.TW;
  };

  if (warp == 0) {
    // ---- activation patches
    const uint32_t bytes = P * p.TH * 128;
    const ptx::Leader one = ptx::elect_leader();
    if (static_cast<int>(blockIdx.x) >= num_tiles && lane < ST) ptx::mbar_arrive(&full[lane]);   // see the weights
    int n = 0;
    for (int t = blockIdx.x; t < num_tiles; t += gridDim.x) {
      int n0, img, ho0, wo0;
      decode(t, &n0, &img, &ho0, &wo0);
      if (p.in_ids) img = p.in_ids[img];
      for (int dy = 0; dy < 3; ++dy)
        for (int cc = 0; cc < cchunks; ++cc, ++n) {
          const int s = n % ST;
          if (n >= ST) ptx::mbar_wait_warp(&empty[s], ((n / ST) - 1) & 1, dead);
          ptx::mbar_expect_tx(one, &full[s], bytes);
          ptx::tma_load_4d(one, stages + s * HALO_STAGE + HALO_B_BYTES, &tmX, cc * 64, wo0 - 1, ho0 - 1 + dy, img, &full[s]);
        }
    }
  } else if (warp == 1) {
    // ---- weights
    if (static_cast<int>(blockIdx.x) >= num_tiles) {
      for (int s = 0; s < ST; ++s) ptx::mbar_wait_warp(&full[s], 0, dead);    // nothing may land after the CTA has gone
    }
    const ptx::Leader one = ptx::elect_leader();
    int n = 0;
    for (int t = blockIdx.x; t < num_tiles; t += gridDim.x) {
      const int n0 = (t % tiles_n) * BN;
      for (int g = 0; g < groups; ++g, ++n) {
        if (n < ST) continue;
        const int s = n % ST;
        ptx::mbar_wait_warp(&empty[s], ((n / ST) - 1) & 1, dead);
        weight_box(one, s, n0, g);
      }
    }
  } else if (warp == 3) {
    // ---- MMA issuer: the whole warp in step, one lane issues (ptx::Leader)
    constexpr uint32_t idesc = ptx::idesc_bf16(128, BN);
    const ptx::Leader one = ptx::elect_leader();
    // straight-line code with the descriptors at hand: a stage is twelve MMAs and nothing but a wait and a commit beside them.
    // (Weights by single taps, or patches that stay for the three kernel rows, fetch less or finer; the arithmetic and the
    // waits they need cost more: 32 images of 512 channels 31.8 us, 256 channels 29.3)
    static_assert(ST == 3, "a tile is a multiple of three stages");
    const uint64_t b0 = ptx::smem_desc_sw128(ptx::smem_u32(stages)), a0 = ptx::smem_desc_sw128(ptx::smem_u32(stages + HALO_B_BYTES));
    uint32_t par = 0;
    int j = 0;
    for (int t = blockIdx.x; t < num_tiles; t += gridDim.x, ++j) {
      const int acc = j & 1;
      if (j >= 2) ptx::mbar_wait_lanes(&tmem_empty[acc], ((j >> 1) - 1) & 1, dead);
      const uint32_t d = tmem + acc * BN;
      for (int r = 0; r < cchunks; ++r, par ^= 1) {
#pragma unroll
        for (int s = 0; s < ST; ++s) {
          const uint64_t ad = a0 + s * (HALO_STAGE >> 4), bd = b0 + s * (HALO_STAGE >> 4);
          ptx::mbar_wait_lanes(&full[s], par, dead);
          ptx::tc_fence_after();
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) ptx::mma_bf16(one, d, ad + 8 * dx + 2 * kk, bd + dx * (BN * 128 / 16) + 2 * kk, idesc, (r | s | dx | kk) != 0);
          __syncwarp();
          ptx::mma_commit(one, &empty[s]);
        }
      }
      ptx::mma_commit(one, &tmem_full[acc]);
    }
  } else if (warp >= 4) {
    // ---- epilogue warps 4..11: passes of 64 channels through two staging buffers (conv_tcgen05.cuh)
    const int e = warp - 4;
    const int q = warp & 3;
    const int half = e >> 2;          // which 32-channel half of the 64-channel pass
    const int et = threadIdx.x - 128; // 0..255
    const int m = q * 32 + lane;      // row of the accumulator
    const int my = m / P, mx = m - my * P;
    const bool live = mx < p.TW && my < p.TH;
    const int row = my * p.TW + mx;   // pixel of the packed tile
    const uint32_t tile_bytes = p.TW * p.TH * 128;
    const float relu2_floor = p.act2 == ACT_RELU ? 0.0f : -INFINITY;
    int j = 0, u = 0;
    auto load_bias = [&](int t) -> float {
      return (p.bias && et < BN && t < num_tiles) ? __bfloat162float(p.bias[(t % tiles_n) * BN + et]) : 0.0f;
    };
    auto load_res = [&](int v, int np, int ho0, int wo0, int img) {
      ptx::mbar_expect_tx(&res_full[v & 1], tile_bytes);
      ptx::tma_load_4d(out_stage + (v & 1) * CONV_STAGE_OUT, &tmRes, np, wo0, ho0, p.res_ids ? p.res_ids[img] : img, &res_full[v & 1]);
    };
    float bias_next = load_bias(blockIdx.x);
    if (HASRES && et == 0 && static_cast<int>(blockIdx.x) < num_tiles) {
      int n0, img, ho0, wo0;
      decode(blockIdx.x, &n0, &img, &ho0, &wo0);
      load_res(0, n0, ho0, wo0, img);
    }
    for (int t = blockIdx.x; t < num_tiles; t += gridDim.x, ++j) {
      const int acc = j & 1;
      int n0, img, ho0, wo0;
      decode(t, &n0, &img, &ho0, &wo0);
      const int img_o = p.out_ids ? p.out_ids[img] : img;
      float* bias_t = bias_s + (j & 1) * BN;
      if (et < BN) bias_t[et] = bias_next;
      bias_next = load_bias(t + gridDim.x);
      conv_epi_bar();                              // the bias of this tile is written
      ptx::mbar_wait_warp(&tmem_full[acc], (j >> 1) & 1, dead);
      ptx::tc_fence_after();
#pragma unroll 1
      for (int ps = 0; ps < BN / 64; ++ps, ++u) {
        const int np = n0 + ps * 64;
        uint8_t* stage = out_stage + (u & 1) * CONV_STAGE_OUT;
        uint8_t* obase = stage + row * 128;
        uint32_t r[32];
        ptx::tmem_ld32(tmem + (static_cast<uint32_t>(q * 32) << 16) + acc * BN + ps * 64 + half * 32, r);
        ptx::tmem_ld_wait();
        if (ps == BN / 64 - 1) {
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&tmem_empty[acc]);
        }
        float v[32];
        bias_act32<ACT>(v, r, bias_t + ps * 64 + half * 32);
        if constexpr (HASRES) ptx::mbar_wait_warp(&res_full[u & 1], (u >> 1) & 1, dead);
        if (live) conv_pixel_to_staging<HASRES>(v, obase, row, half, relu2_floor);
        ptx::fence_proxy_async();
        if (et == 0) bulk_wait_read0();              // the pass before has left its buffer
        conv_epi_bar();
        if (et == 0) {
          if constexpr (HASRES) {
            if (ps + 1 < BN / 64) {
              load_res(u + 1, np + 64, ho0, wo0, img);
            } else if (t + static_cast<int>(gridDim.x) < num_tiles) {
              int n1, img1, ho1, wo1;
              decode(t + gridDim.x, &n1, &img1, &ho1, &wo1);
              load_res(u + 1, n1, ho1, wo1, img1);
            }
          }
          tma_store_4d(&tmOut, stage, np, wo0, ho0, img_o);
          bulk_commit();
        }
        if (p.gap_sum) {
          const uint32_t inv = 65536u / p.TW + 1;    // px / TW for px < 128 and TW <= 126: exact
          gap_accumulate_tile(stage, et, p.gap_sum + static_cast<long long>(img_o) * p.Cout + np, [&](int px) {
            const int y = static_cast<int>((px * inv) >> 16);
            return y < p.TH && ho0 + y < p.Ho && wo0 + px - y * p.TW < p.Wo;
          });
        }
      }
    }
    if (et == 0) bulk_wait0();
  }
  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 3) ptx::tmem_dealloc(tmem, 2 * BN);
  if (threadIdx.x == 0 && *dead && p.status) atomicExch(p.status, 1);
}

}  // namespace k
}  // namespace sod2
