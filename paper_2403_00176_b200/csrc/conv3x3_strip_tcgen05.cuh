// 3x3 / stride 1 / pad 1 convolution, 64 -> 64 channels (channels-last, bf16, tcgen05), in vertical strips.
//
// An MMA of N = 64 columns occupies the tensor pipe for 48 cycles, one of N = 192 for 96: with one tap per
// instruction a 64-channel layer cannot pass two thirds of the pipe's rate.  Here an instruction carries the three dy taps of
// one dx: the operand B is [dy = 2 | dy = 1 | dy = 0] x 64 output channels, and the result is what input row i gives to
// the output rows i - 1, i and i + 1, whose accumulators lie side by side in tensor memory (a ring of eight 64-column
// blocks; where the three blocks wrap around its end the instruction is cut in two).  Tensor-core instructions are only
// documented to take effect in the order of issue where accumulator and shape are the same.  Consecutive rows share two of
// their three blocks, so a row's first instruction waits until the row before has completed (its commit passes the turn),
// and within a row every block sees one shape only: no instruction starts a block from zero, the epilogue clears it when it
// has read it (0 + x: the same bits).  The hand-over costs a row about 200 cycles.
// The dx taps are the same rows of shared memory through descriptors whose start address is shifted by a pixel.  So a CTA
// walks down a column of tiles of 128 pixels, every input row is loaded ONCE per strip (one box of 130 pixels, zero-filled
// outside the image = the padding), and takes 12 instructions instead of 36.
//
// Work is the list of all (request, image, column tile, row) tiles in that order; CTA b takes an equal, contiguous
// share, which it walks in segments that do not leave their column.  A segment of L rows costs L + 2 input rows.
//
// Warps: 0 activation and weight TMA, 1 and 3 MMA issuers (alternate rows), 2 staging agent (residual prefetch + output
// stores), 4..19 epilogue: two groups of eight that take alternate rows (a row's accumulator -> activation -> residual -> staging is a
// chain of about 2000 cycles against 1300 of the main loop).
// Measured on B200, 640x480 + 416x416 + 224x608 + 544x320 (6976 tiles): 92 us a layer with one tap per instruction, 57 here, at an
// SM clock of 1.4 GHz (power); one 640x480 image 22 us.  A row takes 1360 cycles (1900 where the window wraps), 1152 of MMAs;
// behind a branch on elect.sync per row it was 1550.  With 192 accumulator columns per input row and the parts added up by the
// epilogue, which needs no order, the epilogue bound (1500 cycles a row).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include "conv3x3_tcgen05.cuh"

namespace sod2 {
namespace k {

constexpr int STRIP_THREADS = 640;
constexpr int STRIP_BLOCKS = 8;              // accumulator ring: 8 x 64 columns
constexpr int STRIP_TAP = 64 * 128;          // one tap of the weights: 64 output channels x 64 input channels
constexpr int STRIP_W = 9 * STRIP_TAP;
constexpr int STRIP_STAGES = 5;              // input rows in shared memory
constexpr int STRIP_NSB = 4;                 // staging buffers (even: a buffer belongs to one epilogue group)
constexpr int STRIP_SMEM = STRIP_W + STRIP_STAGES * C3_A_SLOT + STRIP_NSB * CONV_STAGE_OUT + 256 /*bias*/ +
                           8 * (2 * STRIP_STAGES + 2 * STRIP_BLOCKS + 2 * STRIP_NSB + 3) + 16 + 1024 /*alignment*/;

// One MMA whose descriptors differ from the others' only in their start addresses (low words, in units of 16 bytes).
template <int BLOCKS>
__device__ __forceinline__ void strip_mma(ptx::Leader one, uint32_t d, uint32_t a_lo, uint32_t b_lo) {
  constexpr uint32_t desc_hi = (1024u >> 4) | 1u << 14 | 2u << 29;      // ptx::smem_desc_sw128: row-group stride, version, 128-byte swizzle
  asm volatile(
      "{\n\t.reg .pred q;\n\t.reg .b64 ad, bd;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "mov.b64 ad, {%1, %4};\n\t"
      "mov.b64 bd, {%2, %4};\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], ad, bd, %3, 1;\n\t}"
      ::"r"(d), "r"(a_lo), "r"(b_lo), "n"(ptx::idesc_bf16(128, 64 * BLOCKS)), "n"(desc_hi), "r"(one.on)
      : "memory");
}
// One input row: three dx taps of 64 input channels onto C1 accumulator blocks from d1 and C2 behind the ring's end.
// Everything but the start addresses is a constant: the issuing thread has one MMA's time (96 cycles) for all its
// arithmetic, beside epilogue warps on its scheduler.
template <int C1, int C2>
__device__ __forceinline__ void strip_row(ptx::Leader one, uint32_t d1, uint32_t d2, uint32_t a_lo, uint32_t b_lo) {
  constexpr uint32_t TAP = STRIP_TAP >> 4;
#pragma unroll
  for (int q = 0; q < 12; ++q) {
    const uint32_t a = a_lo + (q >> 2) * 8 + 2 * (q & 3), b = b_lo + (q >> 2) * (3 * TAP) + 2 * (q & 3);
    strip_mma<C1>(one, d1, a, b);
    if constexpr (C2 > 0) strip_mma<C2>(one, d2, a, b + C1 * TAP);
  }
}

// A warp's share of an accumulator block (32 lanes, 32 columns) becomes zero and is handed to the issuers.
__device__ __forceinline__ void strip_hand_over(uint32_t tmem, int blk, int q, int half, int lane, uint64_t* bar) {
  uint32_t zero[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) zero[i] = 0u;
  ptx::tmem_st32(tmem + (static_cast<uint32_t>(q * 32) << 16) + blk * 64 + half * 32, zero);
  ptx::tmem_st_wait();
  ptx::tc_fence_before();
  __syncwarp();
  if (lane == 0) ptx::mbar_arrive(bar);
}

// B.tx: {64, W, H, N}, box {64, 130, 1, 1};  tmW: k-chunk view {64, 64, 9} of the weights in (dy, dx, ci) order, box
// {64, 64, 1};  B.to / B.tr: {64, W, H, N}, box {64, 128, 1, 1}.  B.tile_start as for the row-halo kernel.
// GAP: p.gap_sum receives the channel sums.  The conversions to fp64 then bound the epilogue (a layer of 32 gated images of 112 x 112
// takes 27 us with them and 18 without), but the pooling passes over three tensors of 51 MB that they replace take longer: the
// gated network of 32 images 785 -> 757 us.  A template parameter because the code for them costs registers: one image of 227 x
// 341 111.2 -> 113.0 us with it everywhere.
template <int ACT, bool HASRES, bool GAP>
__global__ void __launch_bounds__(STRIP_THREADS, 1)
conv3x3_strip_bf16_tcgen05(const __grid_constant__ Conv3Batch B, const __grid_constant__ CUtensorMap tmW, ConvParams p) {
  constexpr int NSB = STRIP_NSB, NB = STRIP_BLOCKS, ST = STRIP_STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* wres = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* rows = wres + STRIP_W;
  uint8_t* out_stage = rows + ST * C3_A_SLOT;
  float* bias_s = reinterpret_cast<float*>(out_stage + NSB * CONV_STAGE_OUT);   // [64]
  uint64_t* full = reinterpret_cast<uint64_t*>(bias_s + 64);
  uint64_t* empty = full + ST;
  uint64_t* tmem_full = empty + ST;
  uint64_t* tmem_empty = tmem_full + NB;
  uint64_t* res_full = tmem_empty + NB;
  uint64_t* stage_ready = res_full + NSB;
  uint64_t* w_full = stage_ready + NSB;
  uint64_t* turn = w_full + 1;             // [2] the other issuer has issued its row
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(turn + 2);
  volatile int* dead = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) { ptx::mbar_init(&full[s], 1); ptx::mbar_init(&empty[s], 1); }
    for (int b = 0; b < NB; ++b) { ptx::mbar_init(&tmem_full[b], 1); ptx::mbar_init(&tmem_empty[b], 8); }
    for (int b = 0; b < NSB; ++b) { ptx::mbar_init(&res_full[b], 1); ptx::mbar_init(&stage_ready[b], 8); }
    ptx::mbar_init(w_full, 1);
    for (int b = 0; b < 2; ++b) ptx::mbar_init(&turn[b], 1);
    *dead = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    ptx::prefetch_tmap(&tmW);
    for (int r = 0; r < B.n_req; ++r) {
      ptx::prefetch_tmap(&B.tx[r]);
      ptx::prefetch_tmap(&B.to[r]);
      if (HASRES) ptx::prefetch_tmap(&B.tr[r]);
    }
  }
  if (threadIdx.x >= 64 && threadIdx.x < 128) bias_s[threadIdx.x - 64] = p.bias ? __bfloat162float(p.bias[threadIdx.x - 64]) : 0.0f;
  if (warp == 3) { ptx::tmem_alloc(tmem_slot, 512); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the weights do not depend on the previous kernel; tap (dy, dx) goes to slot dx * 3 + 2 - dy
  if (warp == 0) {
    const ptx::Leader one = ptx::elect_leader();
    ptx::mbar_expect_tx(one, w_full, STRIP_W);
    for (int dx = 0; dx < 3; ++dx)
      for (int dy = 2; dy >= 0; --dy) ptx::tma_load_3d(one, wres + (dx * 3 + 2 - dy) * STRIP_TAP, &tmW, 0, 0, dy * 3 + dx, w_full);
  }
  // the accumulator ring starts from zero: each epilogue warp clears its share of its group's blocks
  if (warp >= 4)
    for (int blk = (warp - 4) >> 3; blk < NB; blk += 2) strip_hand_over(tmem, blk, warp & 3, ((warp - 4) & 7) >> 2, lane, &tmem_empty[blk]);
  ptx::pdl_wait();
  ptx::pdl_launch();
  int total = B.tile_start[B.n_req];
  if (p.n_img_ptr) {   // gated sub-batch (single request): the image count is on the device
    const int n_img = min(p.n_img, max(0, p.cnt_a + p.cnt_b * static_cast<int>(*p.n_img_ptr)));
    total = ((B.Wo[0] + 127) / 128) * B.Ho[0] * n_img;
  }
  const int begin = static_cast<int>(static_cast<long long>(total) * blockIdx.x / gridDim.x);
  const int end = static_cast<int>(static_cast<long long>(total) * (blockIdx.x + 1) / gridDim.x);

  // tile index -> request, image, row, first pixel; rows of a column vary fastest
  auto decode = [&](int t, int* img, int* row, int* w0) -> int {
    int r = 0;
    while (r + 1 < B.n_req && t >= B.tile_start[r + 1]) ++r;
    t -= B.tile_start[r];
    const int per_img = ((B.Wo[r] + 127) / 128) * B.Ho[r];
    *img = t / per_img;
    const int rem = t - *img * per_img;
    const int wt = rem / B.Ho[r];
    *row = rem - wt * B.Ho[r];
    *w0 = wt * 128;
    return r;
  };

  if (warp == 0) {
    {
      // ---- input rows: a segment's L output rows need the L + 2 rows around them
      const ptx::Leader one = ptx::elect_leader();
      int n = 0;
      for (int t = begin; t < end;) {
        int img, row, w0;
        const int rq = decode(t, &img, &row, &w0);
        const int len = min(end - t, B.Ho[rq] - row);
        if (p.in_ids) img = p.in_ids[img];
        for (int i = row - 1; i <= row + len; ++i, ++n) {
          const int s = n % ST;
          if (n >= ST) ptx::mbar_wait_warp(&empty[s], ((n / ST) - 1) & 1, dead);
          ptx::mbar_expect_tx(one, &full[s], C3_A_BYTES);
          ptx::tma_load_4d(one, rows + s * C3_A_SLOT, &B.tx[rq], 0, w0 - 1, i, img, &full[s]);
        }
        t += len;
      }
    }
  } else if (warp == 1 || warp == 3) {
    {
      // ---- MMA issuers: rows alternate between the leading lanes of two warps.  A row starts when the row before has completed: its issuer
      // commits to this one's `turn`, so the commit of an output row also covers what the other thread issued for it.  The
      // next row's thread has done its address arithmetic and its other waits by then.  (A thread may wait on `full` and
      // `tmem_empty` for its own rows only: its row n - 2 was issued after every earlier row had seen its barriers, so at row
      // n each barrier is at most one phase away from the one waited for.  A warp's other lanes have left its waits before
      // it commits, so they are no further behind.)
      // Output row o of the segment accumulates in block (j + o) % 8; input row ii (counted from the row above the segment)
      // gives to the output rows ii - 2 (dy = 2), ii - 1 and ii, as far as they belong to the segment.
      ptx::mbar_wait_lanes(w_full, 0, dead);
      const uint64_t wdesc = ptx::smem_desc_sw128(ptx::smem_u32(wres));
      const ptx::Leader one = ptx::elect_leader();
      const auto mma_commit = [&](uint64_t* bar) { ptx::mma_commit(one, bar); };
      const int me = warp == 1 ? 0 : 1;
      int n = 0, j = 0;
      for (int t = begin; t < end;) {
        int img, row, w0;
        const int rq = decode(t, &img, &row, &w0);
        const int len = min(end - t, B.Ho[rq] - row);
        for (int ii = 0; ii < len + 2; ++ii, ++n) {
          const int s = n % ST;
          if ((n & 1) != me) continue;
          const bool fresh = ii < len;
          const int lo = max(ii - 2, 0), cnt = min(ii, len - 1) - lo + 1;
          const int b0 = (j + lo) % NB;
          const int c1 = min(cnt, NB - b0), c2 = cnt - c1;            // blocks before and behind the ring's end
          const uint64_t wb = wdesc + (lo - (ii - 2)) * (STRIP_TAP >> 4);
          const uint32_t d1 = tmem + b0 * 64;
          if (fresh) ptx::mbar_wait_lanes(&tmem_empty[(j + ii) % NB], ((j + ii) / NB) & 1, dead);
          ptx::mbar_wait_lanes(&full[s], (n / ST) & 1, dead);
          const uint64_t ad = ptx::smem_desc_sw128(ptx::smem_u32(rows + s * C3_A_SLOT));
          const uint32_t a_lo = static_cast<uint32_t>(ad), b_lo = static_cast<uint32_t>(wb);
          uint64_t* const done = &tmem_full[(j + ii + NB - 2) % NB];
          if (n > 0) ptx::mbar_wait_lanes(&turn[me], me ? (n >> 1) & 1 : ((n >> 1) - 1) & 1, dead);
          ptx::tc_fence_after();
          if (c1 == 3) strip_row<3, 0>(one, d1, tmem, a_lo, b_lo);
          else
            switch (c1 * 4 + c2) {
              case 9: strip_row<2, 1>(one, d1, tmem, a_lo, b_lo); break;
              case 6: strip_row<1, 2>(one, d1, tmem, a_lo, b_lo); break;
              case 8: strip_row<2, 0>(one, d1, tmem, a_lo, b_lo); break;
              case 5: strip_row<1, 1>(one, d1, tmem, a_lo, b_lo); break;
              case 4: strip_row<1, 0>(one, d1, tmem, a_lo, b_lo); break;
            }
          __syncwarp();
          mma_commit(&turn[me ^ 1]);
          mma_commit(&empty[s]);
          if (ii >= 2) mma_commit(done);
        }
        j += len;
        t += len;
      }
    }
  } else if (warp == 2) {
    {
      // ---- staging agent: unit u = this CTA's u-th tile, in buffer u % NSB.  prepare(u) hands the buffer to the
      // epilogue warps: with a residual it is TMA-loaded into the buffer (updated in place), otherwise a plain arrive.
      // The buffer of unit u - 1 is free for unit u + NSB - 1 once its store, issued one unit ago, has read it.
      // Both walk the tiles with a cursor: decoding every tile (divisions, indexed parameters) made this thread the
      // slowest of the kernel.
      const int U = end - begin;
      struct Cursor { int t, rq, img, row, w0, left; };
      auto open = [&](Cursor& c, const int* ids) {
        c.left = 0;
        if (c.t >= end) return;
        c.rq = decode(c.t, &c.img, &c.row, &c.w0);
        c.left = min(end - c.t, B.Ho[c.rq] - c.row);
        if (ids) c.img = ids[c.img];
      };
      auto next = [&](Cursor& c, const int* ids) {
        ++c.t;
        ++c.row;
        if (--c.left == 0) open(c, ids);
      };
      Cursor in{begin, 0, 0, 0, 0, 0}, out{begin, 0, 0, 0, 0, 0};
      if (HASRES) open(in, p.res_ids);
      open(out, p.out_ids);
      auto prepare = [&](int bsel) {
        if (ptx::elect_one()) {
          if (HASRES) {
            ptx::mbar_expect_tx(&res_full[bsel], CONV_STAGE_OUT);
            ptx::tma_load_4d(out_stage + bsel * CONV_STAGE_OUT, &B.tr[in.rq], 0, in.w0, in.row, in.img, &res_full[bsel]);
          } else {
            ptx::mbar_arrive(&res_full[bsel]);
          }
        }
        __syncwarp();
        if (HASRES) next(in, p.res_ids);
      };
      for (int u = 0; u < NSB && u < U; ++u) prepare(u);
      for (int u = 0; u < U; ++u) {
        const int bsel = u % NSB;
        ptx::mbar_wait_lanes(&stage_ready[bsel], (u / NSB) & 1, dead);
        if (ptx::elect_one()) {        // (always the same lane: bulk groups belong to a thread)
          tma_store_4d(&B.to[out.rq], out_stage + bsel * CONV_STAGE_OUT, 0, out.w0, out.row, out.img);
          bulk_commit();
          if (u >= 1 && u + NSB - 1 < U) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        }
        __syncwarp();
        if (u >= 1 && u + NSB - 1 < U) prepare((u + NSB - 1) % NSB);
        next(out, p.out_ids);
      }
      if (ptx::elect_one()) bulk_wait0();
    }
  } else if (warp >= 4) {
    // ---- epilogue: group g (eight warps) takes the tiles j = g, g + 2, ...; warp (q, half) of a group owns TMEM lanes
    // 32q..32q+31 and a 32-column half, a thread one pixel
    const int g = (warp - 4) >> 3, e = (warp - 4) & 7;
    const int q = warp & 3, half = e >> 2;
    const int et = threadIdx.x - 128 - g * 256;
    const int row = q * 32 + lane;
    const float relu2_floor = p.act2 == ACT_RELU ? 0.0f : -INFINITY;
    // sums of the stored values of one image (p.gap_sum): kept by the threads while the CTA's tiles stay in it
    [[maybe_unused]] double gap0 = 0.0, gap1 = 0.0;
    [[maybe_unused]] int gap_img = -1;
    auto group_bar = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + g) : "memory"); };
    for (int j = g; j < end - begin; j += 2) {
      const int blk = j % NB, bsel = j % NSB;
      ptx::mbar_wait_warp(&tmem_full[blk], (j / NB) & 1, dead);
      ptx::tc_fence_after();
      uint32_t r[32];
      ptx::tmem_ld32(tmem + (static_cast<uint32_t>(q * 32) << 16) + blk * 64 + half * 32, r);
      ptx::tmem_ld_wait();
      strip_hand_over(tmem, blk, q, half, lane, &tmem_empty[blk]);
      float v[32];
      bias_act32<ACT>(v, r, bias_s + half * 32);
      uint8_t* obase = out_stage + bsel * CONV_STAGE_OUT + row * 128;
      ptx::mbar_wait_warp(&res_full[bsel], (j / NSB) & 1, dead);
      conv_pixel_to_staging<HASRES>(v, obase, row, half, relu2_floor);
      if constexpr (GAP) {
        group_bar();                               // every row of the tile is in the staging buffer
        int img, trow, w0;
        const int rq = decode(begin + j, &img, &trow, &w0);
        const int wo = B.Wo[rq];
        if (img != gap_img) {
          if (gap_img >= 0) gap_flush(gap0, gap1, et, p.gap_sum + static_cast<long long>(p.out_ids ? p.out_ids[gap_img] : gap_img) * 64);
          gap_img = img;
          gap0 = gap1 = 0.0;
        }
        gap_add_tile(out_stage + bsel * CONV_STAGE_OUT, et, &gap0, &gap1, [&](int px) { return w0 + px < wo; });
      }
      ptx::fence_proxy_async();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&stage_ready[bsel]);
    }
    if constexpr (GAP) {
      if (gap_img >= 0) gap_flush(gap0, gap1, et, p.gap_sum + static_cast<long long>(p.out_ids ? p.out_ids[gap_img] : gap_img) * 64);
    }
  }
  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 3) ptx::tmem_dealloc(tmem, 512);
  if (threadIdx.x == 0 && *dead && p.status) atomicExch(p.status, 1);
}

}  // namespace k
}  // namespace sod2
