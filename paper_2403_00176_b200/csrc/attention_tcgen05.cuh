// Fused attention group on tcgen05 / TMEM for packed variable-length requests, head dim 64:
//   O = softmax(Q K^T * scale) V  per (request, head), bf16 in / fp32 accumulate / bf16 out.
// The score and probability tensors never reach global memory (the fusion argument of Section 4.2).
// A work item is 128 query rows of one (request, head); it walks the request's keys in blocks of 64:
//   S_n = Q K_n^T          tcgen05.mma, M=128, N=64, K=64; Q and K_n are K-major TMA tiles
//   P_n = exp2(S_n*c - m)  one thread per query row: its 64 scores go from TMEM into registers, P_n back as packed bf16
//                          pairs into 32 columns of TMEM
//   O  += P_n V_n          tcgen05.mma with the A operand in TMEM, M=128, N=64, K = the block's live keys; V_n is the
//                          natural [key, d] tile, used as an MN-major B operand
//   (O *= corr)            only when a block's maximum moves the exponent reference by more than 2^8
// The special-function pipe bounds it: 128 x 64 exponentials are 512 cycles of an SM.  Everything else is arranged so
// that the pipe waits for nothing: two CTAs per SM (while one reads scores, reduces the row maximum or writes its output,
// the other has the pipe); S and P double buffered, so that a score tile (600 to 1000 cycles from the release of its
// buffer to the softmax warps seeing it) is under way a whole block ahead -- 64 keys are what TMEM holds twice at two
// CTAs per SM; no exchange between threads (with two threads per row, the scores read twice and the row maximum exchanged
// through shared memory, 128 keys took 3600 cycles of an SM); two scores per instruction where the FMA pipe has the form.
// The CTAs are persistent and take items back and forth, longest request first (16 requests of 238 to 780 tokens, 6 heads:
// the busiest CTA has 23 blocks, round robin 26; at 0.7 of the tokens 11 against 15); phases run on from item to item: the
// softmax warps go straight on to the next item's first block and write an item's output between that block's
// exponentials and its P, by when the last product has landed.
// Q, K, V are 2-D tensor maps over the packed [tokens, row stride] buffers; a tile that runs past a
// request's rows reads the next request's rows (finite data) or zeros past the end of the buffer, and
// those keys are masked to -inf before the softmax; query rows past the request are never written.
// Warps: 0..3 softmax (warp w owns TMEM lanes 32w..32w+31), 4 loads Q and K, 5 issues S = Q K^T,
// 6 issues O += P V, 7 loads V (a thread of its own: V waits for products, K must not wait with it).
// Every wait is bounded (ptx.cuh).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include "ptx.cuh"

namespace sod2 {
namespace k {

constexpr int ATC_MAX_REQ = 64;
constexpr int ATC_THREADS = 256;
struct AtcReq {
  int L;                       // tokens of this request
  int q_row, k_row, v_row;     // first row of the request in the Q / K / V tensor maps
  long long o_off;             // element offset of the request's output view
};
struct AtcParams {
  __nv_bfloat16* o;
  int n_req, H;
  int q_col, k_col, v_col;     // column of head 0 in the Q / K / V tensor maps
  int q_hs, k_hs, v_hs;        // head strides in columns
  int o_ts, o_hs;              // output token / head strides in elements (multiples of 8)
  float scale_log2e;
  int* status;
  int tile_start[ATC_MAX_REQ + 1];   // prefix sum of ceil(L / 128); requests in descending L
  AtcReq r[ATC_MAX_REQ];
};

constexpr int ATC_KB = 64;                // keys per block
constexpr int ATC_ST = 4;                 // K and V stages
constexpr int ATC_Q_BYTES = 128 * 128;    // 128 rows x 64 bf16
constexpr int ATC_KV_BYTES = ATC_KB * 128;   // 64 keys x 64 bf16
constexpr int ATC_SMEM = 2 * ATC_Q_BYTES + 2 * ATC_ST * ATC_KV_BYTES + 1024 /*align*/ + 256 /*barriers*/ +
                         ATC_MAX_REQ * 28 /*request table*/;
constexpr uint32_t ATC_TMEM_S = 0, ATC_TMEM_O = 128, ATC_TMEM_P = 192;   // columns: scores [2 x 64], output, probabilities [2 x 32 packed bf16 pairs]

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// maximum of 32 scores, three operands per instruction
__device__ __forceinline__ float atc_max32(float mx, const uint32_t* s) {
  float mx0 = mx, mx1 = -INFINITY;
#pragma unroll
  for (int e = 0; e < 32; e += 4) {
    mx0 = fmaxf(fmaxf(mx0, __uint_as_float(s[e])), __uint_as_float(s[e + 1]));
    mx1 = fmaxf(fmaxf(mx1, __uint_as_float(s[e + 2])), __uint_as_float(s[e + 3]));
  }
  return fmaxf(mx0, mx1);
}
// 32 probabilities 2^(s*c - m*c) as 16 packed bf16 pairs, their sum added to l: the scale rides in the FMA that feeds ex2
__device__ __forceinline__ void atc_exp32(const uint32_t* s, uint32_t* pk, float2 c2, float2 mc2, float2* l) {
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    const float2 t = ptx::fma_x2(make_float2(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), c2, mc2);
    const float2 q = make_float2(ex2_approx(t.x), ex2_approx(t.y));
    *l = ptx::add_x2(*l, q);
    const __nv_bfloat162 pb = __floats2bfloat162_rn(q.x, q.y);
    pk[e >> 1] = *reinterpret_cast<const uint32_t*>(&pb);
  }
}

__global__ void __launch_bounds__(ATC_THREADS, 2)
attention_tcgen05_bf16(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AtcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sQ = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));   // [2], also the output staging
  uint8_t* sK = sQ + 2 * ATC_Q_BYTES;       // [4]
  uint8_t* sV = sK + ATC_ST * ATC_KV_BYTES; // [4]
  // n counts the CTA's key blocks, i its items
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + ATC_ST * ATC_KV_BYTES);
  uint64_t* q_full = bars;            // [2] Q of item i landed
  uint64_t* q_free = bars + 2;        // [2] item i's output has left the buffer
  uint64_t* s_full = bars + 4;        // [2] S_n done
  uint64_t* s_free = bars + 6;        // [2] S_n is in registers
  uint64_t* p_full = bars + 8;        // [2] P_n written
  uint64_t* o_full = bars + 10;       // [2] O_n done: the P columns are free
  uint64_t* k_full = bars + 12;       // [4] K_n landed
  uint64_t* k_free = bars + 16;       // [4] S_n done
  uint64_t* v_full = bars + 20;       // [4] V_n landed
  uint64_t* v_free = bars + 24;       // [4] O_n done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 28);
  volatile int* dead = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // item = tile * H + head, tiles ordered by descending request length; called by whole warps
  const int items = p.tile_start[p.n_req] * p.H;
  // (from a copy of the request table in shared memory: lanes with different addresses serialise in the constant cache)
  AtcReq* reqs = reinterpret_cast<AtcReq*>(bars + 32);
  int* starts = reinterpret_cast<int*>(reqs + ATC_MAX_REQ);
  for (int t = threadIdx.x; t < ATC_MAX_REQ; t += ATC_THREADS) {
    starts[t] = t < p.n_req ? p.tile_start[t] : 0x7fffffff;
    if (t < p.n_req) reqs[t] = p.r[t];
  }
  // the CTA's i-th item: rounds go back and forth, so that who has the longest item of one round has the shortest of the next
  auto nth_item = [&](int i) { return i * static_cast<int>(gridDim.x) + static_cast<int>((i & 1) ? gridDim.x - 1 - blockIdx.x : blockIdx.x); };
  struct Item { int head, q0, L, nkv, ri; };
  auto locate = [&](int item) {
    Item it;
    const int tile = item / p.H;
    it.head = item - tile * p.H;
    it.ri = __popc(__ballot_sync(0xffffffffu, tile >= starts[lane])) + __popc(__ballot_sync(0xffffffffu, tile >= starts[lane + 32])) - 1;
    it.L = reqs[it.ri].L;
    it.q0 = (tile - starts[it.ri]) * 128;
    it.nkv = (it.L + ATC_KB - 1) / ATC_KB;
    return it;
  };

  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&q_full[b], 1); ptx::mbar_init(&q_free[b], 4);
      ptx::mbar_init(&s_full[b], 1); ptx::mbar_init(&s_free[b], 4);
      ptx::mbar_init(&p_full[b], 4); ptx::mbar_init(&o_full[b], 1);
    }
    for (int b = 0; b < ATC_ST; ++b) {
      ptx::mbar_init(&k_full[b], 1); ptx::mbar_init(&k_free[b], 1);
      ptx::mbar_init(&v_full[b], 1); ptx::mbar_init(&v_free[b], 1);
    }
    *dead = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    ptx::prefetch_tmap(&tmQ);
    ptx::prefetch_tmap(&tmK);
    ptx::prefetch_tmap(&tmV);
  }
  if (warp == 5) { ptx::tmem_alloc(tmem_slot, 256); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  ptx::pdl_launch();
  if (threadIdx.x == 0) { SOD2_TRACE(0, 1) }

  if (warp == 4 || warp == 7) {
    // ---- TMA producers: warp 4 Q and K, warp 7 V
    const bool is_k = warp == 4;
    const ptx::Leader one = ptx::elect_leader();
    ptx::pdl_wait();
    int n = 0, i = 0;
    for (int item; (item = nth_item(i)) < items; ++i) {
      const Item it = locate(item);
      const AtcReq R = reqs[it.ri];
      if (is_k) {
        const int qs = i & 1;
        if (i >= 2) ptx::mbar_wait_warp(&q_free[qs], ((i >> 1) - 1) & 1, dead);
        ptx::mbar_expect_tx(one, &q_full[qs], ATC_Q_BYTES);
        ptx::tma_load_2d(one, sQ + qs * ATC_Q_BYTES, &tmQ, p.q_col + it.head * p.q_hs, R.q_row + it.q0, &q_full[qs]);
      }
      uint64_t* full = is_k ? k_full : v_full;
      uint64_t* free_ = is_k ? k_free : v_free;
      uint8_t* dst = is_k ? sK : sV;
      const CUtensorMap* tm = is_k ? &tmK : &tmV;
      const int col = is_k ? p.k_col + it.head * p.k_hs : p.v_col + it.head * p.v_hs, row = is_k ? R.k_row : R.v_row;
      for (int j = 0; j < it.nkv; ++j, ++n) {
        const int b = n % ATC_ST;
        if (n >= ATC_ST) ptx::mbar_wait_warp(&free_[b], ((n / ATC_ST) - 1) & 1, dead);
        ptx::mbar_expect_tx(one, &full[b], ATC_KV_BYTES);
        ptx::tma_load_2d(one, dst + b * ATC_KV_BYTES, tm, col, row + j * ATC_KB, &full[b]);
        SOD2_TRACE(0, (is_k ? 800 : 840) + n)
      }
    }
  } else if (warp == 5) {
    // ---- S issuer: S_n once S_{n-2} is in registers
    constexpr uint32_t idesc_qk = ptx::idesc_bf16(128, ATC_KB);
    const ptx::Leader one = ptx::elect_leader();
    int n = 0, i = 0;
    for (int item; (item = nth_item(i)) < items; ++i) {
      const Item it = locate(item);
      const uint64_t dQ = ptx::smem_desc_sw128(ptx::smem_u32(sQ + (i & 1) * ATC_Q_BYTES));
      ptx::mbar_wait_warp(&q_full[i & 1], (i >> 1) & 1, dead);
      for (int j = 0; j < it.nkv; ++j, ++n) {
        const uint64_t dK = ptx::smem_desc_sw128(ptx::smem_u32(sK + (n % ATC_ST) * ATC_KV_BYTES));
        ptx::mbar_wait_lanes(&k_full[n % ATC_ST], (n / ATC_ST) & 1, dead);
        if (n >= 2) ptx::mbar_wait_lanes(&s_free[n & 1], ((n >> 1) - 1) & 1, dead);
        ptx::tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) ptx::mma_bf16(one, tmem + ATC_TMEM_S + (n & 1) * 64, dQ + 2 * kk, dK + 2 * kk, idesc_qk, kk != 0);
        __syncwarp();
        ptx::mma_commit(one, &s_full[n & 1]);
        ptx::mma_commit(one, &k_free[n % ATC_ST]);
        if (lane == 0) { SOD2_TRACE(1, 100 + n) }
      }
    }
  } else if (warp == 6) {
    // ---- O issuer: O += P_n V_n.  The softmax warps rescale O (rarely) before they hand over P_n, and read an item's O
    // before they hand over the next item's first P, so the accumulator needs no barrier of its own.
    constexpr uint32_t idesc_pv = ptx::idesc_bf16(128, 64) | (1u << 16);   // B (= V tile) is MN-major
    const ptx::Leader one = ptx::elect_leader();
    int n = 0;
    for (int i = 0, item; (item = nth_item(i)) < items; ++i) {
      const Item it = locate(item);
      for (int j = 0; j < it.nkv; ++j, ++n) {
        const int steps = (it.L - j * ATC_KB + 15) >> 4;       // keys past the request are left out
        const uint32_t aV = ptx::smem_u32(sV + (n % ATC_ST) * ATC_KV_BYTES);
        ptx::mbar_wait_lanes(&v_full[n % ATC_ST], (n / ATC_ST) & 1, dead);
        ptx::mbar_wait_lanes(&p_full[n & 1], (n >> 1) & 1, dead);
        ptx::tc_fence_after();
        // 16 keys per step: 8 packed columns of P in tensor memory, 16 rows (2048 B) down V
#pragma unroll
        for (int kk = 0; kk < ATC_KB / 16; ++kk)
          if (kk < steps) ptx::mma_bf16_a_tmem(one, tmem + ATC_TMEM_O, tmem + ATC_TMEM_P + (n & 1) * 32 + kk * 8, ptx::smem_desc_sw128(aV + kk * 2048), idesc_pv, (j | kk) != 0);
        __syncwarp();
        ptx::mma_commit(one, &o_full[n & 1]);
        ptx::mma_commit(one, &v_free[n % ATC_ST]);
        if (lane == 0) { SOD2_TRACE(1, 200 + n) }
      }
    }
  } else {
    // ---- softmax warps 0..3, a thread per query row
    const int row = threadIdx.x;
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    const bool tracer = threadIdx.x == 0;
    const float c = p.scale_log2e;
    const uint32_t o_addr = tmem + lane_base + ATC_TMEM_O;
    ptx::pdl_wait();
    Item prev{};
    bool prev_live = false;
    float prev_l = 1.f;
    // Output of item `pi`, the one before: O / l, staged (swizzled) in the item's Q buffer, which nothing reads any more, and
    // written four full 128-byte rows per instruction; a warp's rows are its own.  `end`: blocks up to the item's last.
    auto finish = [&](int pi, int end) {
      ptx::mbar_wait_warp(&o_full[(end - 1) & 1], ((end - 1) >> 1) & 1, dead);   // every product has landed
      ptx::tc_fence_after();
      uint8_t* stage = sQ + (pi & 1) * ATC_Q_BYTES;
      if (prev_live) {
        const float inv = 1.0f / prev_l;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t r[32];
          ptx::tmem_ld32(o_addr + h * 32, r);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            uint4 v;
            __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
            for (int e = 0; e < 4; ++e) h2[e] = __floats2bfloat162_rn(__uint_as_float(r[g * 8 + 2 * e]) * inv, __uint_as_float(r[g * 8 + 2 * e + 1]) * inv);
            *reinterpret_cast<uint4*>(stage + row * 128 + (((h * 4 + g) ^ (row & 7)) << 4)) = v;
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        __nv_bfloat16* og = p.o + reqs[prev.ri].o_off + static_cast<long long>(prev.head) * p.o_hs;
        uint4 v[8];
        const int r0 = warp * 32 + (lane >> 3), ch = lane & 7;
#pragma unroll
        for (int g = 0; g < 8; ++g) v[g] = *reinterpret_cast<const uint4*>(stage + (r0 + g * 4) * 128 + ((ch ^ ((r0 + g * 4) & 7)) << 4));
        // the buffer is handed back before the rows go out: a proxy fence behind them would wait for the stores
        ptx::fence_proxy_async();
        __syncwarp();
        ptx::mbar_arrive_warp(&q_free[pi & 1]);
#pragma unroll
        for (int g = 0; g < 8; ++g)
          if (prev.q0 + r0 + g * 4 < prev.L) *reinterpret_cast<uint4*>(og + static_cast<long long>(prev.q0 + r0 + g * 4) * p.o_ts + ch * 8) = v[g];
      } else {
        ptx::mbar_arrive_warp(&q_free[pi & 1]);
      }
      if (tracer) { SOD2_TRACE(2, 700 + pi) }
    };
    // maximum of the first `live_cols` scores of a tile in tensor memory (registers are few where this is needed)
    auto max_ahead = [&](uint32_t addr, int live_cols) {
      float mx = -INFINITY;
#pragma unroll 1
      for (int h = 0; h < ATC_KB && h < live_cols; h += 8) {
        uint32_t r[8];
        ptx::tmem_ld8(addr + h, r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) if (h + e < live_cols) mx = fmaxf(mx, __uint_as_float(r[e]));
      }
      return mx;
    };
    int n = 0, i = 0;
    bool s_seen = false;
    for (int item; (item = nth_item(i)) < items; ++i) {
      const Item it = locate(item);
      const bool live = it.q0 + warp * 32 < it.L;    // a warp whose 32 rows are all past the request only keeps the barriers moving
      // Online softmax with a lazily updated reference: the exponent reference m starts as the row maximum of the first
      // 128 keys and then only moves when a block's row maximum exceeds it by more than 2^8 after scaling, so p stays
      // <= 256 (exact enough in bf16 and fp32) and the accumulator O in TMEM is rescaled only then -- for almost every block
      // nothing is read back from TMEM.  l and O always refer to the same m, so O / l at the end is the softmax average.
      // References are chosen over pairs of blocks, the second block's scores looked at ahead: the largest p of those keys is
      // then exactly 1, where bf16 does not round it.  (A reference out of 64 keys alone rounds the weight that dominates
      // a row: against fp64, scores of standard deviation 2 and 128 keys, 1.17 times the error.)
      float m = -INFINITY;
      float2 l = make_float2(0.f, 0.f);
      for (int j = 0; j < it.nkv; ++j, ++n) {
        const int buf = n & 1;
        const uint32_t s_addr = tmem + lane_base + ATC_TMEM_S + buf * 64, p_addr = tmem + lane_base + ATC_TMEM_P + buf * 32;
        if (!s_seen) ptx::mbar_wait_warp(&s_full[buf], (n >> 1) & 1, dead);
        const bool o_seen = ptx::mbar_test_wait_warp(&o_full[buf], ((n >> 1) - 1) & 1);     // consumed below (n >= 2)
        ptx::tc_fence_after();
        if (tracer) { SOD2_TRACE(2, 300 + n) }
        if (__builtin_expect(!live, 0)) {
          __syncwarp();
          ptx::mbar_arrive_warp(&s_free[buf]);
          if (j == 0 && i > 0) finish(i - 1, n);
          // not before P_{n-2} is through: an arrival too many would complete that phase early
          if (n >= 2) ptx::mbar_wait_warp(&o_full[buf], ((n >> 1) - 1) & 1, dead);
          ptx::mbar_arrive_warp(&p_full[buf]);
          s_seen = false;
          continue;
        }
        const int valid = it.L - j * ATC_KB;     // keys of the block inside the request
        const bool pair = !(j & 1) && valid > ATC_KB;
        const uint32_t s_next = s_addr ^ 64;     // the other score tile
        uint32_t s[64];
        if (__builtin_expect(j == 0 && pair, 0)) {
          ptx::mbar_wait_warp(&s_full[buf ^ 1], ((n + 1) >> 1) & 1, dead);
          ptx::tc_fence_after();
          if (valid >= 2 * ATC_KB) {           // half a tile is reduced while the next half is under way
            ptx::tmem_ld32(s_next, s);
            ptx::tmem_ld_wait();
            ptx::tmem_ld32(s_next + 32, s + 32);
            m = atc_max32(m, s);
            ptx::tmem_ld_wait();
            ptx::tmem_ld32(s_addr, s);
            m = atc_max32(m, s + 32);
          } else {
            m = max_ahead(s_next, valid - ATC_KB);
            ptx::tmem_ld32(s_addr, s);
          }
        } else {
          ptx::tmem_ld32(s_addr, s);
        }
        ptx::tmem_ld32(s_addr + 32, s + 32);
        ptx::tmem_ld_wait();
        ptx::tc_fence_before();
        __syncwarp();
        ptx::mbar_arrive_warp(&s_free[buf]);
        if (__builtin_expect(valid < ATC_KB, 0)) {
#pragma unroll
          for (int e = 0; e < 64; ++e) if (e >= valid) s[e] = 0xff800000u;   // -inf
        }
        const float mx = atc_max32(atc_max32(-INFINITY, s), s + 32);
        if (tracer) { SOD2_TRACE(2, 600 + n) }
        // move the reference if the block asks for it
        const bool move = (mx - m) * c > 8.0f;
        if (j == 0) m = fmaxf(m, mx);
        if (__builtin_expect(j > 0 && __any_sync(0xffffffffu, move), 0)) {
          float ref = mx;
          if (pair) {
            ptx::mbar_wait_warp(&s_full[buf ^ 1], ((n + 1) >> 1) & 1, dead);
            ptx::tc_fence_after();
            ref = fmaxf(mx, max_ahead(s_next, valid - ATC_KB));
          }
          float corr = 1.f;
          if (move) { corr = ex2_approx((m - ref) * c); m = ref; l.x *= corr; l.y *= corr; }
          // all products issued so far must have landed in O before it is scaled
          ptx::mbar_wait_warp(&o_full[(n - 1) & 1], ((n - 1) >> 1) & 1, dead);
          ptx::tc_fence_after();
#pragma unroll 1
          for (int h = 0; h < 8; ++h) {
            uint32_t r[8];
            ptx::tmem_ld8(o_addr + h * 8, r);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 8; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * corr);
            ptx::tmem_st8(o_addr + h * 8, r);
          }
          ptx::tmem_st_wait();
          ptx::tc_fence_before();
        }
        const float2 c2 = make_float2(c, c), mc2 = make_float2(-m * c, -m * c);
        // P_n into tensor memory, 16 columns at a time; the product that read these columns two blocks ago has finished
        uint32_t pk[16];
        atc_exp32(s, pk, c2, mc2, &l);
        if (n >= 2 && !o_seen) ptx::mbar_wait_warp(&o_full[buf], ((n >> 1) - 1) & 1, dead);
        ptx::tc_fence_after();
        ptx::tmem_st16(p_addr, pk);
        if (__builtin_expect(valid > 32, 1)) {
          atc_exp32(s + 32, pk, c2, mc2, &l);
          ptx::tmem_st16(p_addr + 16, pk);
        }
        if (tracer) { SOD2_TRACE(2, 400 + n) }
        if (__builtin_expect(j == 0 && i > 0, 0)) finish(i - 1, n);
        s_seen = ptx::mbar_test_wait_warp(&s_full[buf ^ 1], ((n + 1) >> 1) & 1);     // the next block's scores are usually there
        ptx::tmem_st_wait();
        ptx::tc_fence_before();
        __syncwarp();
        ptx::mbar_arrive_warp(&p_full[buf]);
        if (tracer) { SOD2_TRACE(2, 500 + n) }
      }
      prev = it;
      prev_live = live;
      prev_l = l.x + l.y;
    }
    if (i > 0) finish(i - 1, n);
  }
  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 5) ptx::tmem_dealloc(tmem, 256);
  if (threadIdx.x == 0 && *dead && p.status) atomicExch(p.status, 1);
  SOD2_TRACE_DUMP()
}

}  // namespace k
}  // namespace sod2
