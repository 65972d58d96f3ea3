// Scan-based compaction for execution-determined operators (Section 3, "Execution Determined
// Output"; Fig. 1(c) TopK): top-k token keeping, NonZero.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "ptx.cuh"

namespace sod2 {
namespace k {

constexpr int COMPACT_MAX_REQ = 32;

// ---------------------------------------------------------------------------------------------
// Token scores: s_i = sum_d y[i,d]^2 accumulated in fp64 (squares of bf16 values are exact in fp64,
// so the score depends on the summation order only at the 2^-53 level; decisions are then taken on
// these fp64 scores). One warp per row, fixed lane-strided order + fixed shuffle tree: deterministic.
struct ScoreParams {
  const __nv_bfloat16* y;   // packed rows of all requests, [rows, D]
  double* score;            // [rows]
  long long rows;
  int D;
};
__global__ void __launch_bounds__(256) row_sumsq_f64(ScoreParams p) {
  ptx::pdl_wait();
  ptx::pdl_launch();
  const int lane = threadIdx.x & 31;
  const long long row = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (row >= p.rows) return;
  const __nv_bfloat16* yr = p.y + row * p.D;
  double acc = 0.0;
  if ((p.D & 7) == 0) {
    const uint4* v = reinterpret_cast<const uint4*>(yr);
    for (int i = lane; i < (p.D >> 3); i += 32) {
      uint4 u = v[i];
      const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float2 f = __bfloat1622float2(h[t]);
        acc += static_cast<double>(f.x) * f.x;
        acc += static_cast<double>(f.y) * f.y;
      }
    }
  } else {
    for (int i = lane; i < p.D; i += 32) { const double f = __bfloat162float(yr[i]); acc += f * f; }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) p.score[row] = acc;
}

// ---------------------------------------------------------------------------------------------
// Keep the k highest-scoring tokens of each request in ascending index order, ties by the lower index:
//   keep_i = s_i > T, or s_i == T and fewer than `rem` equal scores before i;  pos_i = #{j < i : keep_j}
//   idx[pos_i] = i;  out[pos_i, :] = y[i, :]
// with T the k-th largest score and `rem` the number of scores equal to T that are kept.  One CTA per chunk of 32 tokens
// (a single request of 577 tokens is 19 CTAs, 16 of 500 are 250); every CTA selects T for itself out of its request's
// scores in shared memory, so nothing has to be exchanged between CTAs and one launch does: scores as 64-bit integers in
// the order of the doubles, radix selection eight bits at a time from the highest bit in which any two scores differ,
// until the digit found is kept whole (two or three passes for scores that differ).
// Bound by latency: the wait for the scores, about 200 cycles per pass, the rows out.  With the score kernel, against a
// kernel that ranked every token with all others in fp64 and one that copied (D = 384): 16 requests of 238 to 780 tokens
// 28.4 -> 9.1 us, one of 577 tokens 9.7 -> 6.2 us.
// LN > 0: the kept rows also leave normalised (the LayerNorm group behind the selection; D <= 256 * LN).  A warp then holds four
// rows of the chunk and has their statistics before it waits for the scores, so that the LayerNorm costs its stores and no
// launch.  The arithmetic is layernorm_bf16's, lane by lane: the same bits.  (One request of 577 tokens through 12 layers 367 -> 359 us,
// 16 requests 541 -> 530 us.)
constexpr int TOPK_CHUNK = 32, TOPK_THREADS = 256;
struct TopkReq {
  long long row0;      // first packed input row of the request
  long long out_row0;  // first packed output row
  long long idx0;      // first packed index entry
  int n, k;
};
struct TopkParams {
  const __nv_bfloat16* y;
  const double* score;       // packed [rows] relative to the first request's row0
  __nv_bfloat16* out;
  long long* idx;            // packed [sum k] int64, per request k entries
  int D;
  int n_req;
  long long first_row;       // row0 of the first request (scores are indexed from it)
  int chunk_start[COMPACT_MAX_REQ + 1];   // prefix sum of ceil(n / TOPK_CHUNK)
  TopkReq r[COMPACT_MAX_REQ];
  // LN > 0: constants of the graph, and the normalised rows, packed like `out`
  const __nv_bfloat16 *gamma, *beta;
  __nv_bfloat16* normed;
  float eps;
};

__device__ __forceinline__ int topk_locate(const TopkParams& p, int cta, int* chunk) {
  int ri = 0;
  while (ri + 1 < p.n_req && cta >= p.chunk_start[ri + 1]) ++ri;
  *chunk = cta - p.chunk_start[ri];
  return ri;
}

template <int LN>
__global__ void __launch_bounds__(TOPK_THREADS) topk_select_gather(const __grid_constant__ TopkParams p) {
  extern __shared__ unsigned long long s_key[];        // [n]
  __shared__ unsigned s_hist[256];
  __shared__ unsigned s_diff[2];
  __shared__ int s_found[3], s_before[2], s_pos[TOPK_CHUNK];
  int chunk;
  const TopkReq R = p.r[topk_locate(p, blockIdx.x, &chunk)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = chunk * TOPK_CHUNK;
  // The rows of the chunk are fetched before the dependency wait: they were written by the kernel before the score
  // kernel, which had completed before any CTA of the score kernel let this one start, so only the scores are still in
  // flight.  Whether a row is kept is not known yet: all rows of the chunk are read.
  const int vec = (p.D * 2) >> 4;  // 16-byte pieces per row (D % 8 == 0 checked on the host)
  const uint4* src = reinterpret_cast<const uint4*>(p.y + (R.row0 + base) * p.D);
  const int items = min(TOPK_CHUNK, R.n - base) * vec;
  constexpr int PRE = LN ? 4 * LN : 6;
  uint4 pre[PRE];                // LN: row warp + 8 u of the chunk, vectors lane + 32 c, in pre[u * LN + c]
  [[maybe_unused]] uint4 g4[LN ? LN : 1], b4[LN ? LN : 1];
  [[maybe_unused]] float mu[4], rstd[4];
  if constexpr (LN > 0) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int c = 0; c < LN; ++c) pre[u * LN + c] = src[min(warp + 8 * u, items / vec - 1) * vec + min(c * 32 + lane, vec - 1)];
#pragma unroll
    for (int c = 0; c < LN; ++c) {
      g4[c] = reinterpret_cast<const uint4*>(p.gamma)[min(c * 32 + lane, vec - 1)];
      b4[c] = reinterpret_cast<const uint4*>(p.beta)[min(c * 32 + lane, vec - 1)];
    }
  } else {
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
      const int it = tid + u * TOPK_THREADS;
      if (it < items) pre[u] = src[it];
    }
  }
  s_hist[tid] = 0;
  if (tid < 2) { s_diff[tid] = 0; s_before[tid] = 0; }
  if constexpr (LN > 0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float s = 0.f, q = 0.f;
#pragma unroll
      for (int c = 0; c < LN; ++c) {
        const bool in = c * 32 + lane < vec;
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&pre[u * LN + c]);
#pragma unroll
        for (int t = 0; t < 4; ++t) { const float2 f = __bfloat1622float2(h[t]); s += in ? f.x + f.y : 0.f; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      mu[u] = s / p.D;
#pragma unroll
      for (int c = 0; c < LN; ++c)
        if (c * 32 + lane < vec) {
          const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&pre[u * LN + c]);
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const float2 f = __bfloat1622float2(h[t]);
            float d = f.x - mu[u]; q += d * d;
            d = f.y - mu[u]; q += d * d;
          }
        }
#pragma unroll
      for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      rstd[u] = rsqrtf(q / p.D + p.eps);
    }
  }
  ptx::pdl_wait();
  ptx::pdl_launch();
  // Scores are sums of squares: as integers with the top bit set they keep their order.  A NaN score (an overflow
  // upstream) becomes 0 and ranks last, ties among NaNs by index, so that exactly k tokens are kept whatever the data.
  const double* sc = p.score + (R.row0 - p.first_row);
  auto key_of = [&](int i) -> unsigned long long {
    const double v = sc[i];
    return v == v ? static_cast<unsigned long long>(__double_as_longlong(v)) | (1ull << 63) : 0ull;
  };
  const unsigned long long key0 = key_of(0);
  unsigned long long diff = 0;
  for (int i = tid; i < R.n; i += TOPK_THREADS) { const unsigned long long q = key_of(i); s_key[i] = q; diff |= q ^ key0; }
  const unsigned d_hi = __reduce_or_sync(0xffffffffu, static_cast<unsigned>(diff >> 32)), d_lo = __reduce_or_sync(0xffffffffu, static_cast<unsigned>(diff));
  __syncthreads();
  if (lane == 0) { if (d_hi) atomicOr(&s_diff[1], d_hi); if (d_lo) atomicOr(&s_diff[0], d_lo); }
  __syncthreads();
  diff = static_cast<unsigned long long>(s_diff[1]) << 32 | s_diff[0];
  // T: keys above it are kept, and the first `rem` of those equal to it
  unsigned long long T = key0;
  int rem = R.k;
  if (R.k >= R.n) { T = 0; rem = R.n; }
  else if (R.k <= 0) { T = ~0ull; rem = 0; }
  else if (diff) {
    int top = 64 - __clzll(static_cast<long long>(diff));        // bits not decided yet; those above are the same in all keys
    unsigned long long high = top < 64 ? key0 >> top : 0ull;
    for (;;) {
      const int width = min(8, top), low = top - width;
      for (int i = tid; i < R.n; i += TOPK_THREADS) {
        const unsigned long long q = s_key[i];
        if ((top < 64 ? q >> top : 0ull) == high) atomicAdd(&s_hist[static_cast<unsigned>(q >> low) & ((1u << width) - 1)], 1u);
      }
      __syncthreads();
      if (warp == 0) {
        // eight digits per lane, from the largest
        int h[8], c = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) { h[u] = static_cast<int>(s_hist[255 - lane * 8 - u]); c += h[u]; }
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += t; }
        int above = incl - c;
        if (above < rem && rem <= incl) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (above < rem && rem <= above + h[u]) { s_found[0] = 255 - lane * 8 - u; s_found[1] = rem - above; s_found[2] = h[u]; }
            above += h[u];
          }
        }
      }
      __syncthreads();
      high = high << width | static_cast<unsigned>(s_found[0]);
      rem = s_found[1];
      top = low;
      if (rem == s_found[2] || top == 0) break;
      s_hist[tid] = 0;
      __syncthreads();
    }
    T = high << top;
    if (top > 0) { T -= 1; rem = 0; }      // the digit is kept whole: everything above T
  }
  // scores above T and equal to it, before the chunk
  int gt = 0, eq = 0;
  for (int j = tid; j < base; j += TOPK_THREADS) { const unsigned long long q = s_key[j]; gt += q > T; eq += q == T; }
  gt = __reduce_add_sync(0xffffffffu, gt);
  eq = __reduce_add_sync(0xffffffffu, eq);
  if (lane == 0 && (gt | eq)) { atomicAdd(&s_before[0], gt); atomicAdd(&s_before[1], eq); }
  __syncthreads();
  if (warp == 0) {
    const int i = base + lane;
    const unsigned long long q = i < R.n ? s_key[i] : 0ull;
    const unsigned bg = __ballot_sync(0xffffffffu, i < R.n && q > T), be = __ballot_sync(0xffffffffu, i < R.n && q == T), lt = (1u << lane) - 1;
    const int eq_before = s_before[1] + __popc(be & lt);
    const bool keep = ((bg >> lane) & 1u) || (((be >> lane) & 1u) && eq_before < rem);
    const int pos = s_before[0] + __popc(bg & lt) + min(eq_before, rem);
    s_pos[lane] = keep ? pos : -1;
    if (keep) p.idx[R.idx0 + pos] = i;
  }
  __syncthreads();
  // write the kept rows: (row, 16-byte piece) items spread over the whole CTA; the first PRE per thread are
  // already in registers, wider rows load the rest now
  uint4* dst = reinterpret_cast<uint4*>(p.out + R.out_row0 * p.D);
  if constexpr (LN > 0) {
    uint4* nrm = reinterpret_cast<uint4*>(p.normed + R.out_row0 * p.D);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int pos = s_pos[warp + 8 * u];
      if (pos < 0) continue;
#pragma unroll
      for (int c = 0; c < LN; ++c)
        if (c * 32 + lane < vec) {
          const uint4 x = pre[u * LN + c];
          uint4 y;
          const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162*>(&x), *gh = reinterpret_cast<const __nv_bfloat162*>(&g4[c]), *bh = reinterpret_cast<const __nv_bfloat162*>(&b4[c]);
          __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&y);
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const float2 f = __bfloat1622float2(h[t]), gf = __bfloat1622float2(gh[t]), bf = __bfloat1622float2(bh[t]);
            oh[t] = __floats2bfloat162_rn((f.x - mu[u]) * rstd[u] * gf.x + bf.x, (f.y - mu[u]) * rstd[u] * gf.y + bf.y);
          }
          dst[static_cast<long long>(pos) * vec + c * 32 + lane] = x;
          nrm[static_cast<long long>(pos) * vec + c * 32 + lane] = y;
        }
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < PRE; ++u) {
    const int it = tid + u * TOPK_THREADS;
    if (it < items) {
      const int t = it / vec, c4 = it - t * vec;
      const int pos = s_pos[t];
      if (pos >= 0) dst[static_cast<long long>(pos) * vec + c4] = pre[u];
    }
  }
#pragma unroll 4
  for (int it = tid + PRE * TOPK_THREADS; it < items; it += TOPK_THREADS) {
    const int t = it / vec, c4 = it - t * vec;
    const int pos = s_pos[t];
    if (pos >= 0) dst[static_cast<long long>(pos) * vec + c4] = src[it];
  }
}

// ---------------------------------------------------------------------------------------------
// NonZero: int64 coordinates [rank, nnz] of the non-zero elements in row-major order, all requests of a batch in two
// launches.  The row pitch of the output is nnz, so no coordinate can be written before everything is counted:
//   nonzero_mask   reads the input once (16-byte loads), leaves one bit per element and a count per chunk in scratch
//   nonzero_write  a CTA per chunk adds up the counts in front of its own (at most NZ_MAX_CHUNKS, from L2), expands its
//                  bits into a list of element indices in shared memory and writes the coordinates from there, so that
//                  neighbouring threads write neighbouring words
// A chunk is NZ_SUB elements, more where a request would have over NZ_MAX_CHUNKS of them.
// Bound by the 16 bytes written per element found and, below a few MB, by the two launches.
// Measured on B200, 1024x1024 + 777x1333 + 3x4095 + 2048x768 in fp32 (38 MB): with three launches per request and one
// element per thread 114 us on the device and 200 us with the counts read back; now 52 us with the counts read back.
constexpr int NZ_THREADS = 256, NZ_SUB = NZ_THREADS * 32, NZ_MAX_CHUNKS = 2048, NZ_MAX_REQ = 8;
struct NonZeroReq {
  const void* x;
  long long numel;
  long long dims[4];      // leading extents are 1 below rank 4
  long long chunk;        // elements per chunk, a multiple of NZ_SUB
  unsigned* mask;         // scratch: one bit per element, whole NZ_SUBs
  int* count;             // scratch: non-zero elements per chunk
  long long* out;         // [rank, nnz]
  long long* count_out;   // device word: nnz
  int first, chunks;      // first CTA of the request in the launch, number of its chunks (at least one)
  int vec_ok;             // x is 16-byte aligned
};
struct NonZeroBatch {
  int n_req, is_bf16, rank;
  NonZeroReq r[NZ_MAX_REQ];
};
__device__ __forceinline__ const NonZeroReq& nz_find(const NonZeroBatch& p) {
  int ri = 0;
  while (ri + 1 < p.n_req && static_cast<int>(blockIdx.x) >= p.r[ri + 1].first) ++ri;
  return p.r[ri];
}
template <class T>
__device__ __forceinline__ T nz_block_sum(T v, T* warp_sums) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = v;
  __syncthreads();
  T t = 0;
#pragma unroll
  for (int w = 0; w < NZ_THREADS / 32; ++w) t += warp_sums[w];
  return t;
}
__global__ void __launch_bounds__(NZ_THREADS) nonzero_mask(const __grid_constant__ NonZeroBatch p) {
  __shared__ int warp_sums[NZ_THREADS / 32];
  const NonZeroReq& R = nz_find(p);
  ptx::pdl_wait();
  ptx::pdl_launch();
  const int chunk = blockIdx.x - R.first, tid = threadIdx.x, lane = tid & 31;
  const long long lo = chunk * R.chunk, hi = min(R.numel, lo + R.chunk);
  int cnt = 0;
  for (long long base = lo; base < hi; base += NZ_SUB) {
    unsigned* words = R.mask + (base >> 5);
    if (R.vec_ok && base + NZ_SUB <= R.numel) {
      if (p.is_bf16) {
        const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(R.x) + base);
        uint4 u[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) u[v] = src[v * NZ_THREADS + tid];
#pragma unroll
        for (int v = 0; v < 4; ++v) {     // eight elements per thread: four threads make a word
          const unsigned q[4] = {u[v].x, u[v].y, u[v].z, u[v].w};
          unsigned b = 0;
#pragma unroll
          for (int t = 0; t < 4; ++t) b |= ((q[t] & 0x7fffu) ? 1u : 0u) << (2 * t) | ((q[t] & 0x7fff0000u) ? 2u : 0u) << (2 * t);
          b <<= 8 * (lane & 3);
          b |= __shfl_xor_sync(0xffffffffu, b, 1);
          b |= __shfl_xor_sync(0xffffffffu, b, 2);
          if ((lane & 3) == 0) { words[(v * NZ_THREADS + tid) >> 2] = b; cnt += __popc(b); }
        }
      } else {
        const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(R.x) + base);
        float4 u[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) u[v] = src[v * NZ_THREADS + tid];
#pragma unroll
        for (int v = 0; v < 8; ++v) {     // four elements per thread: eight threads make a word
          unsigned b = (u[v].x != 0.f ? 1u : 0u) | (u[v].y != 0.f ? 2u : 0u) | (u[v].z != 0.f ? 4u : 0u) | (u[v].w != 0.f ? 8u : 0u);
          b <<= 4 * (lane & 7);
          b |= __shfl_xor_sync(0xffffffffu, b, 1);
          b |= __shfl_xor_sync(0xffffffffu, b, 2);
          b |= __shfl_xor_sync(0xffffffffu, b, 4);
          if ((lane & 7) == 0) { words[(v * NZ_THREADS + tid) >> 3] = b; cnt += __popc(b); }
        }
      }
      continue;
    }
    // the request's last piece, or a caller's buffer that is not 16-byte aligned: a warp makes a word at a time
    for (int w = tid >> 5; w < NZ_SUB / 32; w += NZ_THREADS / 32) {
      const long long i = base + w * 32 + lane;
      bool f = false;
      if (i < R.numel)
        f = p.is_bf16 ? (__bfloat162float(reinterpret_cast<const __nv_bfloat16*>(R.x)[i]) != 0.0f) : (reinterpret_cast<const float*>(R.x)[i] != 0.0f);
      const unsigned b = __ballot_sync(0xffffffffu, f);
      if (lane == 0) { words[w] = b; cnt += __popc(b); }
    }
  }
  const int total = nz_block_sum(cnt, warp_sums);
  if (tid == 0) R.count[chunk] = total;
}
__global__ void __launch_bounds__(NZ_THREADS) nonzero_write(const __grid_constant__ NonZeroBatch p) {
  __shared__ long long totals[2][NZ_THREADS / 32];       // (a request may hold more than 2^31 non-zero elements)
  __shared__ int sums[NZ_THREADS / 32];
  __shared__ unsigned short list[NZ_SUB];
  const NonZeroReq& R = nz_find(p);
  const int chunk = blockIdx.x - R.first, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long lo = chunk * R.chunk, hi = min(R.numel, lo + R.chunk);
  ptx::pdl_wait();
  ptx::pdl_launch();
  long long before = 0, all = 0;
  for (int j = tid; j < R.chunks; j += NZ_THREADS) { const int c = R.count[j]; all += c; before += j < chunk ? c : 0; }
  before = nz_block_sum(before, totals[0]);
  const long long nnz = nz_block_sum(all, totals[1]);
  if (chunk == 0 && tid == 0) *R.count_out = nnz;
  long long off = before;
  for (long long base = lo; base < hi; base += NZ_SUB) {
    unsigned m = R.mask[(base >> 5) + tid];
    const int mine = __popc(m);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    __syncthreads();                     // the previous piece's list and sums have been read
    if (lane == 31) sums[warp] = inc;
    __syncthreads();
    int at = inc - mine, cnt = 0;
#pragma unroll
    for (int w = 0; w < NZ_THREADS / 32; ++w) { const int t = sums[w]; at += w < warp ? t : 0; cnt += t; }
    while (m) {
      const int b = __ffs(m) - 1;
      m &= m - 1;
      list[at++] = static_cast<unsigned short>(tid * 32 + b);
    }
    __syncthreads();
    long long* out = R.out + off;
    if (R.numel < (1ll << 32)) {
      const unsigned d1 = static_cast<unsigned>(R.dims[1]), d2 = static_cast<unsigned>(R.dims[2]), d3 = static_cast<unsigned>(R.dims[3]);
      for (int j = tid; j < cnt; j += NZ_THREADS) {
        const unsigned e = static_cast<unsigned>(base) + list[j];
        long long* o = out + j + (p.rank - 1) * nnz;
        unsigned q = e / d3;
        *o = e - q * d3;
        if (p.rank > 1) {
          if (p.rank == 2) { o[-nnz] = q; continue; }
          const unsigned q2 = q / d2;
          o[-nnz] = q - q2 * d2;
          if (p.rank == 3) { o[-2 * nnz] = q2; continue; }
          const unsigned q1 = q2 / d1;
          o[-2 * nnz] = q2 - q1 * d1;
          o[-3 * nnz] = q1;
        }
      }
    } else {
      for (int j = tid; j < cnt; j += NZ_THREADS) {
        long long e = base + list[j];
        for (int d = p.rank - 1; d >= 0; --d) {
          const long long ext = R.dims[4 - p.rank + d];
          out[d * nnz + j] = e % ext;
          e /= ext;
        }
      }
    }
    off += cnt;
  }
}

}  // namespace k
}  // namespace sod2
