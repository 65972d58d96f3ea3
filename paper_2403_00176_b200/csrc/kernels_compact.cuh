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
// Keep the k highest-scoring tokens of each request in ascending index order.
//   rank_i = #{j : s_j > s_i} + #{j < i : s_j == s_i};  keep_i = rank_i < k
//   pos_i  = exclusive scan of keep;  idx[pos_i] = i;  out[pos_i, :] = y[i, :]
// Two kernels over the same grid, one CTA per chunk of 64 tokens of a request (so a batch of 16
// requests spreads over about a hundred SMs instead of 16):
//   topk_flags   the request's fp64 scores staged in shared memory; four threads share a token's
//                ranking (a quarter of the comparisons each); writes keep_i as a byte
//   topk_gather  counts the kept tokens before the chunk, scans the chunk's 64 flags with two ballots,
//                writes the indices and copies the kept rows, one warp per row, 128-bit accesses
constexpr int TOPK_CHUNK = 64;
struct TopkReq {
  long long row0;      // first packed input row of the request
  long long out_row0;  // first packed output row
  long long idx0;      // first packed index entry
  int n, k;
};
struct TopkParams {
  const __nv_bfloat16* y;
  const double* score;       // packed [rows] relative to the first request's row0
  unsigned char* keep;       // packed [rows], same indexing as score
  __nv_bfloat16* out;
  long long* idx;            // packed [sum k] int64, per request k entries
  int D;
  int n_req;
  long long first_row;       // row0 of the first request (score / keep are indexed from it)
  int chunk_start[COMPACT_MAX_REQ + 1];   // prefix sum of ceil(n / 64)
  TopkReq r[COMPACT_MAX_REQ];
};

__device__ __forceinline__ int topk_locate(const TopkParams& p, int cta, int* chunk) {
  int ri = 0;
  while (ri + 1 < p.n_req && cta >= p.chunk_start[ri + 1]) ++ri;
  *chunk = cta - p.chunk_start[ri];
  return ri;
}

__global__ void __launch_bounds__(256) topk_flags(const __grid_constant__ TopkParams p) {
  extern __shared__ double s_score[];                  // [n]
  int chunk;
  const TopkReq R = p.r[topk_locate(p, blockIdx.x, &chunk)];
  ptx::pdl_wait();
  ptx::pdl_launch();
  const int tid = threadIdx.x;
  const double* sc = p.score + (R.row0 - p.first_row);
  // a NaN score (an overflow upstream) compares false with everything and would be kept by every chunk: it ranks
  // last instead, ties among NaNs by index, so that exactly k tokens are kept whatever the data
  for (int i = tid; i < R.n; i += 256) { const double v = sc[i]; s_score[i] = v == v ? v : -INFINITY; }
  __syncthreads();
  const int i = chunk * TOPK_CHUNK + (tid >> 2), part = tid & 3;
  int rank = 0;
  if (i < R.n) {
    const double si = s_score[i];
    const int per = (R.n + 3) >> 2, j0 = part * per, j1 = min(R.n, j0 + per);
    for (int j = j0; j < j1; ++j) {
      const double sj = s_score[j];
      rank += (sj > si) || (sj == si && j < i);
    }
  }
  rank += __shfl_xor_sync(0xffffffffu, rank, 1);
  rank += __shfl_xor_sync(0xffffffffu, rank, 2);
  if (i < R.n && part == 0) p.keep[R.row0 - p.first_row + i] = rank < R.k;
}

__global__ void __launch_bounds__(256) topk_gather(const __grid_constant__ TopkParams p) {
  __shared__ int warp_cnt[8];
  __shared__ int s_pos[TOPK_CHUNK];
  int chunk;
  const TopkReq R = p.r[topk_locate(p, blockIdx.x, &chunk)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = chunk * TOPK_CHUNK;
  // The rows of the chunk are fetched before the dependency wait: they were written by the kernel before the
  // score kernel, which had completed before the flag kernel (the one waited for here) let this one start, so
  // only the flags are still in flight.  Whether a row is kept is not known yet: all rows of the chunk are read.
  const int vec = (p.D * 2) >> 4;  // 16-byte pieces per row (D % 8 == 0 checked on the host)
  const uint4* src = reinterpret_cast<const uint4*>(p.y + (R.row0 + base) * p.D);
  const int items = min(TOPK_CHUNK, R.n - base) * vec;
  constexpr int PRE = 12;
  uint4 pre[PRE];
#pragma unroll
  for (int u = 0; u < PRE; ++u) {
    const int it = tid + u * 256;
    if (it < items) pre[u] = src[it];
  }
  ptx::pdl_wait();
  ptx::pdl_launch();
  const unsigned char* kp = p.keep + (R.row0 - p.first_row);
  // kept tokens before this chunk
  int c = 0;
  for (int j = tid; j < base; j += 256) c += kp[j];
#pragma unroll
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) warp_cnt[warp] = c;
  __syncthreads();
  int carry = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) carry += warp_cnt[w];
  // the chunk's own 64 flags: warps 0 and 1 take 32 each
  if (warp < 2) {
    const int i = base + tid;
    const int keep = i < R.n ? kp[i] : 0;
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    const int pre = __popc(bal & ((1u << lane) - 1));
    if (lane == 0) warp_cnt[warp] = __popc(bal);
    __syncwarp();
    s_pos[tid] = keep ? pre : -1;
  }
  __syncthreads();
  if (tid < TOPK_CHUNK && s_pos[tid] >= 0) {
    s_pos[tid] += carry + (tid >= 32 ? warp_cnt[0] : 0);
    p.idx[R.idx0 + s_pos[tid]] = base + tid;
  }
  __syncthreads();
  // write the kept rows: (row, 16-byte piece) items spread over the whole CTA; the first PRE per thread are
  // already in registers, wider rows load the rest now
  uint4* dst = reinterpret_cast<uint4*>(p.out + R.out_row0 * p.D);
#pragma unroll
  for (int u = 0; u < PRE; ++u) {
    const int it = tid + u * 256;
    if (it < items) {
      const int t = it / vec, c4 = it - t * vec;
      const int pos = s_pos[t];
      if (pos >= 0) dst[static_cast<long long>(pos) * vec + c4] = pre[u];
    }
  }
#pragma unroll 4
  for (int it = tid + PRE * 256; it < items; it += 256) {
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
// element per thread 114 us on the device and 200 us with the counts read back; now 65 us with the counts read back.
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
__device__ __forceinline__ int nz_block_sum(int v, int* warp_sums) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = 0;
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
  __shared__ int sums[3][NZ_THREADS / 32];
  __shared__ unsigned short list[NZ_SUB];
  const NonZeroReq& R = nz_find(p);
  const int chunk = blockIdx.x - R.first, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long lo = chunk * R.chunk, hi = min(R.numel, lo + R.chunk);
  ptx::pdl_wait();
  ptx::pdl_launch();
  int before = 0, all = 0;
  for (int j = tid; j < R.chunks; j += NZ_THREADS) { const int c = R.count[j]; all += c; before += j < chunk ? c : 0; }
  before = nz_block_sum(before, sums[0]);
  const long long nnz = nz_block_sum(all, sums[1]);
  if (chunk == 0 && tid == 0) *R.count_out = nnz;
  long long off = before;
  for (long long base = lo; base < hi; base += NZ_SUB) {
    unsigned m = R.mask[(base >> 5) + tid];
    const int mine = __popc(m);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    __syncthreads();                     // the previous piece's list and sums have been read
    if (lane == 31) sums[2][warp] = inc;
    __syncthreads();
    int at = inc - mine, cnt = 0;
#pragma unroll
    for (int w = 0; w < NZ_THREADS / 32; ++w) { const int t = sums[2][w]; at += w < warp ? t : 0; cnt += t; }
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
