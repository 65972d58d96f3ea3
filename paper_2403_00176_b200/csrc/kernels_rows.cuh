// HBM-bound row kernels: the fp32 fused group (MatMul + bias + GELU + residual + LayerNorm in one
// kernel), LayerNorm / softmax over a run-time number of rows, and the generic fused
// broadcast-elementwise chain with an optional trailing row reduction (Section 4.2 of the paper:
// once RDP resolves every broadcast dim to "1" or "same", one fused loop nest suffices).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "ptx.cuh"

namespace sod2 {
namespace k {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float act_apply(int act, float x) {
  if (act == 1) return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
  if (act == 2) return fmaxf(x, 0.0f);
  if (act == 3) return 1.0f / (1.0f + __expf(-x));
  return x;
}

// ---------------------------------------------------------------------------------------------
// Y[M,N] = LN( act(X[M,K] W[K,N] + bias) + R ) in fp32 on CUDA cores; K, N <= 128, N % 32 == 0.
// W sits in shared memory, one warp per row, lane j owns columns j, j+32, ...; LayerNorm by warp
// shuffles. fp32 has to stay on FFMA: TF32 tensor cores cannot meet a 1e-5 tolerance.
struct MlpLnParams {
  const float* X; const float* W; const float* bias; const float* R; const float* gamma; const float* beta;
  float* Y;
  int M, K, N;
  int act;       // 0 none, 1 gelu(erf), 2 relu
  int has_ln;
  float eps;
};

template <int NC>  // NC = N / 32
__global__ void __launch_bounds__(256) fused_mlp_ln_f32(MlpLnParams p) {
  extern __shared__ float smem_f[];
  float* Ws = smem_f;                 // [K][N]
  float* Xs = smem_f + p.K * p.N;     // [8 warps][K]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // The group is a few thousand elements per request, so its time is its chain of round trips to memory:
  // everything the warp's first row needs (the row, the per-column constants, its residual) is requested
  // together with W, before the first wait.
  const int row0 = blockIdx.x * 8 + warp;
  float xpre[4];                      // K <= 128
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int kk = lane + 32 * q;
    xpre[q] = (row0 < p.M && kk < p.K) ? p.X[static_cast<long long>(row0) * p.K + kk] : 0.f;
  }
  float bias_r[NC], gam[NC], bet[NC], res[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int col = c * 32 + lane;
    bias_r[c] = p.bias ? p.bias[col] : 0.f;
    gam[c] = p.has_ln ? p.gamma[col] : 1.f;
    bet[c] = p.has_ln ? p.beta[col] : 0.f;
    res[c] = (p.R && row0 < p.M) ? p.R[static_cast<long long>(row0) * p.N + col] : 0.f;
  }
  if ((reinterpret_cast<uintptr_t>(p.W) & 15) == 0) {      // K * N is a multiple of 32
    const float4* W4 = reinterpret_cast<const float4*>(p.W);
    float4* Ws4 = reinterpret_cast<float4*>(Ws);
#pragma unroll 4
    for (int i = threadIdx.x; i < (p.K * p.N) >> 2; i += 256) Ws4[i] = W4[i];
  } else {
    for (int i = threadIdx.x; i < p.K * p.N; i += 256) Ws[i] = p.W[i];
  }
  __syncthreads();
  float* xs = Xs + warp * p.K;
  for (int row = row0; row < p.M; row += gridDim.x * 8) {
    if (row == row0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) { const int kk = lane + 32 * q; if (kk < p.K) xs[kk] = xpre[q]; }
    } else {
      for (int kk = lane; kk < p.K; kk += 32) xs[kk] = p.X[static_cast<long long>(row) * p.K + kk];
      if (p.R) {
#pragma unroll
        for (int c = 0; c < NC; ++c) res[c] = p.R[static_cast<long long>(row) * p.N + c * 32 + lane];
      }
    }
    __syncwarp();
    float acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.f;
    for (int kk = 0; kk < p.K; ++kk) {
      const float x = xs[kk];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = fmaf(x, Ws[kk * p.N + c * 32 + lane], acc[c]);
    }
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float v = acc[c];
      if (p.bias) v += bias_r[c];
      v = act_apply(p.act, v);
      if (p.R) v += res[c];
      acc[c] = v;
      s += v;
    }
    if (p.has_ln) {
      const float mu = warp_sum(s) / p.N;
      float q = 0.f;
#pragma unroll
      for (int c = 0; c < NC; ++c) { const float d = acc[c] - mu; q += d * d; }
      const float rstd = rsqrtf(warp_sum(q) / p.N + p.eps);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = (acc[c] - mu) * rstd * gam[c] + bet[c];
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) p.Y[static_cast<long long>(row) * p.N + c * 32 + lane] = acc[c];
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------------
// LayerNorm over the last dim of a packed [rows, D] bf16 matrix, rows known only at run time.
// One warp per row, 128-bit loads, the row lives in registers (D <= 256 * CH), fp32 math.
// FULL: D == CH * 256, every lane owns CH full vectors: no guards, so the loads of a row are issued
// back to back (a guard per vector puts every load into a basic block of its own and serialises their
// latencies).
template <int CH, bool FULL>
__global__ void __launch_bounds__(256) layernorm_bf16(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ gamma,
                                                       const __nv_bfloat16* __restrict__ beta, __nv_bfloat16* __restrict__ y,
                                                       long long rows, int D, float eps) {
  // gamma and beta are constants of the graph: fetch them before waiting for the previous kernel
  const int lane = threadIdx.x & 31;
  const long long row = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const int nvec = D >> 3;
  uint4 g4[CH], b4[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = FULL ? c * 32 + lane : min(c * 32 + lane, nvec - 1);
    g4[c] = reinterpret_cast<const uint4*>(gamma)[i];
    b4[c] = reinterpret_cast<const uint4*>(beta)[i];
  }
  ptx::pdl_launch();
  ptx::pdl_wait();
  if (row >= rows) return;
  const uint4* xr = reinterpret_cast<const uint4*>(x + row * D);
  float v[CH][8];
  float s = 0.f;
  // all loads of the row first, unconditionally (a lane past the row's end re-reads the last vector and
  // discards it): guarded loads would sit in basic blocks of their own and wait for one another
  uint4 u4[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) u4[c] = xr[FULL ? c * 32 + lane : min(c * 32 + lane, nvec - 1)];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const bool in = FULL || c * 32 + lane < nvec;
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u4[c]);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float2 f = __bfloat1622float2(h[t]);
      v[c][2 * t] = in ? f.x : 0.f;
      v[c][2 * t + 1] = in ? f.y : 0.f;
      s += in ? f.x + f.y : 0.f;
    }
  }
  const float mu = warp_sum(s) / D;
  float q = 0.f;
#pragma unroll
  for (int c = 0; c < CH; ++c)
    if (FULL || c * 32 + lane < nvec) {
#pragma unroll
      for (int t = 0; t < 8; ++t) { const float d = v[c][t] - mu; q += d * d; }
    }
  const float rstd = rsqrtf(warp_sum(q) / D + eps);
  uint4* yr = reinterpret_cast<uint4*>(y + row * D);
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = c * 32 + lane;
    if (FULL || i < nvec) {
      uint4 o;
      const __nv_bfloat162* gh = reinterpret_cast<const __nv_bfloat162*>(&g4[c]);
      const __nv_bfloat162* bh = reinterpret_cast<const __nv_bfloat162*>(&b4[c]);
      __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float2 gf = __bfloat1622float2(gh[t]), bf = __bfloat1622float2(bh[t]);
        oh[t] = __floats2bfloat162_rn((v[c][2 * t] - mu) * rstd * gf.x + bf.x, (v[c][2 * t + 1] - mu) * rstd * gf.y + bf.y);
      }
      yr[i] = o;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Finish of a split-K GEMM whose group ends in LayerNorm:
//   y = LayerNorm(sum_s acc[s] + bias + residual) * gamma + beta,  acc = fp32 [splits, rows, D] workspace
// holding the K ranges' partial products, added in slab order (deterministic).  The pre-normalisation
// row never exists in bf16.
template <int CH>
__global__ void __launch_bounds__(256) splitk_ln_finish(const float* __restrict__ acc, int splits, const __nv_bfloat16* __restrict__ bias,
                                                         const __nv_bfloat16* __restrict__ res, long long ldr,
                                                         const __nv_bfloat16* __restrict__ gamma, const __nv_bfloat16* __restrict__ beta,
                                                         __nv_bfloat16* __restrict__ y, long long rows, int D, float eps) {
  const int lane = threadIdx.x & 31;
  const long long row = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const int nvec = D >> 3;
  uint4 g4[CH], b4[CH], c4[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = c * 32 + lane;
    if (i < nvec) {
      g4[c] = reinterpret_cast<const uint4*>(gamma)[i]; b4[c] = reinterpret_cast<const uint4*>(beta)[i];
      c4[c] = bias ? reinterpret_cast<const uint4*>(bias)[i] : make_uint4(0, 0, 0, 0);
    }
  }
  ptx::pdl_launch();
  ptx::pdl_wait();
  if (row >= rows) return;
  const float4* ar = reinterpret_cast<const float4*>(acc + row * D);
  const long long slab4 = rows * D / 4;      // float4 per slab
  const uint4* rr = res ? reinterpret_cast<const uint4*>(res + row * ldr) : nullptr;
  float v[CH][8];
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = c * 32 + lane;
    if (i < nvec) {
      float4 a0 = ar[2 * i], a1 = ar[2 * i + 1];
      for (int sp = 1; sp < splits; ++sp) {
        const float4 b0 = ar[sp * slab4 + 2 * i], b1 = ar[sp * slab4 + 2 * i + 1];
        a0.x += b0.x; a0.y += b0.y; a0.z += b0.z; a0.w += b0.w;
        a1.x += b1.x; a1.y += b1.y; a1.z += b1.z; a1.w += b1.w;
      }
      const uint4 ru = rr ? rr[i] : make_uint4(0, 0, 0, 0);
      const __nv_bfloat162* rh = reinterpret_cast<const __nv_bfloat162*>(&ru);
      const __nv_bfloat162* ch = reinterpret_cast<const __nv_bfloat162*>(&c4[c]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float2 rf = __bfloat1622float2(rh[t]), cf = __bfloat1622float2(ch[t]);
        v[c][2 * t] = a[2 * t] + cf.x + rf.x;
        v[c][2 * t + 1] = a[2 * t + 1] + cf.y + rf.y;
        s += v[c][2 * t] + v[c][2 * t + 1];
      }
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) v[c][t] = 0.f;
    }
  }
  const float mu = warp_sum(s) / D;
  float q = 0.f;
#pragma unroll
  for (int c = 0; c < CH; ++c)
    if (c * 32 + lane < nvec) {
#pragma unroll
      for (int t = 0; t < 8; ++t) { const float d = v[c][t] - mu; q += d * d; }
    }
  const float rstd = rsqrtf(warp_sum(q) / D + eps);
  uint4* yr = reinterpret_cast<uint4*>(y + row * D);
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = c * 32 + lane;
    if (i < nvec) {
      uint4 o;
      const __nv_bfloat162* gh = reinterpret_cast<const __nv_bfloat162*>(&g4[c]);
      const __nv_bfloat162* bh = reinterpret_cast<const __nv_bfloat162*>(&b4[c]);
      __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float2 gf = __bfloat1622float2(gh[t]), bf = __bfloat1622float2(bh[t]);
        oh[t] = __floats2bfloat162_rn((v[c][2 * t] - mu) * rstd * gf.x + bf.x, (v[c][2 * t + 1] - mu) * rstd * gf.y + bf.y);
      }
      yr[i] = o;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Generic fused chain (the paper's Fig. 4 form): v = load(in0); v = op_i(v [, operand_i]) ...; optional softmax /
// LayerNorm over the last dim; store.  Index space = the group's output [d0..d3] (rank <= 4 after
// right-alignment); every operand is read through its own strides, 0 on the dims RDP resolved to "broadcast".
// All requests of a batch run in ONE launch through a request table (up to CHAIN_MAX_REQ entries): the operands of
// the requests live in the same packed buffers, so an entry is extents, element offsets and strides.
//   chain_elementwise       no trailing reduction: vectors over the flat output index, see the kernel
//   chain_rowreduce_warp    a warp per row (rows up to ROWRED_WARP_COLS), the row staged in the warp's slice of shared
//                           memory, statistics by shuffles: no CTA barrier, eight rows in flight per CTA
//   chain_rowreduce         a CTA per row for longer rows
constexpr int CHAIN_NV = 4;                  // chain_elementwise: 16-byte vectors per thread
constexpr int CHAIN_MAX_OPS = 8;
constexpr int CHAIN_MAX_REQ = 8;
constexpr int ROWRED_WARP_COLS = 2048;
enum ChainOp : int { C_ADD = 0, C_SUB, C_RSUB, C_MUL, C_DIV, C_RDIV, C_RELU, C_GELU, C_SIGMOID };
enum ChainRed : int { RED_NONE = 0, RED_SOFTMAX = 1, RED_LAYERNORM = 2 };

// How an operand is read by chain_elementwise, per request.
//   FLAT   laid out like the output: element e of the output reads element e of the operand, 16-byte vectors
//   BCAST  one value along the last (collapsed) dim
//   VEC    unit stride along the last dim and 16-byte vectors wherever a column is a multiple of 8 (a bias row)
//   INNER  anything else: one load per element
//   SCALAR a constant of the graph (base == nullptr)
enum ChainCls : int { CC_FLAT = 0, CC_BCAST = 1, CC_INNER = 2, CC_SCALAR = 3, CC_VEC = 4 };
struct ChainReq {
  int dim[4];                               // output extents (chain_elementwise: adjacent dims collapsed where every operand allows)
  int numel;                                // chain_elementwise: elements of the output
  int first_vec;                            // chain_elementwise: first operand that is not one value along a row, -1 if none
  int fast;                                 // chain_elementwise: no operand is CC_INNER, all are of the output's type, rows are a vector or longer
  int cls[1 + CHAIN_MAX_OPS];               // ChainCls
  long long first;                          // first work item of this request in the launch (chain_elementwise: first tile)
  long long out_off;                        // elements from `out`
  long long off[1 + CHAIN_MAX_OPS];         // elements from base[k]; k = 0 is in0, k = 1 + i operand i
  int stride[1 + CHAIN_MAX_OPS][4];         // elements
};
struct ChainBatch {
  const void* base[1 + CHAIN_MAX_OPS];      // nullptr: use scalar[k]
  float scalar[1 + CHAIN_MAX_OPS];
  int is_bf16[1 + CHAIN_MAX_OPS];
  int op[CHAIN_MAX_OPS];
  int n_ops;
  void* out;                                // every request's output instance is contiguous
  int out_bf16;
  int red;
  const void* gamma; const void* beta; int gb_bf16; float eps;
  int n_req;
  int vec_ok;                               // chain_elementwise: `out` is 16-byte aligned
  long long total;                          // work items of all requests (chain_elementwise: tiles)
  ChainReq r[CHAIN_MAX_REQ];
};

__device__ __forceinline__ int chain_find_req(const ChainBatch& p, long long item) {
  int ri = 0;
  while (ri + 1 < p.n_req && item >= p.r[ri + 1].first) ++ri;
  return ri;
}
__device__ __forceinline__ float chain_apply(int op, float v, float w) {
  switch (op) {
    case C_ADD: return v + w;
    case C_SUB: return v - w;
    case C_RSUB: return w - v;
    case C_MUL: return v * w;
    case C_DIV: return v / w;
    case C_RDIV: return w / v;
    case C_RELU: return fmaxf(v, 0.f);
    case C_GELU: return act_apply(1, v);
    default: return act_apply(3, v);
  }
}
__device__ __forceinline__ float chain_load1(const ChainBatch& p, const ChainReq& R, int k, int i0, int i1, int i2, int i3) {
  if (!p.base[k]) return p.scalar[k];
  const long long off = R.off[k] + static_cast<long long>(i0) * R.stride[k][0] + static_cast<long long>(i1) * R.stride[k][1] +
                        static_cast<long long>(i2) * R.stride[k][2] + static_cast<long long>(i3) * R.stride[k][3];
  return p.is_bf16[k] ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.base[k])[off]) : reinterpret_cast<const float*>(p.base[k])[off];
}
__device__ __forceinline__ float chain_eval(const ChainBatch& p, const ChainReq& R, int i0, int i1, int i2, int i3) {
  float v = chain_load1(p, R, 0, i0, i1, i2, i3);
  for (int k = 0; k < p.n_ops; ++k) {
    const int op = p.op[k];
    v = chain_apply(op, v, op >= C_RELU ? 0.f : chain_load1(p, R, 1 + k, i0, i1, i2, i3));
  }
  return v;
}
__device__ __forceinline__ void chain_store1(const ChainBatch& p, long long lin, float v) {
  if (p.out_bf16) reinterpret_cast<__nv_bfloat16*>(p.out)[lin] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(p.out)[lin] = v;
}

__device__ __forceinline__ void chain_split_row(const ChainReq& R, int row, int* i0, int* i1, int* i2) {
  *i0 = 0; *i1 = 0; *i2 = row;
  if (R.dim[0] * R.dim[1] > 1) {        // after collapsing, most chains have one leading dim left
    const unsigned t2 = static_cast<unsigned>(row) / static_cast<unsigned>(R.dim[2]);
    *i2 = row - static_cast<int>(t2) * R.dim[2];
    *i0 = static_cast<int>(t2 / static_cast<unsigned>(R.dim[1]));
    *i1 = static_cast<int>(t2) - *i0 * R.dim[1];
  }
}

template <bool BF16> struct ChainVec;     // one 16-byte vector
template <> struct ChainVec<true> {
  static constexpr int E = 8;
  using Raw = uint4;
  __device__ static void unpack(const Raw& u, float* f) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int t = 0; t < 4; ++t) { const float2 q = __bfloat1622float2(h[t]); f[2 * t] = q.x; f[2 * t + 1] = q.y; }
  }
  __device__ static Raw pack(const float* f) {
    Raw u;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
    for (int t = 0; t < 4; ++t) h[t] = __floats2bfloat162_rn(f[2 * t], f[2 * t + 1]);
    return u;
  }
};
template <> struct ChainVec<false> {
  static constexpr int E = 4;
  using Raw = float4;
  __device__ static void unpack(const Raw& u, float* f) { f[0] = u.x; f[1] = u.y; f[2] = u.z; f[3] = u.w; }
  __device__ static Raw pack(const float* f) { return make_float4(f[0], f[1], f[2], f[3]); }
};

// The NV vectors of one thread: vector n is the outputs from flat index e + n * 256 vectors on.  No operand is CC_INNER
// (the host's `fast`).  UNI: all lie in row `row`, vector 0 at column i3.  Otherwise every vector finds its own row; one
// that reaches past the row's end takes broadcast operands from two rows (rows are at least a vector long then), one that
// lies past the last element (n >= live) is read from where vector 0 is and not stored.
template <bool BF16, bool UNI>
__device__ __forceinline__ void chain_eval_vec(const ChainBatch& p, const ChainReq& R, int e, int row, int i3, int live) {
  using V = ChainVec<BF16>;
  constexpr int E = V::E, NV = CHAIN_NV, NR = UNI ? 1 : NV;
  int i0[NR], i1[NR], i2[NR], col[NR], cut[NR];     // cut: elements of the vector before the row's end
#pragma unroll
  for (int n = 0; n < NR; ++n) {
    int r = row;
    col[n] = i3;
    if constexpr (!UNI) {
      const int en = n < live ? e + n * (256 * E) : e;
      r = static_cast<int>(static_cast<unsigned>(en) / static_cast<unsigned>(R.dim[3]));
      col[n] = en - r * R.dim[3];
    }
    cut[n] = UNI ? E : R.dim[3] - col[n];
    chain_split_row(R, r, &i0[n], &i1[n], &i2[n]);
  }
  auto one_value = [&](int k) { return R.cls[k] == CC_BCAST || R.cls[k] == CC_SCALAR; };
  auto load = [&](int k, typename V::Raw* u) {
    const char* base = static_cast<const char*>(p.base[k]) + R.off[k] * (16 / E);
    if (R.cls[k] == CC_FLAT) {
      const typename V::Raw* src = reinterpret_cast<const typename V::Raw*>(base) + e / E;
#pragma unroll
      for (int n = 0; n < NV; ++n) u[n] = src[(UNI || n < live) ? n * 256 : 0];
    } else {
#pragma unroll
      for (int n = 0; n < NV; ++n) {
        const int m = UNI ? 0 : n;
        const long long off = static_cast<long long>(i0[m]) * R.stride[k][0] + static_cast<long long>(i1[m]) * R.stride[k][1] +
                              static_cast<long long>(i2[m]) * R.stride[k][2] + col[m] + (UNI ? n * (256 * E) : 0);
        u[n] = reinterpret_cast<const typename V::Raw*>(base)[off / E];
      }
    }
  };
  // one value of operand k for the row of vector n, or for the row after it
  auto value = [&](int k, int n) { return chain_load1(p, R, k, i0[n], i1[n], i2[n], 0); };
  auto value_after = [&](int k, int n) {
    int a0 = i0[n], a1 = i1[n], a2 = i2[n] + 1;
    if (a2 == R.dim[2]) { a2 = 0; if (++a1 == R.dim[1]) { a1 = 0; ++a0; } }
    return chain_load1(p, R, k, a0, a1, a2, 0);
  };
  float v[NV][E];
  typename V::Raw u[NV];
  // the first vector operand is requested before anything else is worked out
  if (R.first_vec >= 0) load(R.first_vec, u);
  int k0 = 0;
  // While every operand so far is one value along the row the values of a vector are one value (two where it straddles
  // rows): that prefix of the chain (Fig. 4: Sigmoid of the [I,1,1] operand) is not evaluated for every element.
  if (one_value(0)) {
    k0 = R.first_vec < 0 ? p.n_ops : R.first_vec - 1;
    float x[NR], y[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) { x[n] = value(0, n); y[n] = (UNI || cut[n] >= E) ? x[n] : value_after(0, n); }
    for (int k = 0; k < k0; ++k) {
      const int op = p.op[k];
#pragma unroll
      for (int n = 0; n < NR; ++n) {
        const float w = op >= C_RELU ? 0.f : value(1 + k, n);
        x[n] = chain_apply(op, x[n], w);
        if (!UNI) y[n] = cut[n] >= E ? x[n] : chain_apply(op, y[n], op >= C_RELU ? 0.f : value_after(1 + k, n));
      }
    }
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
      for (int t = 0; t < E; ++t) v[n][t] = UNI ? x[0] : t < cut[n % NR] ? x[n % NR] : y[n % NR];
  } else {
#pragma unroll
    for (int n = 0; n < NV; ++n) V::unpack(u[n], v[n]);
  }
#pragma unroll 1
  for (int k = k0; k < p.n_ops; ++k) {
    const int op = p.op[k];
    if (op >= C_RELU) {
      // the operator is chosen once per thread; the elements run through straight-line code
#define SOD2_CHAIN_UNARY(OP_) { _Pragma("unroll") for (int n = 0; n < NV; ++n) _Pragma("unroll") for (int t = 0; t < E; ++t) v[n][t] = chain_apply(OP_, v[n][t], 0.f); }
      if (op == C_RELU) SOD2_CHAIN_UNARY(C_RELU)
      else if (op == C_GELU) SOD2_CHAIN_UNARY(C_GELU)
      else SOD2_CHAIN_UNARY(C_SIGMOID)
#undef SOD2_CHAIN_UNARY
      continue;
    }
    float x[NR], y[NR];
    const bool one = one_value(1 + k);
    if (one) {
#pragma unroll
      for (int n = 0; n < NR; ++n) { x[n] = value(1 + k, n); y[n] = (UNI || cut[n] >= E) ? x[n] : value_after(1 + k, n); }
    } else if (1 + k != R.first_vec) {
      load(1 + k, u);
    }
    switch (op) {
#define SOD2_CHAIN_CASE(OP_)                                                                                   \
      case OP_:                                                                                                \
        _Pragma("unroll") for (int n = 0; n < NV; ++n) {                                                       \
          float w[E];                                                                                          \
          V::unpack(u[n], w);                                                                                  \
          _Pragma("unroll") for (int t = 0; t < E; ++t)                                                        \
            v[n][t] = chain_apply(OP_, v[n][t], !one ? w[t] : (UNI || t < cut[n % NR]) ? x[n % NR] : y[n % NR]); \
        }                                                                                                      \
        break;
      SOD2_CHAIN_CASE(C_ADD)
      SOD2_CHAIN_CASE(C_SUB)
      SOD2_CHAIN_CASE(C_RSUB)
      SOD2_CHAIN_CASE(C_MUL)
      SOD2_CHAIN_CASE(C_DIV)
      default:
      SOD2_CHAIN_CASE(C_RDIV)
#undef SOD2_CHAIN_CASE
    }
  }
  typename V::Raw* dst = reinterpret_cast<typename V::Raw*>(static_cast<char*>(p.out) + R.out_off * (16 / E)) + e / E;
#pragma unroll
  for (int n = 0; n < NV; ++n)
    if (UNI || n < live) dst[n * 256] = V::pack(v[n]);
}

// Elementwise chains, bound by HBM.  Work is cut over the FLAT output index, not over rows: a tile is 1024 16-byte
// vectors of consecutive outputs of one request, a thread takes four of them, so neither a row length that is no
// multiple of 8 nor a request of such rows among others costs the batch its 16-byte accesses.  The host collapses
// adjacent dims wherever every operand allows it (Fig. 4: [I,J,K] -> [I, J*K]), so that most tiles lie inside one row:
// then the row index and every broadcast operand are the same for the whole CTA and cost one evaluation per thread and
// tile.  In the other tiles every vector finds its own row (its loads in flight with the others': one after the other
// they made these tiles four round trips long, and the last of them the kernel's tail).  A request's last, incomplete
// vector, rows shorter than a vector, operands of other strides and operands of mixed types go element by element.
// Measured on B200, Fig. 4 chain in bf16, requests 64x128x784 + 37x101x333 + 64x77x1024 + 3x250x49 (51 MB):
// 120 -> 16 us a pass (0.42 -> 3.2 TB/s): one request with rows of 333 or 49 used to put the whole batch on one element
// per thread and three 64-bit divisions.  Now bound by HBM latency and instruction fetch in short CTAs, not by bytes.
template <bool BF16>
__global__ void __launch_bounds__(256, 4) chain_elementwise(const __grid_constant__ ChainBatch p) {
  constexpr int E = ChainVec<BF16>::E, TILE = 256 * CHAIN_NV * E;
  ptx::pdl_wait();
  ptx::pdl_launch();
  const ChainReq& R = p.r[chain_find_req(p, blockIdx.x)];
  const int e0 = (static_cast<int>(blockIdx.x) - static_cast<int>(R.first)) * TILE;
  const int inner = R.dim[3];
  auto by_element = [&](int e) {
    const int row = static_cast<int>(static_cast<unsigned>(e) / static_cast<unsigned>(inner));
    int i0, i1, i2;
    chain_split_row(R, row, &i0, &i1, &i2);
    chain_store1(p, R.out_off + e, chain_eval(p, R, i0, i1, i2, e - row * inner));
  };
  // (a request may have up to 2^31 - 1 elements: its last tile must not be added to)
  const int rest = R.numel - e0;
  if (!(p.vec_ok && R.fast)) {
    for (int d = threadIdx.x; d < min(TILE, rest); d += 256) by_element(e0 + d);
    return;
  }
  const int row0 = static_cast<int>(static_cast<unsigned>(e0) / static_cast<unsigned>(inner));
  const int col0 = e0 - row0 * inner;
  const int d = threadIdx.x * E;
  if (TILE <= inner - col0) {
    chain_eval_vec<BF16, true>(p, R, e0 + d, row0, col0 + d, CHAIN_NV);
    return;
  }
  const int whole = rest / E * E;                        // the tail behind the last whole vector: one element per thread
  const int left = whole - d;
  if (left > 0) chain_eval_vec<BF16, false>(p, R, e0 + d, 0, 0, min(CHAIN_NV, (left + 256 * E - 1) / (256 * E)));
  if (whole < TILE && whole + static_cast<int>(threadIdx.x) < rest) by_element(e0 + whole + threadIdx.x);
}

__device__ __forceinline__ void chain_row_index(const ChainReq& R, long long row, int* i0, int* i1, int* i2) {
  *i2 = static_cast<int>(row % R.dim[2]); row /= R.dim[2];
  *i1 = static_cast<int>(row % R.dim[1]);
  *i0 = static_cast<int>(row / R.dim[1]);
}
__device__ __forceinline__ float chain_gb(const ChainBatch& p, const void* v, int c) {
  return p.gb_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(v)[c]) : reinterpret_cast<const float*>(v)[c];
}

// trailing row reduction, a warp per row: work item = row; dynamic shared memory = 8 rows of `max_cols` floats
__global__ void __launch_bounds__(256) chain_rowreduce_warp(const __grid_constant__ ChainBatch p, int max_cols) {
  extern __shared__ float rowbuf_all[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* rowbuf = rowbuf_all + static_cast<size_t>(warp) * max_cols;
  for (long long item = static_cast<long long>(blockIdx.x) * 8 + warp; item < p.total; item += static_cast<long long>(gridDim.x) * 8) {
    const ChainReq& R = p.r[chain_find_req(p, item)];
    const long long row = item - R.first;
    const int cols = R.dim[3];
    int i0, i1, i2;
    chain_row_index(R, row, &i0, &i1, &i2);
    float m = -INFINITY, s = 0.f;
    for (int c = lane; c < cols; c += 32) {
      const float v = chain_eval(p, R, i0, i1, i2, c);
      rowbuf[c] = v;
      m = fmaxf(m, v);
      s += v;
    }
    const float st0 = p.red == RED_SOFTMAX ? warp_max(m) : warp_sum(s) / cols;
    float q = 0.f;
    for (int c = lane; c < cols; c += 32) {
      if (p.red == RED_SOFTMAX) { const float e = __expf(rowbuf[c] - st0); rowbuf[c] = e; q += e; }
      else { const float d = rowbuf[c] - st0; q += d * d; }
    }
    q = warp_sum(q);
    const float st1 = p.red == RED_SOFTMAX ? 1.0f / q : rsqrtf(q / cols + p.eps);
    const long long obase = R.out_off + row * cols;
    for (int c = lane; c < cols; c += 32) {
      const float v = p.red == RED_SOFTMAX ? rowbuf[c] * st1 : (rowbuf[c] - st0) * st1 * chain_gb(p, p.gamma, c) + chain_gb(p, p.beta, c);
      chain_store1(p, obase + c, v);
    }
    __syncwarp();
  }
}

// trailing row reduction, a CTA per row (long rows): dynamic shared memory = one row
__global__ void __launch_bounds__(256) chain_rowreduce(const __grid_constant__ ChainBatch p) {
  extern __shared__ float rowbuf[];
  __shared__ float red[8];
  __shared__ float bc[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long item = blockIdx.x; item < p.total; item += gridDim.x) {
    const ChainReq& R = p.r[chain_find_req(p, item)];
    const long long row = item - R.first;
    const int cols = R.dim[3];
    int i0, i1, i2;
    chain_row_index(R, row, &i0, &i1, &i2);
    float m = -INFINITY, s = 0.f;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
      const float v = chain_eval(p, R, i0, i1, i2, c);
      rowbuf[c] = v;
      m = fmaxf(m, v);
      s += v;
    }
    // first statistic: max (softmax) or mean (LayerNorm)
    float a = p.red == RED_SOFTMAX ? warp_max(m) : warp_sum(s);
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = red[0];
      for (int w = 1; w < 8; ++w) t = p.red == RED_SOFTMAX ? fmaxf(t, red[w]) : t + red[w];
      bc[0] = p.red == RED_SOFTMAX ? t : t / cols;
    }
    __syncthreads();
    const float st0 = bc[0];
    float q = 0.f;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
      if (p.red == RED_SOFTMAX) { const float e = __expf(rowbuf[c] - st0); rowbuf[c] = e; q += e; }
      else { const float d = rowbuf[c] - st0; q += d * d; }
    }
    q = warp_sum(q);
    __syncthreads();
    if (lane == 0) red[warp] = q;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (int w = 0; w < 8; ++w) t += red[w];
      bc[1] = p.red == RED_SOFTMAX ? 1.0f / t : rsqrtf(t / cols + p.eps);
    }
    __syncthreads();
    const float st1 = bc[1];
    const long long obase = R.out_off + row * cols;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
      const float v = p.red == RED_SOFTMAX ? rowbuf[c] * st1 : (rowbuf[c] - st0) * st1 * chain_gb(p, p.gamma, c) + chain_gb(p, p.beta, c);
      chain_store1(p, obase + c, v);
    }
    __syncthreads();
  }
}

}  // namespace k
}  // namespace sod2
