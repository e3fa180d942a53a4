// Attention of one encoder layer in fp32, head width 64: one kernel forward, one backward, in the place of
// the batched products and the softmax passes between them (3 and 5 launches).
//   forward   P = softmax over valid keys of scale * Q K^T (kept for the backward), C = P V
//   backward  dP = dC V^T, dS = P o (dP - rowsum(dC o C)) * scale, dQ = dS K, dK = dS^T Q, dV = P^T dC
// A block of 128 threads owns 32 rows of one (sequence, head): queries in the forward and for dQ, keys for
// dK and dV, which form their part of dP again with the operands exchanged, so that no sums cross
// blocks.  The 32 x S scores stay in shared memory; the other operand passes through two buffers of 64
// rows filled by asynchronous copies one step ahead.  A thread holds 4 x 4 outputs of packed multiply-adds.
// Bound by launches and the chain copy - product - softmax - product where sequences are few, by the
// shared-memory reads of the products otherwise (2 x 4 outputs on twice the threads: backward 36.7 -> 51.6 us).
// 16 heads x 64 keys: forward 8.3 -> 5.5 us and one launch in the place of three, backward 13.0 -> 7.8 us and
// one for five; 96 x 128 keys: 17 and 37 us.  A step of two layers is faster with it at every batch and head count
// tried, 16 to 1536 items (8 x 64 keys x 2 heads 310 -> 296 us, 32 x 128 x 12 3276 -> 3157, 64 x 128 x 16 9445 -> 9376,
// 128 x 128 x 12 11768 -> 11533), so the rule looks at the row length only.  Rows of at most 128 keys: steps of 2 to 3 layers with
// 256 keys take the same time either way (476 and 477 us, 2 234 and 2 219 us), with 512 keys the batched
// products and their larger tiles are ahead (517 against 551 us).
#include <mutex>
#include <stdio.h>

#include "common.cuh"
#include "gemm.h"

namespace mslt {
namespace {

constexpr int FA_QT = 32;     // rows of a block
constexpr int FA_KC = 64;     // rows of a buffer
constexpr int FA_D = 64;      // head width
constexpr int FA_PITCH = 68;  // floats between rows of a tile: 16-byte reads down a column hit all banks
constexpr int FA_RPT = 4;     // rows of a thread's 4-column tile
constexpr int FA_NT = 16 * FA_QT / FA_RPT;
constexpr int FA_TPR = FA_NT / FA_QT;  // threads of a row where each row is taken by itself

struct AttnF32Params {
  const float *qkv, *P, *C, *dC;
  float *P_out, *C_out, *dqkv;
  const int* seq_lens;
  int S, A, tiles;
  float scale;
};

// rows 0 .. ROWS - 1 of a tile from global rows of pitch ld; rows from n on are zero
template <int ROWS>
__device__ __forceinline__ void fa_load(float* dst, const float* src, int n, int64_t ld) {
#pragma unroll
  for (int i = 0; i < ROWS * (FA_D / 4) / FA_NT; i++) {
    const int idx = threadIdx.x + i * FA_NT, r = idx >> 4, c = (idx & 15) * 4;
    const int bytes = r < n ? 16 : 0;
    const float* g = src + (r < n ? r * ld : 0) + c;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + r * FA_PITCH + c)),
                 "l"(g), "r"(bytes)
                 : "memory");
  }
}
__device__ __forceinline__ void fa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void fa_wait() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// s[i][c] = a row (FA_RPT ty + i) . b row (tx + 16 c)
__device__ __forceinline__ void fa_scores(const float* a, const float* b, int ty, int tx, float (&s)[FA_RPT][4]) {
  float2 acc[FA_RPT][4];
#pragma unroll
  for (int i = 0; i < FA_RPT; i++)
#pragma unroll
    for (int c = 0; c < 4; c++) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int k = 0; k < FA_D; k += 4) {
    float4 x[FA_RPT], y[4];
#pragma unroll
    for (int i = 0; i < FA_RPT; i++) x[i] = *reinterpret_cast<const float4*>(a + (FA_RPT * ty + i) * FA_PITCH + k);
#pragma unroll
    for (int c = 0; c < 4; c++) y[c] = *reinterpret_cast<const float4*>(b + (tx + 16 * c) * FA_PITCH + k);
#pragma unroll
    for (int i = 0; i < FA_RPT; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) {
        acc[i][c] = __ffma2_rn(make_float2(x[i].x, x[i].y), make_float2(y[c].x, y[c].y), acc[i][c]);
        acc[i][c] = __ffma2_rn(make_float2(x[i].z, x[i].w), make_float2(y[c].z, y[c].w), acc[i][c]);
      }
  }
#pragma unroll
  for (int i = 0; i < FA_RPT; i++)
#pragma unroll
    for (int c = 0; c < 4; c++) s[i][c] = acc[i][c].x + acc[i][c].y;
}

// o[i] (columns 4 tx ..) += sum over j < n of p[FA_RPT ty + i][j] * v[j]; n a multiple of 4
__device__ __forceinline__ void fa_values(const float* p, int pitch, const float* v, int n, int ty, int tx, float2 (&o)[FA_RPT][2]) {
#pragma unroll 4
  for (int j = 0; j < n; j += 4) {
    float4 w[FA_RPT], y[4];
#pragma unroll
    for (int i = 0; i < FA_RPT; i++) w[i] = *reinterpret_cast<const float4*>(p + (FA_RPT * ty + i) * pitch + j);
#pragma unroll
    for (int e = 0; e < 4; e++) y[e] = *reinterpret_cast<const float4*>(v + (j + e) * FA_PITCH + 4 * tx);
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
      for (int i = 0; i < FA_RPT; i++) {
        const float f = e == 0 ? w[i].x : e == 1 ? w[i].y : e == 2 ? w[i].z : w[i].w;
        o[i][0] = __ffma2_rn(make_float2(f, f), make_float2(y[e].x, y[e].y), o[i][0]);
        o[i][1] = __ffma2_rn(make_float2(f, f), make_float2(y[e].z, y[e].w), o[i][1]);
      }
  }
}

__device__ __forceinline__ void fa_store(float* dst, int64_t ld, int n, int ty, int tx, const float2 (&o)[FA_RPT][2]) {
#pragma unroll
  for (int i = 0; i < FA_RPT; i++)
    if (FA_RPT * ty + i < n) *reinterpret_cast<float4*>(dst + (FA_RPT * ty + i) * ld + 4 * tx) = make_float4(o[i][0].x, o[i][0].y, o[i][1].x, o[i][1].y);
}

__device__ __forceinline__ void fa_zero(float2 (&o)[FA_RPT][2]) {
#pragma unroll
  for (int i = 0; i < FA_RPT; i++) o[i][0] = o[i][1] = make_float2(0.f, 0.f);
}

__global__ void __launch_bounds__(FA_NT, 3) attn_f32_fwd_kernel(const AttnF32Params p) {
  extern __shared__ __align__(16) float fa_smem[];
  float* tile = fa_smem;
  float* buf = tile + FA_QT * FA_PITCH;
  float* sc = buf + 2 * FA_KC * FA_PITCH;
  const int S = p.S, pitch = S + 4;  // S % 8 == 0, so 16-byte reads down a column of scores hit all banks too
  const int z = blockIdx.x / p.tiles, q0 = (blockIdx.x - z * p.tiles) * FA_QT;
  const int b = z / p.A, h = z - b * p.A;
  const int64_t H = (int64_t)p.A * FA_D, ld = 3 * H;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  pdl_begin();
  const int len = p.seq_lens ? min(max(p.seq_lens[b], 1), S) : S;
  const float* base = p.qkv + (int64_t)b * S * ld + h * FA_D;
  const int n = (len + FA_KC - 1) / FA_KC;  // K blocks, then as many V blocks
  auto issue = [&](int t) {
    if (t < 2 * n) {
      const int r0 = (t < n ? t : t - n) * FA_KC;
      fa_load<FA_KC>(buf + (t & 1) * FA_KC * FA_PITCH, base + (t < n ? H : 2 * H) + r0 * ld, S - r0, ld);
    }
    fa_commit();
  };
  fa_load<FA_QT>(tile, base + q0 * ld, S - q0, ld);
  issue(0);
  issue(1);
  for (int t = 0; t < n; t++) {
    fa_wait();
    __syncthreads();
    float s[FA_RPT][4];
    fa_scores(tile, buf + (t & 1) * FA_KC * FA_PITCH, ty, tx, s);
#pragma unroll
    for (int i = 0; i < FA_RPT; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const int j = t * FA_KC + tx + 16 * c;
        if (j < S) sc[(FA_RPT * ty + i) * pitch + j] = s[i][c] * p.scale;
      }
    __syncthreads();
    issue(t + 2);
  }
  // softmax: FA_TPR threads a row, 16 bytes at a time
  {
    const int r = threadIdx.x / FA_TPR, j1 = (threadIdx.x % FA_TPR) * 4;
    float* row = sc + r * pitch;
    float m = -INFINITY;
#pragma unroll 4
    for (int j = j1; j < len; j += 4 * FA_TPR) {
      const float4 v = *reinterpret_cast<const float4*>(row + j);
      m = fmaxf(m, v.x);
      if (j + 1 < len) m = fmaxf(m, v.y);
      if (j + 2 < len) m = fmaxf(m, v.z);
      if (j + 3 < len) m = fmaxf(m, v.w);
    }
#pragma unroll
    for (int o = 1; o < FA_TPR; o *= 2) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float sum = 0.f;
#pragma unroll 4
    for (int j = j1; j < len; j += 4 * FA_TPR) {
      float4 v = *reinterpret_cast<const float4*>(row + j);
      v.x = expf(v.x - m);
      v.y = j + 1 < len ? expf(v.y - m) : 0.f;
      v.z = j + 2 < len ? expf(v.z - m) : 0.f;
      v.w = j + 3 < len ? expf(v.w - m) : 0.f;
      *reinterpret_cast<float4*>(row + j) = v;
      sum += (v.x + v.y) + (v.z + v.w);
    }
#pragma unroll
    for (int o = 1; o < FA_TPR; o *= 2) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float inv = 1.0f / sum;
    float* g = p.P_out && q0 + r < S ? p.P_out + ((int64_t)z * S + q0 + r) * S : nullptr;
#pragma unroll 4
    for (int j = j1; j < S; j += 4 * FA_TPR) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < len) {
        v = *reinterpret_cast<const float4*>(row + j);
        v.x *= inv; v.y *= inv; v.z *= inv; v.w *= inv;
      }
      *reinterpret_cast<float4*>(row + j) = v;
      if (g) *reinterpret_cast<float4*>(g + j) = v;
    }
  }
  float2 o[FA_RPT][2];
  fa_zero(o);
  for (int t = n; t < 2 * n; t++) {
    fa_wait();
    __syncthreads();
    const int j0 = (t - n) * FA_KC;
    fa_values(sc + j0, pitch, buf + (t & 1) * FA_KC * FA_PITCH, min(FA_KC, S - j0), ty, tx, o);
    __syncthreads();
    issue(t + 2);
  }
  fa_store(p.C_out + ((int64_t)b * S + q0) * H + h * FA_D, H, S - q0, ty, tx, o);
}

__global__ void __launch_bounds__(FA_NT, 3) attn_f32_bwd_kernel(const AttnF32Params p) {
  extern __shared__ __align__(16) float fa_smem[];
  float* tile = fa_smem;
  float* buf = tile + FA_QT * FA_PITCH;
  float* sc = buf + 2 * FA_KC * FA_PITCH;
  const int S = p.S, pitch = S + 4;
  float* delta = sc + FA_QT * pitch;  // rowsum(dC o C): of the block's queries, or of all
  const int per_mode = gridDim.x / 2;
  const bool keys = (int)blockIdx.x < per_mode;  // dK and dV: the longer blocks, started first
  const int x = keys ? blockIdx.x : blockIdx.x - per_mode;
  const int z = x / p.tiles, r0 = (x - z * p.tiles) * FA_QT;
  const int b = z / p.A, h = z - b * p.A;
  const int64_t H = (int64_t)p.A * FA_D, ld = 3 * H;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_begin();
  const int len = p.seq_lens ? min(max(p.seq_lens[b], 1), S) : S;
  const float* base = p.qkv + (int64_t)b * S * ld + h * FA_D;
  const float* C = p.C + (int64_t)b * S * H + h * FA_D;
  const float* dC = p.dC + (int64_t)b * S * H + h * FA_D;
  const float* P = p.P + (int64_t)z * S * S;
  float* out = p.dqkv + ((int64_t)b * S + r0) * ld + h * FA_D;
  // FA_TPR threads a row
  auto row_deltas = [&](int first, int count) {
#pragma unroll 2
    for (int r = threadIdx.x / FA_TPR; r < count; r += FA_QT) {
      float v = 0.f;
      if (first + r < S) {
#pragma unroll
        for (int e = 0; e < FA_D / 4 / FA_TPR; e++) {
          const int64_t at = (first + r) * H + (threadIdx.x % FA_TPR) * (FA_D / FA_TPR) + e * 4;
          const float4 u = *reinterpret_cast<const float4*>(C + at), w = *reinterpret_cast<const float4*>(dC + at);
          v += u.x * w.x + u.y * w.y + u.z * w.z + u.w * w.w;
        }
      }
#pragma unroll
      for (int o = 1; o < FA_TPR; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (threadIdx.x % FA_TPR == 0) delta[r] = v;
    }
  };
  float2 o[FA_RPT][2];
  fa_zero(o);
  if (!keys) {
    // dQ of 32 queries: V blocks form dP, K blocks take dS
    const int n = (len + FA_KC - 1) / FA_KC;
    auto issue = [&](int t) {
      if (t < 2 * n) {
        const int k0 = (t < n ? t : t - n) * FA_KC;
        fa_load<FA_KC>(buf + (t & 1) * FA_KC * FA_PITCH, base + (t < n ? 2 * H : H) + k0 * ld, S - k0, ld);
      }
      fa_commit();
    };
    fa_load<FA_QT>(tile, dC + r0 * H, S - r0, H);
    issue(0);
    issue(1);
    row_deltas(r0, FA_QT);
    for (int t = 0; t < n; t++) {
      fa_wait();
      __syncthreads();
      float pr[FA_RPT][4], s[FA_RPT][4];
#pragma unroll
      for (int i = 0; i < FA_RPT; i++)
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const int j = t * FA_KC + tx + 16 * c;
          pr[i][c] = j < S && r0 + FA_RPT * ty + i < S ? P[(int64_t)(r0 + FA_RPT * ty + i) * S + j] : 0.f;
        }
      fa_scores(tile, buf + (t & 1) * FA_KC * FA_PITCH, ty, tx, s);
#pragma unroll
      for (int i = 0; i < FA_RPT; i++)
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const int j = t * FA_KC + tx + 16 * c;
          if (j < S) sc[(FA_RPT * ty + i) * pitch + j] = pr[i][c] * (s[i][c] - delta[FA_RPT * ty + i]) * p.scale;
        }
      __syncthreads();
      issue(t + 2);
    }
    for (int t = n; t < 2 * n; t++) {
      fa_wait();
      __syncthreads();
      const int j0 = (t - n) * FA_KC;
      fa_values(sc + j0, pitch, buf + (t & 1) * FA_KC * FA_PITCH, min(FA_KC, S - j0), ty, tx, o);
      __syncthreads();
      issue(t + 2);
    }
    fa_store(out, ld, S - r0, ty, tx, o);
    return;
  }
  // dK and dV of 32 keys
  if (r0 >= len) {  // no query attends to them
    fa_store(out + H, ld, S - r0, ty, tx, o);
    fa_store(out + 2 * H, ld, S - r0, ty, tx, o);
    return;
  }
  const int n = (S + FA_KC - 1) / FA_KC;  // dC blocks, then Q blocks
  auto issue = [&](int t) {
    if (t < 2 * n) {
      const int i0 = (t < n ? t : t - n) * FA_KC;
      fa_load<FA_KC>(buf + (t & 1) * FA_KC * FA_PITCH, t < n ? dC + i0 * H : base + i0 * ld, S - i0, t < n ? H : ld);
    }
    fa_commit();
  };
  fa_load<FA_QT>(tile, base + 2 * H + r0 * ld, S - r0, ld);
  issue(0);
  issue(1);
  // P^T of the block's keys: four queries at a time, so that it can be stored 16 bytes wide
#pragma unroll 4
  for (int i = warp * 4; i < S; i += FA_NT / 8) {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; e++) v[e] = r0 + lane < S ? P[(int64_t)(i + e) * S + r0 + lane] : 0.f;
    *reinterpret_cast<float4*>(sc + lane * pitch + i) = make_float4(v[0], v[1], v[2], v[3]);
  }
  row_deltas(0, (S + 31) & ~31);
  for (int t = 0; t < n; t++) {
    fa_wait();
    __syncthreads();
    const int i0 = t * FA_KC;
    const float* dc = buf + (t & 1) * FA_KC * FA_PITCH;
    fa_values(sc + i0, pitch, dc, min(FA_KC, S - i0), ty, tx, o);
    float s[FA_RPT][4];
    fa_scores(tile, dc, ty, tx, s);
    __syncthreads();  // P^T of these queries has been used: dS^T takes its place
#pragma unroll
    for (int i = 0; i < FA_RPT; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const int q = i0 + tx + 16 * c;
        if (q < S) {
          float* at = sc + (FA_RPT * ty + i) * pitch + q;
          *at = *at * (s[i][c] - delta[q]) * p.scale;
        }
      }
    issue(t + 2);
  }
  fa_store(out + 2 * H, ld, S - r0, ty, tx, o);
  fa_zero(o);
  for (int t = n; t < 2 * n; t++) {
    fa_wait();
    __syncthreads();
    const int i0 = (t - n) * FA_KC;
    fa_values(sc + i0, pitch, buf + (t & 1) * FA_KC * FA_PITCH, min(FA_KC, S - i0), ty, tx, o);
    __syncthreads();
    issue(t + 2);
  }
  fa_store(out + H, ld, S - r0, ty, tx, o);
}

size_t fa_smem_bytes(int S) {
  return sizeof(float) * (size_t)(FA_QT * FA_PITCH + 2 * FA_KC * FA_PITCH + FA_QT * (S + 4) + ((S + 31) & ~31));
}

// both kernels take more shared memory than a launch gets by default: opt in once per device
int fa_opt_in(char* err) {
  static std::mutex mu;
  static bool done[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    snprintf(err, 256, "attention: no CUDA device");
    return MSLT_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return 0;
  const int bytes = (int)fa_smem_bytes(128);
  cudaError_t e = cudaFuncSetAttribute(attn_f32_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_f32_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) {
    snprintf(err, 256, "attention: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    return MSLT_ERR_CUDA;
  }
  done[dev] = true;
  return 0;
}

int fa_launch(bool backward, const AttnF32Params& p, int B, cudaStream_t st, char* err) {
  if (p.S < 8 || p.S > 128 || p.S % 8 || B < 1 || p.A < 1) {
    snprintf(err, 256, "attention: the fp32 kernels need S a multiple of 8 in [8, 128]");
    return MSLT_ERR_ARG;
  }
  int rc = fa_opt_in(err);
  if (rc) return rc;
  const int blocks = p.tiles * B * p.A;
  cudaError_t e = backward ? launch_pdl(attn_f32_bwd_kernel, 2 * blocks, FA_NT, fa_smem_bytes(p.S), st, p)
                           : launch_pdl(attn_f32_fwd_kernel, blocks, FA_NT, fa_smem_bytes(p.S), st, p);
  if (e != cudaSuccess) {
    snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e));
    return MSLT_ERR_CUDA;
  }
  return 0;
}
}  // namespace

int attn_f32_fwd_launch(const float* qkv, float* probs, float* ctx, const int* seq_lens, int B, int S, int A, float scale,
                        cudaStream_t st, char* err) {
  AttnF32Params p = {};
  p.qkv = qkv; p.P_out = probs; p.C_out = ctx; p.seq_lens = seq_lens;
  p.S = S; p.A = A; p.scale = scale; p.tiles = (S + FA_QT - 1) / FA_QT;
  return fa_launch(false, p, B, st, err);
}

int attn_f32_bwd_launch(const float* qkv, const float* probs, const float* ctx, const float* dctx, float* dqkv,
                        const int* seq_lens, int B, int S, int A, float scale, cudaStream_t st, char* err) {
  AttnF32Params p = {};
  p.qkv = qkv; p.P = probs; p.C = ctx; p.dC = dctx; p.dqkv = dqkv; p.seq_lens = seq_lens;
  p.S = S; p.A = A; p.scale = scale; p.tiles = (S + FA_QT - 1) / FA_QT;
  return fa_launch(true, p, B, st, err);
}

}  // namespace mslt
