// Shared by the two fp32 contraction kernels (CUDA cores, and tensor cores on split operands): launch
// parameters, the fused epilogue, and the addition of partial tiles inside a cluster.
#pragma once
#include "common.cuh"
#include "gemm.h"

namespace mslt {
namespace {

struct F32Params {
  mslt_gemm_desc d;
  int splits, kb_per_split, n_tiles;
  int early;    // B is not written by the kernels before this one: read ahead of the wait for them
  int vec_out;  // D, aux, residual and bias rows allow 16-byte access
};

__device__ __forceinline__ uint32_t f32_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// What the epilogue reads beside the sums, for four columns of a row.  Where a thread has one piece of a small tile
// (kLoaded) it asks for them ahead of the main loop; asked for at the end they add a trip to L2 to every launch.  Larger
// tiles read them piece by piece (1 % of the split-operand kernel).
struct Extra4 { float4 bias, aux, residual; };
__device__ __forceinline__ Extra4 load_extra4(const F32Params& p, int64_t zoff, int m, int n) {
  const mslt_gemm_desc& d = p.d;
  Extra4 x;
  x.bias = x.aux = x.residual = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!p.vec_out || m >= d.M || n + 4 > d.N) return x;
  const int64_t o = zoff + (int64_t)m * d.ldd + n;
  if (d.bias) x.bias = *reinterpret_cast<const float4*>(d.bias + n);
  if (d.act == 2) x.aux = *reinterpret_cast<const float4*>((const float*)d.aux + o);
  if (d.residual) x.residual = *reinterpret_cast<const float4*>((const float*)d.residual + o);
  return x;
}

template <bool kLoaded>
__device__ __forceinline__ void epilogue4(const F32Params& p, int64_t zoff, int m, int n, float4 v4, const Extra4& x4) {
  const mslt_gemm_desc& d = p.d;
  if (m >= d.M || n >= d.N) return;
  const int64_t o = zoff + (int64_t)m * d.ldd + n;
  float v[4] = {d.alpha * v4.x, d.alpha * v4.y, d.alpha * v4.z, d.alpha * v4.w};
  float* D = (float*)d.D;
  if (p.vec_out && n + 4 <= d.N) {
    if (d.bias) {
      const float4 b = kLoaded ? x4.bias : *reinterpret_cast<const float4*>(d.bias + n);
      v[0] += b.x; v[1] += b.y; v[2] += b.z; v[3] += b.w;
    }
    if (d.act == 1) {
      if (d.aux) *reinterpret_cast<float4*>((float*)d.aux + o) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
      for (int e = 0; e < 4; e++) v[e] = gelu_f(v[e]);
    } else if (d.act == 2) {
      const float4 u = kLoaded ? x4.aux : *reinterpret_cast<const float4*>((const float*)d.aux + o);
      v[0] *= gelu_grad_f(u.x); v[1] *= gelu_grad_f(u.y); v[2] *= gelu_grad_f(u.z); v[3] *= gelu_grad_f(u.w);
    }
    if (d.residual) {
      const float4 r = kLoaded ? x4.residual : *reinterpret_cast<const float4*>((const float*)d.residual + o);
      v[0] += r.x; v[1] += r.y; v[2] += r.z; v[3] += r.w;
    }
    if (d.accumulate)
      asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(D + o), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
    else *reinterpret_cast<float4*>(D + o) = make_float4(v[0], v[1], v[2], v[3]);
    return;
  }
#pragma unroll
  for (int e = 0; e < 4; e++) {
    if (n + e >= d.N) return;
    float x = v[e];
    if (d.bias) x += d.bias[n + e];
    if (d.act == 1) {
      if (d.aux) ((float*)d.aux)[o + e] = x;
      x = gelu_f(x);
    } else if (d.act == 2) {
      x *= gelu_grad_f(((const float*)d.aux)[o + e]);
    }
    if (d.residual) x += ((const float*)d.residual)[o + e];
    if (d.accumulate) atomicAdd(D + o + e, x); else D[o + e] = x;
  }
}

// Partial tiles [BMT][BNT] (rows PITCH floats apart) of the blocks of a cluster are added in rank order;
// each block finishes its share of the rows.  A block may itself hold KG partial tiles, one after the
// other.  Without a split the tile just leaves through the epilogue.  mine: load_extra4 of the thread's first piece (KG > 1).
template <int BNT>
__device__ __forceinline__ void first_piece(const F32Params& p, int rank, int share, int* r, int* c) {
  *r = rank * share + (int)threadIdx.x / (BNT / 4);
  *c = ((int)threadIdx.x % (BNT / 4)) * 4;
}
template <int BMT, int BNT, int NT, int PITCH = BNT, int KG = 1>
__device__ __forceinline__ void cluster_add_and_finish(const F32Params& p, int rank, float* tile, int64_t zoff, int m0, int n0, const Extra4& mine) {
  const uint32_t base = f32_smem(tile);
  if (p.splits == 1) __syncthreads();
  else asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  // Beyond the output nothing is read: a read that no store waits for could be under way at the meeting below.
  // (Tested piece by piece it keeps the reads of neighbouring pieces apart: 1 % of the split-operand kernel.)
  const int share = BMT / p.splits, c = ((int)threadIdx.x % (BNT / 4)) * 4;
  static_assert(NT % (BNT / 4) == 0, "a thread's pieces lie in the same columns");
  const int rows = n0 + c < p.d.N ? min(share, p.d.M - m0 - rank * share) : 0;
  for (int idx = threadIdx.x; idx < rows * (BNT / 4); idx += NT) {
    const int r = rank * share + idx / (BNT / 4);
    const uint32_t at = base + (uint32_t)(r * PITCH + c) * 4u;
    Extra4 x;
    if (KG > 1) x = idx == (int)threadIdx.x ? mine : load_extra4(p, zoff, m0 + r, n0 + c);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.splits == 1) {
#pragma unroll
      for (int g = 0; g < KG; g++) {
        const float4 t = *reinterpret_cast<const float4*>(tile + g * BMT * PITCH + r * PITCH + c);
        s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
      }
    }
    for (int q = 0; q < (p.splits > 1 ? p.splits : 0); q++) {
      uint32_t far;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(far) : "r"(at), "r"(q));
#pragma unroll
      for (int g = 0; g < KG; g++) {
        float4 t;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(far + g * BMT * PITCH * 4) : "memory");
        s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
      }
    }
    epilogue4<(KG > 1)>(p, zoff, m0 + r, n0 + c, s, x);
  }
  // No block leaves while its tile is read.  The meeting orders no memory, so stores on their way do not hold it up;
  // every read of a peer has returned by then, because what is stored was formed from it.
  if (p.splits > 1) asm volatile("barrier.cluster.arrive.relaxed;\n\tbarrier.cluster.wait;" ::: "memory");
}

}  // namespace
}  // namespace mslt
