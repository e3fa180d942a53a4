// bf16 contraction for outputs of few tiles (a few hundred rows), bound by latency, not by any rate:
// one 128 x 64 tile per block, k shared by the blocks of a cluster, and up to eight 64-deep operand tiles
// of a block in flight at once.
//   warp 0: TMA producer.  The B tiles of a product whose B nobody writes in the two kernels before
//           (weights) are requested before the wait for the preceding kernel.
//   warp 1: issues tcgen05.mma into 64 columns of tensor memory
//   warps 2-5: move the accumulator to shared memory; then all warps add the cluster's partial tiles
//           through distributed shared memory in rank order (same bits on every run) and apply the
//           epilogue, rows dealt out over the blocks.
// Measured against the persistent kernel (back-to-back launches, us): 64 x 768 x 768 6.1 -> 5.1,
// 64 x 2304 x 768 6.2 -> 5.9, 64 x 768 x 3072 13.2 -> 6.6, 200 x 768 x 3072 13.8 -> 9.3,
// 512 x 768 x 3072 14.2 -> 13.3; at 1024 rows the persistent kernel is level or ahead.
#include <algorithm>
#include <mutex>

#include "gemm.h"
#include "tc_common.cuh"

namespace mslt {
namespace {

constexpr int TS_BN = 64, TS_ROUNDS = 8, TS_THREADS = 192, TS_PITCH = TS_BN + 4;
constexpr int TS_STAGE = A_STAGE_BYTES + TS_BN * BK * 2;

struct TcSmallParams {
  mslt_gemm_desc d;
  int splits, kb_total, kb_per_split, a_mn, b_mn, early;
  int a_perm, b_perm;  // slot of the strided matrix index
  const int* rows;     // device row count, or null
  uint32_t idesc;
  long long wait_limit;
  int starve;
  int* status;
};

template <int SPLITS>
__global__ void __launch_bounds__(TS_THREADS)
gemm_tc_small_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const TcSmallParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t full_bar[TS_ROUNDS], empty_bar[TS_ROUNDS], acc_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) int flags[4];  // abort flag, then the wait limit (read by every bounded wait)
  volatile int* abort_flag = (volatile int*)flags + 1;
  const mslt_gemm_desc& d = p.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % SPLITS, nt = blockIdx.x / SPLITS;
  const int m0 = blockIdx.y * BM, n0 = nt * TS_BN;
  const int kb0 = min(p.kb_total, rank * p.kb_per_split), n_kb = min(p.kb_total, kb0 + p.kb_per_split) - kb0;
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmA);
    prefetch_map(&tmB);
  }
  if (threadIdx.x == 0) {
    for (int r = 0; r < TS_ROUNDS; r++) {
      mbar_init(smem_u32(&full_bar[r]), 1);
      mbar_init(smem_u32(&empty_bar[r]), 1);
    }
    mbar_init(smem_u32(&acc_bar), 1);
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TS_BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  bool active = true;
  // the epilogue's share of this block: rows [rank * share, r_end) of the tile, eight columns per thread
  const int rows_here = min(BM, d.M - m0), share = (rows_here + SPLITS - 1) / SPLITS;
  const int r_end = min(rows_here, (rank + 1) * share);
  uint4 x, res;
  float4 b0, b1;
  // its global operands; those of a thread's first piece are requested before the accumulator is waited for
  auto load_extra = [&](int idx) {
    x = res = make_uint4(0, 0, 0, 0);
    b0 = b1 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int r = rank * share + idx / (TS_BN / 8), n = n0 + idx % (TS_BN / 8) * 8;
    if (r >= r_end || n >= d.N) return;
    const int64_t o = (int64_t)(m0 + r) * d.ldd + n;
    if (d.act == 2) x = *reinterpret_cast<const uint4*>((const bf16*)d.aux + o);
    if (d.residual) res = *reinterpret_cast<const uint4*>((const bf16*)d.residual + o);
    if (d.bias) {
      b0 = *reinterpret_cast<const float4*>(d.bias + n);
      b1 = *reinterpret_cast<const float4*>(d.bias + n + 4);
    }
  };

  if (warp == 0) {
    auto load_b = [&](int r) {
      const int slot = r % TS_ROUNDS;
      const uint32_t fb = smem_u32(&full_bar[slot]);
      mbar_expect_more(fb, TS_STAGE - A_STAGE_BYTES);
      int c[4] = {0, 0, 0, 0};
      if (p.b_mn) { c[0] = n0; c[p.b_perm] = (kb0 + r) * BK; } else { c[0] = (kb0 + r) * BK; c[p.b_perm] = n0; }
      tma_load_4d(smem_u32(smem) + slot * TS_STAGE + A_STAGE_BYTES, &tmB, fb, c[0], c[1], c[2], c[3]);
    };
    const bool mine = !p.starve && elect_one();
    const int n_early = p.early ? min(n_kb, TS_ROUNDS) : 0;
    if (mine)
      for (int r = 0; r < n_early; r++) load_b(r);
    pdl_begin();
    if (p.rows) active = m0 < *p.rows;
    if (mine && active) {
      bool ok = true;
      for (int r = 0; r < n_kb; r++) {
        const int slot = r % TS_ROUNDS;
        if (r >= TS_ROUNDS && !mbar_wait(smem_u32(&empty_bar[slot]), (r / TS_ROUNDS - 1) & 1, abort_flag, p.status)) { ok = false; break; }
        if (r >= n_early) load_b(r);
        mbar_expect_tx(smem_u32(&full_bar[slot]), A_STAGE_BYTES);
        for (int h = 0; h < (p.a_mn ? 2 : 1); h++) {
          int c[4] = {0, 0, 0, 0};
          if (p.a_mn) { c[0] = m0 + h * 64; c[p.a_perm] = (kb0 + r) * BK; } else { c[0] = (kb0 + r) * BK; c[p.a_perm] = m0; }
          tma_load_4d(smem_u32(smem) + slot * TS_STAGE + h * (64 * BK * 2), &tmA, smem_u32(&full_bar[slot]), c[0], c[1], c[2], c[3]);
        }
      }
      if (!ok) {  // give the copies in flight time to land before the block leaves
        const long long t0 = now_cycles();
        while (now_cycles() - t0 < 4000000ll) {}
      }
    }
    if (mine && !active)  // beyond the rows that exist: the early tiles land before the block leaves
      for (int r = 0; r < n_early; r++) {
        mbar_arrive(smem_u32(&full_bar[r]));
        if (!mbar_wait(smem_u32(&full_bar[r]), 0, abort_flag, p.status)) break;
      }
    __syncwarp();
    if (active) load_extra(threadIdx.x);
  } else {
    pdl_begin();
    if (p.rows) active = m0 < *p.rows;
    if (active) load_extra(threadIdx.x);
    if (warp == 1 && active && elect_one()) {
      const uint64_t a0 = make_smem_desc(smem_u32(smem), p.a_mn ? 64 * BK * 2 : 16);
      const uint64_t bd0 = make_smem_desc(smem_u32(smem) + A_STAGE_BYTES, p.b_mn ? 64 * BK * 2 : 16);
      const uint32_t a_ks = (p.a_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4, b_ks = (p.b_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      bool ok = true;
      for (int r = 0; r < n_kb; r++) {
        const int slot = r % TS_ROUNDS;
        if (!mbar_wait(smem_u32(&full_bar[slot]), (r / TS_ROUNDS) & 1, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; k++)
          tc_mma(tmem_base, a0 + slot * (TS_STAGE >> 4) + k * a_ks, bd0 + slot * (TS_STAGE >> 4) + k * b_ks, p.idesc, (r | k) ? 1u : 0u);
        if (r + TS_ROUNDS < n_kb) tc_commit(smem_u32(&empty_bar[slot]));
      }
      tc_commit(smem_u32(&acc_bar));
      if (!ok) {  // let issued copies and products end before the block leaves
        const long long t0 = now_cycles();
        while (now_cycles() - t0 < 4000000ll) {}
      }
    }
    if (warp >= 2 && active) {
      const int q = warp & 3;
      float2 v0[16], v1[16];
      const bool ok = mbar_wait(smem_u32(&acc_bar), 0, abort_flag, p.status);
      tc_fence_after();
      if (ok && n_kb > 0) {
        tc_ld32(tmem_base + ((uint32_t)(q * 32) << 16), v0);
        tc_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + 32, v1);
      } else {
#pragma unroll
        for (int j = 0; j < 16; j++) v0[j] = v1[j] = make_float2(0.f, 0.f);
      }
      // every product has read its operands: the tile takes their place
      float* row = reinterpret_cast<float*>(smem) + (q * 32 + lane) * TS_PITCH;
#pragma unroll
      for (int j = 0; j < 8; j++) {
        *reinterpret_cast<float4*>(row + 4 * j) = make_float4(v0[2 * j].x, v0[2 * j].y, v0[2 * j + 1].x, v0[2 * j + 1].y);
        *reinterpret_cast<float4*>(row + 32 + 4 * j) = make_float4(v1[2 * j].x, v1[2 * j].y, v1[2 * j + 1].x, v1[2 * j + 1].y);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TS_BN) : "memory");
  }
  if (!active) return;  // the same for every block of the cluster
  if (SPLITS > 1) cluster_sync_all();
  for (int idx = threadIdx.x; idx < share * (TS_BN / 8); idx += TS_THREADS) {
    const int r = rank * share + idx / (TS_BN / 8), c = idx % (TS_BN / 8) * 8, n = n0 + c;
    if (idx != (int)threadIdx.x) load_extra(idx);
    if (r >= r_end || n >= d.N) continue;
    const int64_t o = (int64_t)(m0 + r) * d.ldd + n;
    float4 t[SPLITS][2];  // every partial result requested before the first is added
    if (SPLITS > 1) {
      const uint32_t at = smem_u32(smem) + (uint32_t)(r * TS_PITCH + c) * 4u;
#pragma unroll
      for (int q = 0; q < SPLITS; q++) {
        const uint32_t far = mapa_u32(at, q);
#pragma unroll
        for (int h = 0; h < 2; h++)
          asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(t[q][h].x), "=f"(t[q][h].y), "=f"(t[q][h].z), "=f"(t[q][h].w) : "r"(far + 16 * h));
      }
    } else {
      const float* l = reinterpret_cast<const float*>(smem) + r * TS_PITCH + c;
      t[0][0] = *reinterpret_cast<const float4*>(l);
      t[0][1] = *reinterpret_cast<const float4*>(l + 4);
    }
    float2 v[4];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      float4 sum = t[0][h];
#pragma unroll
      for (int q = 1; q < SPLITS; q++) { sum.x += t[q][h].x; sum.y += t[q][h].y; sum.z += t[q][h].z; sum.w += t[q][h].w; }
      v[2 * h] = make_float2(sum.x, sum.y);
      v[2 * h + 1] = make_float2(sum.z, sum.w);
    }
    const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
    auto pack = [&](uint4& out) {
      __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
      for (int e = 0; e < 4; e++) h[e] = __float22bfloat162_rn(v[e]);
    };
#pragma unroll
    for (int e = 0; e < 4; e++) v[e] = __ffma2_rn(v[e], splat2(d.alpha), b[e]);
    if (d.act == 1) {
      if (d.aux) {
        uint4 u;
        pack(u);
        *reinterpret_cast<uint4*>((bf16*)d.aux + o) = u;
      }
      gelu_fast2(v);
    } else if (d.act == 2) {
      const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
      float2 g[4] = {bf162_to_f2(xw[0]), bf162_to_f2(xw[1]), bf162_to_f2(xw[2]), bf162_to_f2(xw[3])};
      gelu_grad_fast2(g);
#pragma unroll
      for (int e = 0; e < 4; e++) v[e] = __fmul2_rn(v[e], g[e]);
    }
    if (d.residual) {
      const uint32_t rw[4] = {res.x, res.y, res.z, res.w};
#pragma unroll
      for (int e = 0; e < 4; e++) v[e] = __fadd2_rn(v[e], bf162_to_f2(rw[e]));
    }
    uint4 out;
    pack(out);
    *reinterpret_cast<uint4*>((bf16*)d.D + o) = out;
  }
  if (SPLITS > 1) cluster_sync_exit();  // no block leaves while its tile is read
}

typedef void (*TcSmallFn)(const CUtensorMap, const CUtensorMap, const TcSmallParams);
const TcSmallFn kKernels[4] = {gemm_tc_small_kernel<1>, gemm_tc_small_kernel<2>, gemm_tc_small_kernel<4>, gemm_tc_small_kernel<8>};
constexpr int kMaxDevices = 64;
bool g_attr[kMaxDevices];
std::mutex g_attr_mu;

}  // namespace

// Split count with the least estimated time (microseconds, *t), or 0 where the kernel does not apply.
int gemm_tc_small_plan(const mslt_gemm_desc& d, int num_sms, const Fills& fills, double* t) {
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  if (d.batch != 1 || d.d_fp32 || d.act == 3 || d.N % 8 || d.ldd % 8 || !al16(d.D) || !al16(d.aux) || !al16(d.residual) ||
      !al16(d.bias) || (d.act == 2 && !d.aux))
    return 0;
  const int kb = (d.K + BK - 1) / BK;
  int best = 0;
  for (int s = 1; s <= 8; s *= 2) {
    const int per = (kb + s - 1) / s;
    if (s > 1 && per < 2) continue;
    // blocks that run at once (200 KB of shared memory each; in clusters of 4 and 8 they leave SMs of a GPC unused)
    const int units = s >= 4 ? num_sms * (s == 4 ? 8 : 7) / 9 : num_sms;
    double mean = 0.;
    bool fits = false;
    for (int i = 0; i < fills.n; i++) {
      const int m = Fills::of(d.M, fills.share[i]);
      const long long blocks = (long long)((m + BM - 1) / BM) * ((d.N + TS_BN - 1) / TS_BN) * s;
      const long long waves = (blocks + units - 1) / units;
      fits |= waves <= 1;
      // fitted to the launches named at the top of the file: start and end, rounds, the exchange in the
      // cluster, rows of the epilogue, blocks that share L2
      const double c = 3.4 + 0.23 * per + (s > 1 ? 0.3 + 0.1 * s : 0.) + (m < BM ? m : BM) / 128. + 0.4 * (waves > 1 ? units : blocks) / num_sms;
      mean += c * waves / fills.n;
    }
    // Made for one wave.  Where the rows are known on the device only, some fill has to give one, and every fill counts with
    // the waves it takes: evaluation of 8 x 128 tokens by 9 layers, split of k chosen for 0.7 of the rows alone | so, full
    // 687 | 555 us, 0.7 filled 562 | 531, 0.4 filled 507 | 518.
    if (!fits) continue;
    if (!best || mean < *t) { best = s; *t = mean; }
  }
  return best;
}

int gemm_tc_small_launch(const mslt_gemm_desc& d, int splits, bool early, int* status, cudaStream_t st, char* err,
                         const int* rows, bool starve) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    snprintf(err, 256, "gemm: no CUDA device");
    return MSLT_ERR_CUDA;
  }
  const size_t smem = (size_t)TS_ROUNDS * TS_STAGE + 1024;
  {
    std::lock_guard<std::mutex> lock(g_attr_mu);
    if (!g_attr[dev]) {
      cudaError_t e = cudaSuccess;
      for (const TcSmallFn f : kKernels)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) { snprintf(err, 256, "gemm: cudaFuncSetAttribute: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
      g_attr[dev] = true;
    }
  }
  TcSmallParams p;
  memset(&p, 0, sizeof(p));
  p.d = d;
  p.a_mn = d.a_rs == 1 && d.a_ks != 1;
  p.b_mn = d.b_rs == 1 && d.b_ks != 1;
  p.splits = splits;
  p.kb_total = (d.K + BK - 1) / BK;
  p.kb_per_split = (p.kb_total + splits - 1) / splits;
  p.early = early && !starve ? 1 : 0;
  p.rows = rows;
  p.starve = starve ? 1 : 0;
  p.wait_limit = starve ? 40000000ll : WAIT_LIMIT_CYCLES;
  p.status = status;
  p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)p.a_mn << 15) | ((uint32_t)p.b_mn << 16) |
            ((uint32_t)(TS_BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
  g_gemm_form = {2, BM, TS_BN, 1, splits};
  MapVal ma, mb;
  int rc = get_map(d.A, d.M, d.K, d.a_rs, d.a_ks, 0, 0, 1, 1, BM, &ma, err);
  if (!rc) rc = get_map(d.B, d.N, d.K, d.b_rs, d.b_ks, 0, 0, 1, 1, TS_BN, &mb, err);
  if (rc) return rc;
  p.a_perm = ma.perm[0];
  p.b_perm = mb.perm[0];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((d.N + TS_BN - 1) / TS_BN * splits, (d.M + BM - 1) / BM, 1);
  cfg.blockDim = dim3(TS_THREADS);
  // as much shared memory as the rounds of a block need, and room for its tile
  const size_t need = (size_t)std::min(std::max(p.kb_per_split, 2), TS_ROUNDS) * TS_STAGE + 1024;
  cfg.dynamicSmemBytes = need;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = splits;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = splits > 1 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kKernels[splits == 8 ? 3 : splits >> 1], ma.map, mb.map, p);
  if (e != cudaSuccess) { snprintf(err, 256, "gemm: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  return 0;
}

}  // namespace mslt
