// fp32 contraction on the tensor cores.  An fp32 operand value is the exact sum of three bf16 values
// (8 + 8 + 8 bits of its 24; the decomposition of Henry, Tang and Heinecke, "Leveraging the bfloat16 artificial
// intelligence datatype for higher-precision computations", 2019), so a product a * b is a sum of nine bf16
// products, each exact in fp32; the three smallest (below 2^-25 of the product) are left out and six remain:
//   a1 b1 + (a1 b2 + a2 b1) + (a1 b3 + a2 b2 + a3 b1).
// Range: the sum is exact from 2^-110 up; of a smaller value the parts below the bf16 range (2^-133) are lost, an
// error of at most 2^-134 per value.  Infinities, and values from 2^62 on, whose plane products could overflow with
// either sign, have no such sum (inf * 0 and inf - inf are NaN): the split reports them, and tiles are then formed
// again by ordinary fp32 multiply-adds of the operands themselves.  NaNs pass through the first plane.
// The tensor core adds with truncation, which would build up over a long k (relative error 3e-6 at k =
// 3072 and 3.5e-5 at 30528 measured, against 1.5e-7 and 6e-7 for a chain of fp32 multiply-adds).  So a
// tensor-memory accumulator only ever holds 64 of k, smallest terms first, and is then added to the
// running sum in registers with ordinary rounded fp32 additions: errors are those of an fp32 sum of
// K / 64 terms or less, at every size.
//
// Bound by shared memory: per 64 of k a CTA takes in three planes of each operand once and the tensor
// core reads each plane pair again, 24 instructions of 128 x BN x 16.  One CTA per tile of 128 x BN:
//   warp 0 / warp 2: TMA producers of the A and B planes, ring of rounds (64 of k)
//   warp 1         : issues the products of a round into one of two accumulators
//   warps 4-11     : add finished accumulators to registers (two warps per TMEM lane quarter)
// Few tiles: the blocks of a cluster share k and add their tiles through distributed shared memory.
#include <mutex>

#include "f32_common.cuh"
#include "tc_common.cuh"

namespace mslt {
namespace {

constexpr int X3_THREADS = 384;
constexpr int X3_STAGES = 2;

struct X3Params {
  F32Params f;
  const int* wide;  // device: not 0 when an operand split in this call held a value the planes cannot stand for
  int a_mn, b_mn, kb_total;
  int a_perm[2], b_perm[2];  // slots of the strided matrix index and of the plane
  uint32_t idesc;
  long long wait_limit;
  int* status;
};

// The block's partial tile by fp32 multiply-adds over k0 .. k1, 32 of k through shared memory at a time.  Called by
// all threads; not on the way of ordinary values, so kept out of the kernel's registers.
template <int BN>
__device__ __noinline__ void plain_tile(const X3Params& p, float* tile, int m0, int n0, int k0, int k1) {
  constexpr int KC = 32, CP = KC + 1, RN = BN / 16, PITCH = BN + 4;
  const mslt_gemm_desc& d = p.f.d;
  const float *A = (const float*)d.A, *B = (const float*)d.B;
  float *as = tile, *bs = tile + BM * CP;
  const int t = (int)threadIdx.x - (X3_THREADS - 256), ty = t >> 4, tx = t & 15;  // 16 x 16 threads of 8 x RN outputs
  float acc[8][RN];
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int j = 0; j < RN; j++) acc[i][j] = 0.f;
  for (int kc = k0; kc < k1; kc += KC) {
    for (int i = threadIdx.x; i < (BM + BN) * KC; i += X3_THREADS) {
      const int r = i / KC, k = kc + i % KC;
      const bool isa = r < BM;
      const int row = isa ? m0 + r : n0 + r - BM;
      float v = 0.f;
      if (k < k1 && row < (isa ? d.M : d.N)) v = isa ? A[row * d.a_rs + k * d.a_ks] : B[row * d.b_rs + k * d.b_ks];
      as[r * CP + i % KC] = v;  // bs follows as
    }
    __syncthreads();
    if (t >= 0)
      for (int k = 0; k < KC; k++) {
        float a[8], b[RN];
#pragma unroll
        for (int i = 0; i < 8; i++) a[i] = as[(ty + 16 * i) * CP + k];
#pragma unroll
        for (int j = 0; j < RN; j++) b[j] = bs[(tx + 16 * j) * CP + k];
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
          for (int j = 0; j < RN; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
    __syncthreads();
  }
  if (t >= 0)
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < RN; j++) tile[(ty + 16 * i) * PITCH + tx + 16 * j] = acc[i][j];
}

template <int BN>
__global__ void __launch_bounds__(X3_THREADS, 1)
gemm_f32x3_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ X3Params p) {
  constexpr int A_PLANE = BM * BK * 2, B_PLANE = BN * BK * 2;
  constexpr int STAGE = 3 * (A_PLANE + B_PLANE), PITCH = BN + 4;
  static_assert(BM * PITCH * 4 <= X3_STAGES * STAGE, "the finished tile reuses the ring");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + X3_STAGES * STAGE);
  uint64_t* full_bar = bars;                      // [X3_STAGES]
  uint64_t* empty_bar = bars + X3_STAGES;         // [X3_STAGES]
  uint64_t* accfull_bar = bars + 2 * X3_STAGES;   // [2]
  uint64_t* accfree_bar = accfull_bar + 2;        // [2]
  uint32_t* tmem_slot = (uint32_t*)(accfull_bar + 4);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmA);
    prefetch_map(&tmB);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < X3_STAGES; s++) {
      mbar_init(smem_u32(&full_bar[s]), 2);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; a++) {
      mbar_init(smem_u32(&accfull_bar[a]), 1);
      mbar_init(smem_u32(&accfree_bar[a]), NUM_EPI_WARPS);
    }
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(2 * BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  const int wide = *reinterpret_cast<const volatile int*>(p.wide);  // looked at when the tile is finished
  const int rank = blockIdx.x % p.f.splits, nt = blockIdx.x / p.f.splits;
  const int m0 = blockIdx.y * BM, n0 = nt * BN;
  const int kb0 = min(p.kb_total, rank * p.f.kb_per_split), kb1 = min(p.kb_total, kb0 + p.f.kb_per_split);
  float acc[BN / 2];

  if ((warp == 0 || warp == 2) && elect_one()) {
    // ------------------------------- TMA producers -------------------------------
    const bool isa = warp == 0;
    const CUtensorMap* map = isa ? &tmA : &tmB;
    const int mn = isa ? p.a_mn : p.b_mn, rows = isa ? BM : BN, row0 = isa ? m0 : n0;
    const int* perm = isa ? p.a_perm : p.b_perm;
    const int plane_bytes = isa ? A_PLANE : B_PLANE;
    const uint32_t base = smem_u32(smem) + (isa ? 0 : 3 * A_PLANE);
    bool ok = true;
    int it = 0;
    for (int kb = kb0; kb < kb1; kb++, it++) {
      const uint32_t s = it % X3_STAGES, ph = (it / X3_STAGES) & 1;
      if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1, abort_flag, p.status)) { ok = false; break; }
      const uint32_t fb = smem_u32(&full_bar[s]);
      mbar_expect_tx(fb, 3 * plane_bytes);
      for (int pl = 0; pl < 3; pl++)
        for (int h = 0; h < (mn ? rows / 64 : 1); h++) {
          int c[4] = {0, 0, 0, 0};
          if (mn) { c[0] = row0 + h * 64; c[perm[0]] = kb * BK; }
          else { c[0] = kb * BK; c[perm[0]] = row0; }
          c[perm[1]] = pl;
          tma_load_4d(base + s * STAGE + pl * plane_bytes + h * (64 * BK * 2), map, fb, c[0], c[1], c[2], c[3]);
        }
    }
    if (!ok || *abort_flag) {  // give the copies in flight time to land before the CTA leaves
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 4000000ll) {}
    }
  } else if (warp == 1 && elect_one()) {
    // ------------------------------- MMA issuer -------------------------------
    const uint64_t a0 = make_smem_desc(smem_u32(smem), p.a_mn ? 64 * BK * 2 : 16);
    const uint64_t b0 = make_smem_desc(smem_u32(smem) + 3 * A_PLANE, p.b_mn ? 64 * BK * 2 : 16);
    const uint32_t a_ks = (p.a_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4, b_ks = (p.b_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4;
    const uint32_t a_hi = (uint32_t)(a0 >> 32), b_hi = (uint32_t)(b0 >> 32), a_lo0 = (uint32_t)a0, b_lo0 = (uint32_t)b0;
    bool ok = true;
    int it = 0;
    for (int kb = kb0; kb < kb1; kb++, it++) {
      const uint32_t s = it % X3_STAGES, ph = (it / X3_STAGES) & 1, b = it & 1, use = it >> 1;
      if (!mbar_wait(smem_u32(&accfree_bar[b]), (use & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      if (!mbar_wait(smem_u32(&full_bar[s]), ph, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      const uint32_t a_lo = a_lo0 + s * (STAGE >> 4), b_lo = b_lo0 + s * (STAGE >> 4);
      // smallest terms first, so that the truncation of early additions is relative to small sums
      constexpr int pa[6] = {2, 1, 0, 1, 0, 0}, pb[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
      for (int t = 0; t < 6; t++)
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; k++) {
          const uint64_t ad = ((uint64_t)a_hi << 32) | (a_lo + pa[t] * (A_PLANE >> 4) + k * a_ks);
          const uint64_t bd = ((uint64_t)b_hi << 32) | (b_lo + pb[t] * (B_PLANE >> 4) + k * b_ks);
          tc_mma(tmem_base + b * BN, ad, bd, p.idesc, (t | k) ? 1u : 0u);
        }
      tc_commit(smem_u32(&empty_bar[s]));
      tc_commit(smem_u32(&accfull_bar[b]));
    }
    if (!ok || *abort_flag) {  // make sure no MMA is still writing tensor memory before it is freed
      tc_commit(smem_u32(&accfull_bar[0]));
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (warp >= 4) {
    // ------------------------------- accumulation -------------------------------
    const int q = warp & 3, half = (warp - 4) >> 2;
    const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + half * (BN / 2);
#pragma unroll
    for (int i = 0; i < BN / 2; i++) acc[i] = 0.f;
    int it = 0;
    for (int kb = kb0; kb < kb1; kb++, it++) {
      const uint32_t b = it & 1, use = it >> 1;
      if (!mbar_wait(smem_u32(&accfull_bar[b]), use & 1, abort_flag, p.status)) break;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < BN / 64; c++) {
        float2 v[16];
        tc_ld32(trow + b * BN + c * 32, v);
#pragma unroll
        for (int j = 0; j < 16; j++) {
          const float2 t = __fadd2_rn(make_float2(acc[c * 32 + 2 * j], acc[c * 32 + 2 * j + 1]), v[j]);
          acc[c * 32 + 2 * j] = t.x;
          acc[c * 32 + 2 * j + 1] = t.y;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&accfree_bar[b]));
    }
  }
  // every round has been multiplied (the accumulating warps saw its accumulator), so the ring is free
  tc_fence_before();
  __syncthreads();
  float* tile = reinterpret_cast<float*>(smem);
  if (wide) {
    plain_tile<BN>(p, tile, m0, n0, kb0 * BK, min(p.f.d.K, kb1 * BK));
  } else if (warp >= 4) {
    const int r = (warp & 3) * 32 + lane, c0 = ((warp - 4) >> 2) * (BN / 2);
#pragma unroll
    for (int i = 0; i < BN / 2; i += 4)
      *reinterpret_cast<float4*>(tile + r * PITCH + c0 + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * BN) : "memory");
  }
  cluster_add_and_finish<BM, BN, X3_THREADS, PITCH>(p.f, rank, tile, 0, m0, n0, Extra4{});
}

// x = p1 + p2 + p3 exactly (bf16 each, rounded to nearest); n a multiple of 8.  *wide is raised for values of 2^62
// and more (see the top of the file).
__global__ void __launch_bounds__(256)
split3_kernel(const float* __restrict__ x, bf16* __restrict__ out, long long n, int* __restrict__ wide) {
  pdl_begin();
  float most = 0.f;
  for (long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * 8; i < n; i += (long long)gridDim.x * 2048) {
    float v[8];
    *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(x + i);
    *reinterpret_cast<float4*>(v + 4) = *reinterpret_cast<const float4*>(x + i + 4);
    __align__(16) bf16 o[3][8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      const bf16 h = __float2bfloat16_rn(v[e]);
      most = fmaxf(most, fabsf(v[e]));  // passes over NaN
      const float r1 = v[e] - __bfloat162float(h);
      const bf16 m = __float2bfloat16_rn(r1);
      o[0][e] = h;
      o[1][e] = m;
      o[2][e] = __float2bfloat16_rn(r1 - __bfloat162float(m));
    }
#pragma unroll
    for (int pl = 0; pl < 3; pl++) *reinterpret_cast<uint4*>(out + pl * n + i) = *reinterpret_cast<const uint4*>(o[pl]);
  }
  if (most >= 4.611686018427387904e18f) atomicOr(wide, 1);
}

constexpr int kMaxDevices = 64;
struct { int sms = 0; } g_dev[kMaxDevices];
std::mutex g_dev_mu;

size_t x3_smem(int bn) { return (size_t)X3_STAGES * 3 * (BM + bn) * BK * 2 + 1024 + 256; }

}  // namespace

void launch_split3(const float* x, void* planes, long long n, int* wide, cudaStream_t st) {
  const long long blocks = (n / 8 + 255) / 256;
  launch_pdl(split3_kernel, (unsigned)(blocks < 148 * 8 ? blocks : 148 * 8), 256, 0, st, x, (bf16*)planes, n, wide);
}

bool gemm_f32x3_accepts(const mslt_gemm_desc& d) {
  if (d.dtype != 0 || d.batch != 1 || d.act == 3 || (d.a_rs != 1 && d.a_ks != 1) || (d.b_rs != 1 && d.b_ks != 1)) return false;
  const long long a_ld = d.a_ks == 1 ? d.a_rs : d.a_ks, b_ld = d.b_ks == 1 ? d.b_rs : d.b_ks;
  return a_ld % 8 == 0 && b_ld % 8 == 0 && (((uintptr_t)d.A | (uintptr_t)d.B) & 15) == 0;
}

bool gemm_f32x3_wins(const mslt_gemm_desc& d, int planes_ready) {
  auto dense = [](long long rows, long long K, long long rs, long long ks) { return ks == 1 ? rows * rs : K * ks; };
  if (!gemm_f32x3_accepts(d)) return false;
  const double flops = 2.0 * d.M * d.N * (double)d.K;
  const double split = 1e-3 * 10. * ((planes_ready & 1 ? 0. : dense(d.M, d.K, d.a_rs, d.a_ks)) + (planes_ready & 2 ? 0. : dense(d.N, d.K, d.b_rs, d.b_ks)));
  // microseconds.  One rate stands for each side: measured 20-38 TFLOP/s on the CUDA cores from 0.6 GFLOP on, 60-200
  // here, splitting at 4.5 TB/s.  Both sides (CUDA cores | product here, + split of one operand, + of both):
  // 512 x 384 x 128 5.1 | 6.3 8.1 9.6, 64 x 768 x 768 8.4 | 8.4 9.9 11.7, 128 x 768 x 768 16.7 | 8.4 10.0 11.8,
  // 192 x 768 x 768 17.0 | 8.7 10.3 12.3, 1024 x 2304 x 768 97 | 18.4 21.1 24.2, 160 x 30520 x 768 232 | 85 87 123.
  // The line falls near 0.2 GFLOP; a split that is there already belongs to a product beyond it.
  const int to_split = (planes_ready & 1 ? 0 : 1) + (planes_ready & 2 ? 0 : 1);
  return 5. + flops / 28e6 > 5. + flops / 130e6 + split / 4.5e3 + 1.5 * to_split;
}

int gemm_f32x3_launch(const mslt_gemm_desc& d, const void* planes_a, const void* planes_b, const int* wide, int* status,
                      cudaStream_t st, char* err) {
  int dev = 0, sms;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    snprintf(err, 256, "gemm: no CUDA device");
    return MSLT_ERR_CUDA;
  }
  {
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (g_dev[dev].sms == 0) {
      cudaError_t e = cudaFuncSetAttribute(gemm_f32x3_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x3_smem(64));
      if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_f32x3_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x3_smem(128));
      if (e != cudaSuccess) { snprintf(err, 256, "gemm: cudaFuncSetAttribute: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
      cudaDeviceGetAttribute(&g_dev[dev].sms, cudaDevAttrMultiProcessorCount, dev);
    }
    sms = g_dev[dev].sms;
  }
  X3Params p;
  memset(&p, 0, sizeof(p));
  p.f.d = d;
  p.wide = wide;
  p.a_mn = d.a_rs == 1 && d.a_ks != 1;
  p.b_mn = d.b_rs == 1 && d.b_ks != 1;
  p.kb_total = (d.K + BK - 1) / BK;
  // tile width and k split, by SM cycles: a round of 64 k, start and end of a block
  int bn = 64, splits = 1;
  double best = 1e30;
  for (int w = 64; w <= 128; w += 64)
    for (int s = 1; s <= 8 && (s == 1 || p.kb_total >= 2 * s); s *= 2) {
      const long long tiles = (long long)((d.M + BM - 1) / BM) * ((d.N + w - 1) / w);
      const int units = s >= 4 ? sms * (s == 4 ? 8 : 7) / 9 : sms;  // one block per SM: clusters of 4 and 8 run 132 and 120 at once
      const double n = (double)((tiles * s + units - 1) / units);
      const double c = n * ((p.kb_total + s - 1) / s * (w == 64 ? 1900. : 2500.) + 4000. + w * 20. + (s > 1 ? 4500. + w * 10. * (s > 2) : 0.));
      if (c < best) { best = c; bn = w; splits = s; }
    }
  p.f.splits = splits;
  p.f.kb_per_split = (p.kb_total + splits - 1) / splits;
  p.f.n_tiles = (d.N + bn - 1) / bn;
  g_gemm_form = {4, BM, bn, 1, splits};
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  p.f.vec_out = al16(d.D) && al16(d.aux) && al16(d.residual) && al16(d.bias) && d.ldd % 4 == 0;
  p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)p.a_mn << 15) | ((uint32_t)p.b_mn << 16) |
            ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
  p.wait_limit = WAIT_LIMIT_CYCLES;
  p.status = status;
  MapVal ma, mb;
  const long long na = p.a_mn ? d.K * d.a_ks : d.M * d.a_rs, nb = p.b_mn ? d.K * d.b_ks : d.N * d.b_rs;  // plane strides
  int rc = get_map(planes_a, d.M, d.K, d.a_rs, d.a_ks, 0, na, 3, 1, BM, &ma, err);
  if (!rc) rc = get_map(planes_b, d.N, d.K, d.b_rs, d.b_ks, 0, nb, 3, 1, bn, &mb, err);
  if (rc) return rc;
  for (int i = 0; i < 2; i++) { p.a_perm[i] = ma.perm[i]; p.b_perm[i] = mb.perm[i]; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.f.n_tiles * splits, (d.M + BM - 1) / BM, 1);
  cfg.blockDim = dim3(X3_THREADS);
  cfg.dynamicSmemBytes = x3_smem(bn);
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
  cudaError_t e = bn == 64 ? cudaLaunchKernelEx(&cfg, gemm_f32x3_kernel<64>, ma.map, mb.map, p)
                           : cudaLaunchKernelEx(&cfg, gemm_f32x3_kernel<128>, ma.map, mb.map, p);
  if (e != cudaSuccess) { snprintf(err, 256, "gemm: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  return 0;
}

}  // namespace mslt
