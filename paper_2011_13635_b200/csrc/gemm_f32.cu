// fp32 contraction on the CUDA cores:  D[z][m][n] = epilogue(alpha * sum_k A[z](m,k) * B[z](n,k)).
// TF32 tensor cores are not used: the fp32 path is held to 1e-4 and every product stays a full
// fp32 multiply-add.  What runs here: the products of small configurations, the attention products, and any
// operands that the split form does not take.  Measured (back-to-back launches): a product of the smallest
// configuration (512 x 128 x 512) 20 us in the 64 x 64 kernel with unpipelined loads that this one replaces, then 6,
// and with four groups of warps sharing the k of a 32 x 32 tile 3.1 to 6.0; 128 x 768 x 768 16.7, 1024 x 2304 x 768
// 97 (24 in gemm_f32x3.cu with both splits).  The fp32 pipe is 50-67 % busy at 128 x 128; 16 warps per SM with
// fragments of one k (128 registers), packed multiply-adds along k and slices of 16 were no faster.
//
// Bound by the fp32 pipe (128 lanes per SM) where there is work for every SM, by the serial chain of
// k slices where there is not.  A block owns an output tile (128 x 128, 64 x 64 or 32 x 32) and walks
// k in slices of 32 through a ring of shared-memory stages filled by cp.async, so several slices
// travel while one is multiplied; a thread keeps 8 x 8 (4 x 4) outputs in registers and uses packed
// two-wide multiply-adds, which leave every other issue slot to the shared-memory loads.
// Products with few tiles split k over the blocks of a cluster, which add their partial tiles through
// distributed shared memory in rank order (same bits on every run).
// Either operand may be k-contiguous or row-contiguous; both are copied as they lie:
//   k-contiguous  : [row][32 k], 16-byte units XOR-ed with (row >> 2) & 7
//   row-contiguous: [32 k][row]
// so that the 16-byte fragment loads of eight neighbouring lanes always hit eight bank groups.
#include <stdio.h>

#include <mutex>

#include "f32_common.cuh"

namespace mslt {
namespace {

constexpr int FK = 32;  // k extent of a stage

__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Copies rows [r0, r0 + ROWS) x k slices of 32 of one operand to shared memory; what lies outside is
// zero.  A thread's 16-byte units lie at one column of the contiguous index and STEP apart along the
// other, so a slice costs it one pointer and one bound, not one of each per unit.
template <int ROWS, int NT, bool MN, bool VEC>
struct SliceLoader {
  static constexpr int CH = MN ? ROWS / 4 : FK / 4;  // 16-byte units along the contiguous index
  static constexpr int STEP = NT / CH, UNITS = ROWS * FK / 4 / NT;
  const float *base, *src;
  int64_t pitch;     // elements between two lines of the strided index
  int first, limit;  // this thread's first line and the number of lines (k-contiguous: rows)
  int left;          // valid elements of the contiguous index from this thread's unit on
  uint32_t at;
  __device__ __forceinline__ void init(const float* b, int64_t rs, int64_t ks, int r0, int rows, int k0, int K) {
    const int o = threadIdx.x / CH, c = threadIdx.x % CH;
    base = b;
    pitch = MN ? ks : rs;
    first = (MN ? k0 : r0) + o;
    limit = MN ? K : rows;
    const int col = (MN ? r0 : k0) + 4 * c;
    left = (MN ? rows : K) - col;
    src = b + (int64_t)first * pitch + col;
    at = (MN ? (uint32_t)(o * ROWS + 4 * c) : (uint32_t)(o * FK + 4 * (c ^ ((o >> 2) & 7)))) * 4u;
  }
  __device__ __forceinline__ void load(uint32_t stage) {
    const int n = left < 0 ? 0 : (left > 4 ? 4 : left);
#pragma unroll
    for (int i = 0; i < UNITS; i++) {
      const bool in = first + i * STEP < limit && n > 0;
      const float* s = in ? src + i * STEP * pitch : base;
      // (o >> 2) & 7 differs between a thread's units only where STEP is no multiple of 32
      uint32_t dst = stage + at + (uint32_t)i * STEP * (MN ? ROWS : FK) * 4u;
      if (!MN && STEP % 32 != 0) {
        const int o = threadIdx.x / CH + i * STEP, c = threadIdx.x % CH;
        dst = stage + (uint32_t)(o * FK + 4 * (c ^ ((o >> 2) & 7))) * 4u;
      }
      if (VEC) {
        cp_async16(dst, s, in ? 4 * n : 0);
      } else {
#pragma unroll
        for (int e = 0; e < 4; e++) cp_async4(dst + 4 * e, in && e < n ? s + e : base, in && e < n ? 4 : 0);
      }
    }
    if (MN) { first += FK; src += FK * pitch; } else { left -= FK; src += FK; }
  }
};

__device__ __forceinline__ float pick(const float4& v, int e) { return e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w)); }

// TM x TN outputs per thread; a warp is 4 (rows) x 8 (columns) threads, a tile WM x WN warps.  KG groups
// of such warps share the k of every slice and add their tiles at the end: a small tile alone on an SM
// is bound by the chain of multiply-adds of its few warps (32 x 32 with KG = 1: 34 cycles per k).
template <int TM, int TN, int WM, int WN, int KG, int STAGES, bool AMN, bool BMN, bool VEC>
__global__ void __launch_bounds__(WM * WN * KG * 32)
gemm_f32_kernel(const F32Params p) {
  constexpr int NT = WM * WN * KG * 32, BMT = WM * 4 * TM, BNT = WN * 8 * TN;
  constexpr int STAGE = (BMT + BNT) * FK;  // floats
  static_assert(KG * BMT * BNT <= STAGE * STAGES, "the partial tile reuses the ring");
  extern __shared__ __align__(128) float f32_ring[];
  const mslt_gemm_desc& d = p.d;
  const int rank = blockIdx.x % p.splits, nt = blockIdx.x / p.splits;
  const int z = blockIdx.z, zo = z / d.hdiv, zi = z - zo * d.hdiv;
  const float* A = (const float*)d.A + zo * d.a_bo + zi * d.a_bi;
  const float* B = (const float*)d.B + zo * d.b_bo + zi * d.b_bi;
  const int64_t zoff = zo * d.d_bo + zi * d.d_bi;
  const int m0 = blockIdx.y * BMT, n0 = nt * BNT;
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % (WM * WN), kg = (threadIdx.x >> 5) / (WM * WN);
  const int lr = lane >> 3, lc = lane & 7;
  const int row_t = (warp / WN) * 4 * TM + lr * 4, col_t = (warp % WN) * 8 * TN + lc * 4;
  const int kb_total = (d.K + FK - 1) / FK;
  const int kb0 = rank * p.kb_per_split, kb1 = min(kb_total, kb0 + p.kb_per_split);
  const uint32_t ring = f32_smem(f32_ring);

  SliceLoader<BMT, NT, AMN, VEC> la;
  SliceLoader<BNT, NT, BMN, VEC> lb;
  la.init(A, d.a_rs, d.a_ks, m0, d.M, kb0 * FK, d.K);
  lb.init(B, d.b_rs, d.b_ks, n0, d.N, kb0 * FK, d.K);
  // Weights are asked for ahead of the wait for the preceding kernel; they join the first slices' groups.
  if (p.early) {
#pragma unroll
    for (int s = 0; s < STAGES - 1; s++)
      if (kb0 + s < kb1) lb.load(ring + (uint32_t)s * STAGE * 4u + BMT * FK * 4u);
  }
  pdl_begin();
  auto issue = [&](int kb) {  // called once for every kb, in order
    if (kb < kb1) {
      const uint32_t st = ring + (uint32_t)((kb - kb0) % STAGES) * STAGE * 4u;
      la.load(st);
      if (!p.early || kb - kb0 >= STAGES - 1) lb.load(st + BMT * FK * 4u);
    }
    cp_commit();  // an empty group keeps the count of groups in step
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; s++) issue(kb0 + s);

  Extra4 mine = {};
  if (KG > 1) {
    int r, c;
    const int share = BMT / p.splits;
    first_piece<BNT>(p, rank, share, &r, &c);
    if ((int)threadIdx.x < share * (BNT / 4)) mine = load_extra4(p, zoff, m0 + r, n0 + c);
  }
  float2 acc[TM][TN / 2];  // pairs of neighbouring columns
#pragma unroll
  for (int i = 0; i < TM; i++)
#pragma unroll
    for (int j = 0; j < TN / 2; j++) acc[i][j] = make_float2(0.f, 0.f);

  for (int kb = kb0; kb < kb1; kb++) {
    cp_wait<STAGES - 2>();
    __syncthreads();          // slice kb is here, and everyone is done with the stage filled next
    issue(kb + STAGES - 1);
    const float* as = f32_ring + (size_t)((kb - kb0) % STAGES) * STAGE;
    const float* bs = as + BMT * FK;
    auto row_of = [&](int i) { return row_t + (i >> 2) * 16 + (i & 3); };
    auto col_of = [&](int j) { return col_t + (j >> 2) * 32 + (j & 3); };
    auto kfrag = [&](const float* t, int r, int q) {
      return *reinterpret_cast<const float4*>(t + r * FK + 4 * (q ^ ((r >> 2) & 7)));
    };
#pragma unroll
    for (int qi = 0; qi < FK / 4 / KG; qi++) {
      const int q = kg * (FK / 4 / KG) + qi;
      // fragments of four k: a k-contiguous operand gives four k of one row per 16 bytes, a
      // row-contiguous one four rows of one k
      float4 a[TM], b[TN];
      if (!AMN) {
#pragma unroll
        for (int i = 0; i < TM; i++) a[i] = kfrag(as, row_of(i), q);
      }
      if (!BMN) {
#pragma unroll
        for (int j = 0; j < TN; j++) b[j] = kfrag(bs, col_of(j), q);
      }
#pragma unroll
      for (int kk = 0; kk < 4; kk++) {
        if (AMN) {
#pragma unroll
          for (int h = 0; h < TM / 4; h++) a[h] = *reinterpret_cast<const float4*>(as + (4 * q + kk) * BMT + row_of(4 * h));
        }
        if (BMN) {
#pragma unroll
          for (int h = 0; h < TN / 4; h++) b[h] = *reinterpret_cast<const float4*>(bs + (4 * q + kk) * BNT + col_of(4 * h));
        }
#pragma unroll
        for (int i = 0; i < TM; i++)
#pragma unroll
          for (int j = 0; j < TN / 2; j++) {
            const float x = AMN ? pick(a[i >> 2], i & 3) : pick(a[i], kk);
            if (BMN) {  // the pair of columns lies side by side: one packed instruction
              const float4& t = b[j >> 1];
              acc[i][j] = __ffma2_rn(make_float2(x, x), j & 1 ? make_float2(t.z, t.w) : make_float2(t.x, t.y), acc[i][j]);
            } else {
              acc[i][j].x = fmaf(x, pick(b[2 * j], kk), acc[i][j].x);
              acc[i][j].y = fmaf(x, pick(b[2 * j + 1], kk), acc[i][j].y);
            }
          }
      }
    }
  }
  auto out4 = [&](int i, int h) { return make_float4(acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x, acc[i][2 * h + 1].y); };
  cp_wait<0>();
  if (KG == 1 && p.splits == 1) {
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
      for (int h = 0; h < TN / 4; h++)
        epilogue4<false>(p, zoff, m0 + row_t + (i >> 2) * 16 + (i & 3), n0 + col_t + h * 32, out4(i, h), mine);
    return;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; i++)
#pragma unroll
    for (int h = 0; h < TN / 4; h++)
      *reinterpret_cast<float4*>(f32_ring + kg * BMT * BNT + (row_t + (i >> 2) * 16 + (i & 3)) * BNT + col_t + h * 32) = out4(i, h);
  cluster_add_and_finish<BMT, BNT, NT, BNT, KG>(p, rank, f32_ring, zoff, m0, n0, mine);
}

typedef void (*F32Fn)(const F32Params);
// [tile][A row-contiguous][B row-contiguous][16-byte copies]
#define F32_SET(...)                                                                           \
  {{{gemm_f32_kernel<__VA_ARGS__, false, false, false>, gemm_f32_kernel<__VA_ARGS__, false, false, true>},   \
    {gemm_f32_kernel<__VA_ARGS__, false, true, false>, gemm_f32_kernel<__VA_ARGS__, false, true, true>}},    \
   {{gemm_f32_kernel<__VA_ARGS__, true, false, false>, gemm_f32_kernel<__VA_ARGS__, true, false, true>},     \
    {gemm_f32_kernel<__VA_ARGS__, true, true, false>, gemm_f32_kernel<__VA_ARGS__, true, true, true>}}}
// 128 x 128, 64 x 64, 32 x 32 with shared k (few tiles), 32 x 32 (many, in batches)
const F32Fn kF32[4][2][2][2] = {F32_SET(8, 8, 4, 2, 1, 3), F32_SET(8, 8, 2, 1, 1, 3), F32_SET(4, 4, 2, 1, 4, 6), F32_SET(4, 4, 2, 1, 1, 4)};
#undef F32_SET
constexpr int kTile[4] = {128, 64, 32, 32}, kThreads[4] = {256, 64, 256, 64}, kStages[4] = {3, 3, 6, 4};

constexpr int kMaxDevices = 64;
struct { int sms = 0; } g_dev[kMaxDevices];
std::mutex g_dev_mu;

}  // namespace

int gemm_f32_launch(const mslt_gemm_desc& d, cudaStream_t st, char* err, bool b_static) {
  if (d.act == 3) {
    snprintf(err, 256, "gemm: the softmax epilogue exists only in the tensor-core kernel");
    return MSLT_ERR_ARG;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    snprintf(err, 256, "gemm: no CUDA device");
    return MSLT_ERR_CUDA;
  }
  int sms;
  {
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (g_dev[dev].sms == 0) {
      for (int t = 0; t < 4; t++)
        for (int i = 0; i < 8; i++) {
          cudaError_t e = cudaFuncSetAttribute((const void*)kF32[t][i >> 2][(i >> 1) & 1][i & 1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               2 * kTile[t] * FK * 4 * kStages[t]);
          if (e != cudaSuccess) { snprintf(err, 256, "gemm: cudaFuncSetAttribute: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
        }
      cudaDeviceGetAttribute(&g_dev[dev].sms, cudaDevAttrMultiProcessorCount, dev);
    }
    sms = g_dev[dev].sms;
  }
  F32Params p;
  p.d = d;
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  auto m4 = [](int64_t v) { return v % 4 == 0; };
  p.early = b_static ? 1 : 0;
  p.vec_out = al16(d.D) && al16(d.aux) && al16(d.residual) && al16(d.bias) && m4(d.ldd) &&
              (d.batch == 1 || (m4(d.d_bo) && m4(d.d_bi)));
  // Tile and split: the estimate below (SM cycles) reproduces the measured order of the choices on
  // every product of BERT-Base at 1024 tokens and of the small configurations.  A block alone on an
  // SM takes `alone` cycles per k, n blocks share the fp32 pipe at `share` cycles each: measured 58 %
  // of the pipe for 128 x 128 (k-contiguous B), 67 % (row-contiguous B, packed multiply-adds), 60 %
  // for 64 x 64 (row-contiguous B only: 45 % otherwise); 32 x 32 is bound by its chain of slices.
  // The epilogue is a chain too: a thread takes its outputs four at a time, and the loads of one four wait for the
  // stores of the last.  With a short k that is most of the time (664 x 1040 x 16 with GELU and its pre-activation
  // 13.6 us in 64 x 64 tiles, 5.3 to 7.1 in 32 x 32; 592 x 1385 x 25 accumulated, rows of odd pitch, 20.8 and 6.8).
  // The blocks of a cluster share out the tile's rows, and their constants have the epilogue in them.  Over 244 timed
  // shapes of all layouts and epilogues the pick is 4.3 % slower than the best form on average and 1.5 times at
  // worst; without the term 10 % and 3.7 times.  (Products with a batch were fitted without it.)
  const bool amn = d.a_rs == 1 && d.a_ks != 1, bmn = d.b_rs == 1 && d.b_ks != 1;
  const int kb_total = (d.K + FK - 1) / FK;
  int t = 0, s = 1;
  double best = 1e30;
  for (int ti = 0; ti < 4; ti++) {
    const long long tiles = (long long)((d.M + kTile[ti] - 1) / kTile[ti]) * ((d.N + kTile[ti] - 1) / kTile[ti]) * d.batch;
    const double share = ti == 0 ? (bmn ? 190. : 220.) : ti == 1 ? (bmn ? 53. : 72.) : ti == 2 ? (bmn ? 16. : 22.) : 16.;
    // products with a batch read short rows of wide matrices: 64 x 64 took 22.8 us on 96 x (128 x 128 x 64)
    // inside a step, 32 x 32 without shared k 11.2
    if (ti == 1 && d.batch > 1) continue;
    if (ti != 0 && (d.M + kTile[ti] - 1) / kTile[ti] > 65535) continue;  // row tiles are the grid's second index
    const double alone = ti == 0 ? share : ti == 1 ? 130. : ti == 2 ? 23. : 34.;
    const int fours = kTile[ti] * kTile[ti] / kThreads[ti] / 4;  // of a thread
    const double per_block = ti == 0 ? 3000. : ti == 1 ? 600. : ti == 2 ? 700. : 150.;
    for (int si = 1; si <= 8 && (si == 1 || kb_total >= si); si *= 2) {
      const double per_split = ti == 0 ? 6000. : ti == 1 ? 1500. : ti == 2 ? 1000. + 400. * si : 2000.;  // exchange of the partial tile
      // one 128 x 128 block fits an SM, so clusters of four and eight leave SMs of a GPC unused: 132 and 120 of
      // 148 blocks run at once (cudaOccupancyMaxActiveClusters)
      const int units = ti == 0 && si >= 4 ? sms * (si == 4 ? 8 : 7) / 9 : sms;
      const double n = (double)((tiles * si + units - 1) / units);
      const double c = (kb_total + si - 1) / si * FK * (n * share > alone ? n * share : alone) + n * (per_block + (si > 1 ? per_split : 0.)) +
                       (si == 1 && d.batch == 1 ? (fours - 1) * (p.vec_out ? 350. : 525.) : 0.) +
                       (ti == 3 ? 3000. : 0.);  // its short rows of threads start and end slowly
      if (c < best) { best = c; t = ti; s = si; }
    }
  }
  p.splits = s;
  p.kb_per_split = (kb_total + s - 1) / s;
  const int tile = kTile[t];
  p.n_tiles = (d.N + tile - 1) / tile;
  g_gemm_form = {3, tile, tile, t == 2 ? 4 : 1, s};
  const bool vec = al16(d.A) && al16(d.B) && m4(amn ? d.a_ks : d.a_rs) && m4(bmn ? d.b_ks : d.b_rs) &&
                   (d.batch == 1 || (m4(d.a_bo) && m4(d.a_bi) && m4(d.b_bo) && m4(d.b_bi)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.n_tiles * s, (d.M + tile - 1) / tile, d.batch);
  if (cfg.gridDim.y > 65535 || cfg.gridDim.z > 65535) {
    snprintf(err, 256, "gemm: grid too large for the CUDA-core kernel");
    return MSLT_ERR_SIZE;
  }
  cfg.blockDim = dim3(kThreads[t]);
  cfg.dynamicSmemBytes = (size_t)2 * tile * FK * 4 * kStages[t];
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = s;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = s > 1 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kF32[t][amn][bmn][vec], p);
  if (e != cudaSuccess) { snprintf(err, 256, "gemm: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  return 0;
}

}  // namespace mslt
