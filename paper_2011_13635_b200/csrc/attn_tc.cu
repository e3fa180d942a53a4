// Fused attention forward for rows of at most 128 keys and 64-wide heads (sm_100a, bf16):
//   P = softmax(mask(scale * Q K^T)),  C = P V      per (sequence, head),
// in one persistent kernel, so the scores never leave the SM and the probabilities reach HBM only
// when the backward pass needs them.  Unfused, the two products are bound by HBM traffic (about
// 32 flop per byte at head width 64); fused, a layer's attention reads Q, K, V once and writes the
// context once.
//   warp 0   : TMA producer: the Q, K and V tiles of a (sequence, head) item, four items deep.
//   warp 1   : one thread issues tcgen05.mma: S = Q K^T into one of two 128-column accumulators,
//              and, once a softmax group has put P into shared memory, C = P V into one of two
//              64-column accumulators.
//   warps 2-5, 6-9: two softmax groups that take alternate items, so that the exponentials of one
//              item overlap the second product and the stores of the other.  A thread owns one
//              query row: it reads the row's 128 scores from tensor memory, applies scale and
//              mask, forms max, exponentials and sum with no exchange between threads, writes the
//              normalised row as the bf16 A operand of the second product (128-byte swizzle, by
//              hand, over the item's dead Q and K tiles) and, for layers that run backward, to
//              global memory; then reads the context tile back from tensor memory and stores it.
// P is rounded to bf16 before the second product, exactly as when it is stored and read back.
// Every wait is bounded: when one runs out the CTA raises a status bit, drains and returns.
#include <atomic>

#include "gemm.h"
#include "tc_common.cuh"

namespace mslt {

namespace {

constexpr int AT_STAGES = 4;
constexpr int AT_TILE_BYTES = 128 * 64 * 2;          // one of Q, K, V: 16 KB
constexpr int AT_STAGE_BYTES = 3 * AT_TILE_BYTES;    // 48 KB
constexpr int AT_STAGING = 2048;                     // per epilogue warp
constexpr uint32_t AT_TMEM_COLS = 512;
constexpr uint32_t AT_O_COL = 256;                   // two context accumulators after the two score buffers
constexpr int AT_GROUP_WARPS = 4;                    // warps of a softmax group

struct AttnParams {
  int S, heads, items;
  float scale;
  const int* seq_lens;
  const int* cu;      // packed rows: sequence b holds rows cu[b] .. cu[b] + len - 1 of qkv and C; null = b * S
  const int* rows;    // packed: {rows in use, the same rounded up, query tiles}; C's rows between the first two are zeroed
  const int* order;   // packed long rows: 8 * sequence + query tile of every tile that exists, longest sequences first
  float* lse;         // long rows: log2 of the row's sum of exponentials, [A][lse_ld] by row; or null
  long long lse_ld;
  bf16* P;            // [B, A, S, S] or null
  long long p_bo, p_bi;
  bf16* C;            // element (b, i, h, e) at C + b * c_bo + h * c_bi + i * c_ld + e
  long long c_ld, c_bo, c_bi;
  int vec_ok_p, vec_ok_c;
  int fast_p, fast_c;  // rows may be stored directly with 32-byte stores
  int q_perm[3], k_perm[3], v_perm[3];
  long long wait_limit;
  int starve;         // test hook: the producer issues no copies, so the first wait runs out
  int* status;
  uint32_t idesc_s, idesc_o;
};

// A thread that owns a whole row stores 32 of its columns (64 contiguous bytes of bf16) with two
// 32-byte stores: every store fills a full sector, and no trip through shared memory is needed.
// dst must be 32-byte aligned (row_fast says whether a buffer qualifies).
__device__ __forceinline__ void store_row32_bf16(bf16* dst, const float2 (&w)[16]) {
  uint32_t h[16];
#pragma unroll
  for (int e = 0; e < 16; e++) {
    const __nv_bfloat162 t = __float22bfloat162_rn(w[e]);
    h[e] = *reinterpret_cast<const uint32_t*>(&t);
  }
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(h[0]), "r"(h[1]), "r"(h[2]),
               "r"(h[3]), "r"(h[4]), "r"(h[5]), "r"(h[6]), "r"(h[7])
               : "memory");
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 16), "r"(h[8]), "r"(h[9]),
               "r"(h[10]), "r"(h[11]), "r"(h[12]), "r"(h[13]), "r"(h[14]), "r"(h[15])
               : "memory");
}
inline int row_fast(const void* ptr, long long ld_elems) {
  return (((uintptr_t)ptr & 31) == 0 && (ld_elems * 2) % 32 == 0) ? 1 : 0;
}

// Packed batches: the rows between the last sequence and the next tile boundary belong to nobody.
// They are zeroed, because later products read whole tiles.  Called by the threads of warps 2..9.
__device__ __forceinline__ void zero_tail_rows(bf16* base, long long ld, long long width, const int* rows) {
  const int r0 = rows[0], n = rows[1] - r0;
  const long long vecs = width / 8;
  const long long step = (long long)gridDim.x * (NUM_EPI_WARPS * 32);
  for (long long i = (long long)blockIdx.x * (NUM_EPI_WARPS * 32) + threadIdx.x - 64; i < n * vecs; i += step)
    *reinterpret_cast<uint4*>(base + (r0 + i / vecs) * ld + (i % vecs) * 8) = make_uint4(0, 0, 0, 0);
}

// A 128-row tile that starts inside a sequence shorter than the tile goes on into the next sequence's rows, or into
// rows that this call has not written.  Their probabilities are zero, but zero times a NaN or an infinity that lies
// there is NaN, so every such row that is an operand along a contraction is cleared in shared memory first, by warps
// of their own, so that no other role waits for it on a tile without such rows.  These warps see every round of a
// ring (the producer waits for their arrival on the slot's empty barrier too); on a tile with rows to clear
// they also complete the slot's clean barrier, which the thread that issues the products then waits for instead of
// the full barrier.  (Cleared by the softmax warps: evaluation of 12 x (200..384) keys 2.79 -> 2.83 ms.)
// Where every tile has such rows the hand-over shows: training steps on 299 x (16..32) keys, 3 layers, 2449 -> 2507 us.
// In the forward of up to 128 keys the contraction therefore ends with the 16 keys that hold the last one, only those
// are cleared, and lengths are asked for one item early (evaluation of 75 x (16..32) keys 908 us without clearing, 914
// with, 912 so); the same in the backward made no difference (2449 -> 2504 us).
constexpr int CLEAR_WARPS = 2;  // a thread's registers stay the same: four schedulers, three or five warps each
// rows r0 .. r1 of a tile (128 bytes each; the swizzle permutes inside a row), shared out over the clearing warps
__device__ __forceinline__ void clear_tile_rows(uint8_t* tile, int r0, int r1, int idx) {
  for (int v = r0 * 8 + idx; v < r1 * 8; v += 32 * CLEAR_WARPS) reinterpret_cast<uint4*>(tile)[v] = make_uint4(0, 0, 0, 0);
}
// Every thread of a clearing warp: the tile's writes are visible to the tensor core once this has returned.
__device__ __forceinline__ void clear_done(uint32_t clean, int lane) {
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive(clean);
}

// Four 32-column reads of a row in flight together, one wait for all.
__device__ __forceinline__ void tc_ld128(uint32_t taddr, float2 (&v)[4][16]) {
  uint32_t r0[32], r1[32], r2[32], r3[32];
  tc_ld32_issue(taddr, r0);
  tc_ld32_issue(taddr + 32, r1);
  tc_ld32_issue(taddr + 64, r2);
  tc_ld32_issue(taddr + 96, r3);
  tc_ld32_wait(r0);
  tc_ld32_wait(r1);
  tc_ld32_wait(r2);
  tc_ld32_wait(r3);
#pragma unroll
  for (int i = 0; i < 16; i++) {
    v[0][i] = make_float2(__uint_as_float(r0[2 * i]), __uint_as_float(r0[2 * i + 1]));
    v[1][i] = make_float2(__uint_as_float(r1[2 * i]), __uint_as_float(r1[2 * i + 1]));
    v[2][i] = make_float2(__uint_as_float(r2[2 * i]), __uint_as_float(r2[2 * i + 1]));
    v[3][i] = make_float2(__uint_as_float(r3[2 * i]), __uint_as_float(r3[2 * i + 1]));
  }
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <bool kPacked>
__global__ void __launch_bounds__(NUM_THREADS + (kPacked ? 32 * CLEAR_WARPS : 0), 1)
attn_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* staging = smem + AT_STAGES * AT_STAGE_BYTES;
  uint64_t* bars = (uint64_t*)(staging + NUM_EPI_WARPS * AT_STAGING);
  uint64_t* full_bar = bars;                 // [AT_STAGES] tiles of an item have landed
  uint64_t* empty_bar = bars + AT_STAGES;    // [AT_STAGES] both products of an item have read them
  uint64_t* sfull_bar = bars + 2 * AT_STAGES;      // [2] scores complete
  uint64_t* sempty_bar = bars + 2 * AT_STAGES + 2; // [2] scores read by every epilogue warp
  uint64_t* pready_bar = bars + 2 * AT_STAGES + 4; // [2] probabilities of a group's item in shared memory
  uint64_t* ofull_bar = bars + 2 * AT_STAGES + 6;  // [2] context of a group's item complete
  uint64_t* clean_bar = bars + 2 * AT_STAGES + 8;  // [AT_STAGES] packed: V's rows beyond the sequence are zero
  uint32_t* tmem_slot = (uint32_t*)(bars + 3 * AT_STAGES + 8);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < AT_STAGES; s++) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1 + (kPacked ? CLEAR_WARPS : 0));
      mbar_init(smem_u32(&clean_bar[s]), CLEAR_WARPS);
    }
    for (int a = 0; a < 2; a++) {
      mbar_init(smem_u32(&sfull_bar[a]), 1);
      mbar_init(smem_u32(&sempty_bar[a]), AT_GROUP_WARPS);
      mbar_init(smem_u32(&pready_bar[a]), AT_GROUP_WARPS);
      mbar_init(smem_u32(&ofull_bar[a]), 1);
    }
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmQ);
    prefetch_map(&tmK);
    prefetch_map(&tmV);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(AT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  const int n_my = ((int)blockIdx.x < p.items) ? (p.items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  auto item_len = [&](int i) {  // valid keys of this block's item i
    return p.seq_lens ? min(max(p.seq_lens[((int)blockIdx.x + i * (int)gridDim.x) / p.heads], 1), p.S) : p.S;
  };

  if (warp == 0 && !p.starve && elect_one()) {
    // ------------------------------- TMA producer -------------------------------
    bool ok = true;
    int issued = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int zo = w / p.heads, zi = w - zo * p.heads;
      const uint32_t s = (uint32_t)(i % AT_STAGES), round = (uint32_t)(i / AT_STAGES);
      if (!mbar_wait(smem_u32(&empty_bar[s]), (round & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      const uint32_t fb = smem_u32(&full_bar[s]);
      mbar_expect_tx(fb, AT_STAGE_BYTES);
      const uint32_t sq = smem_u32(smem + (size_t)s * AT_STAGE_BYTES);
      const int row0 = kPacked ? p.cu[zo] : 0, zseq = kPacked ? 0 : zo;
      int c[4];
      c[0] = 0; c[p.q_perm[0]] = row0; c[p.q_perm[1]] = zi; c[p.q_perm[2]] = zseq;
      tma_load_4d(sq, &tmQ, fb, c[0], c[1], c[2], c[3]);
      c[0] = 0; c[p.k_perm[0]] = row0; c[p.k_perm[1]] = zi; c[p.k_perm[2]] = zseq;
      tma_load_4d(sq + AT_TILE_BYTES, &tmK, fb, c[0], c[1], c[2], c[3]);
      // V is read with the head dimension contiguous: two boxes of 64 keys
      c[0] = 0; c[p.v_perm[1]] = zi; c[p.v_perm[2]] = zseq;
      c[p.v_perm[0]] = row0;
      tma_load_4d(sq + 2 * AT_TILE_BYTES, &tmV, fb, c[0], c[1], c[2], c[3]);
      c[p.v_perm[0]] = row0 + 64;
      tma_load_4d(sq + 2 * AT_TILE_BYTES + AT_TILE_BYTES / 2, &tmV, fb, c[0], c[1], c[2], c[3]);
      issued = i + 1;
    }
    if (!ok || *abort_flag) {
      // give up: let the copies already in flight land before the CTA leaves
      const int n = issued < AT_STAGES ? issued : AT_STAGES;
      for (int k = 0; k < n; k++) {
        const int j = issued - 1 - k;
        const uint32_t fb = smem_u32(&full_bar[j % AT_STAGES]);
        const long long t0 = now_cycles();
        while (!mbar_try_wait(fb, (uint32_t)(j / AT_STAGES) & 1) && now_cycles() - t0 < 200000000ll) {}
      }
    }
  } else if (warp == 1 && elect_one()) {
    // ------------------------------- MMA issuer -------------------------------
    bool ok = true;
    const uint32_t hi = (uint32_t)(make_smem_desc(0, 16) >> 32);           // same for both operand forms
    const uint32_t lbo_mn_lo = (uint32_t)make_smem_desc(0, 64 * BK * 2);   // low word carries the LBO field
    uint32_t cleaned = 0;  // parity of every stage's clean barrier
    auto issue_pv = [&](int j, int len) -> bool {  // C = P V of item j; P lies over the item's Q and K tiles
      const uint32_t s = (uint32_t)(j % AT_STAGES), g = (uint32_t)j & 1;
      if (kPacked && (len & 15)) {
        if (!mbar_wait(smem_u32(&clean_bar[s]), (cleaned >> s) & 1, abort_flag, p.status)) return false;
        cleaned ^= 1u << s;
        tc_fence_after();
      }
      const uint32_t sq = smem_u32(smem + (size_t)s * AT_STAGE_BYTES);
      const uint32_t p_lo = (uint32_t)make_smem_desc(sq, 16);
      const uint32_t v_lo = lbo_mn_lo | (((sq + 2 * AT_TILE_BYTES) & 0x3FFFFu) >> 4);
      uint32_t accum = 0;
#pragma unroll
      for (int kb = 0; kb < 2; kb++)
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; k++) {
          if (kPacked && kb * BK + k * UMMA_K >= len) continue;  // keys beyond the sequence
          const uint64_t ad = ((uint64_t)hi << 32) | (p_lo + kb * (AT_TILE_BYTES / 16) + k * (UMMA_K * 2 / 16));
          const uint64_t bd = ((uint64_t)hi << 32) | (v_lo + kb * (AT_TILE_BYTES / 2 / 16) + k * (UMMA_K * 128 / 16));
          tc_mma(tmem_base + AT_O_COL + g * 64, ad, bd, p.idesc_o, accum);
          accum = 1;
        }
      tc_commit(smem_u32(&ofull_bar[g]));
      tc_commit(smem_u32(&empty_bar[s]));  // the item's tiles are no longer needed
      return true;
    };
    int len_before = 0;  // a length is asked for one item before it is needed
    for (int i = 0; i < n_my && ok; i++) {
      const int len = kPacked ? item_len(i) : 128;
      const uint32_t s = (uint32_t)(i % AT_STAGES), round = (uint32_t)(i / AT_STAGES);
      const uint32_t b = (uint32_t)i & 1, use = (uint32_t)i >> 1;
      if (!mbar_wait(smem_u32(&full_bar[s]), round & 1, abort_flag, p.status)) { ok = false; break; }
      if (!mbar_wait(smem_u32(&sempty_bar[b]), (use & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      const uint32_t sq = smem_u32(smem + (size_t)s * AT_STAGE_BYTES);
      const uint32_t q_lo = (uint32_t)make_smem_desc(sq, 16), k_lo = (uint32_t)make_smem_desc(sq + AT_TILE_BYTES, 16);
#pragma unroll
      for (int k = 0; k < BK / UMMA_K; k++) {
        const uint64_t ad = ((uint64_t)hi << 32) | (q_lo + k * (UMMA_K * 2 / 16));
        const uint64_t bd = ((uint64_t)hi << 32) | (k_lo + k * (UMMA_K * 2 / 16));
        tc_mma(tmem_base + b * 128, ad, bd, p.idesc_s, k > 0 ? 1u : 0u);
      }
      tc_commit(smem_u32(&sfull_bar[b]));
      if (i > 0) {  // the previous item's probabilities: its group has been at work since S(i-1)
        const uint32_t g = (uint32_t)(i - 1) & 1, guse = (uint32_t)(i - 1) >> 1;
        if (!mbar_wait(smem_u32(&pready_bar[g]), guse & 1, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        if (!issue_pv(i - 1, len_before)) { ok = false; break; }
      }
      len_before = len;
    }
    if (ok && n_my > 0) {
      const uint32_t g = (uint32_t)(n_my - 1) & 1, guse = (uint32_t)(n_my - 1) >> 1;
      if (mbar_wait(smem_u32(&pready_bar[g]), guse & 1, abort_flag, p.status)) {
        tc_fence_after();
        ok = issue_pv(n_my - 1, len_before);
      } else {
        ok = false;
      }
    }
    if (!ok || *abort_flag) {
      // make sure no MMA is still writing tensor memory before it is freed
      tc_commit(smem_u32(&sfull_bar[0]));
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (kPacked && warp >= 2 + NUM_EPI_WARPS) {
    // ------------------------------- clearing of rows beyond the sequence -------------------------------
    int next = n_my ? item_len(0) : 0;
    for (int i = 0; i < n_my; i++) {
      const int len = next;
      if (i + 1 < n_my) next = item_len(i + 1);
      const uint32_t s = (uint32_t)(i % AT_STAGES);
      if (!mbar_wait(smem_u32(&full_bar[s]), (i / AT_STAGES) & 1, abort_flag, p.status)) break;
      if (len & 15) {
        clear_tile_rows(smem + (size_t)s * AT_STAGE_BYTES + 2 * AT_TILE_BYTES, len, (len + 15) & ~15, threadIdx.x - NUM_THREADS);
        clear_done(smem_u32(&clean_bar[s]), lane);
      }
      if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }
  } else if (warp >= 2) {
    // ------------------------------- softmax groups -------------------------------
    const int q = warp & 3;              // TMEM lane quarter this warp may read
    const int g = (warp - 2) >> 2;       // softmax group: items g, g + 2, ...
    uint8_t* stg = staging + (size_t)(warp - 2) * AT_STAGING;
    const int r = q * 32 + lane;         // query row this thread owns
    bool ok = true;
    for (int i = g; i < n_my && ok; i += 2) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int zo = w / p.heads, zi = w - zo * p.heads;
      const uint32_t s = (uint32_t)(i % AT_STAGES), use = (uint32_t)i >> 1;
      const int len = item_len(i);
      if (!mbar_wait(smem_u32(&sfull_bar[g]), use & 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      float2 v[4][16];  // the row's 128 scores, then its probabilities
      const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)g * 128;
#pragma unroll
      for (int c = 0; c < 4; c++) tc_ld32(trow + c * 32, v[c]);
      // the scores are in registers: hand the accumulator back
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sempty_bar[g]));
      // Row maximum over the valid keys: one chain per 32-column chunk keeps the dependent
      // chains short; only a chunk that crosses the length needs element-wise masking.
      float mc[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        mc[c] = -INFINITY;
        if ((c + 1) * 32 > len) {
#pragma unroll
          for (int j = 0; j < 16; j++) {
            if (c * 32 + 2 * j >= len) v[c][j].x = -INFINITY;
            if (c * 32 + 2 * j + 1 >= len) v[c][j].y = -INFINITY;
          }
        }
#pragma unroll
        for (int j = 0; j < 16; j++) mc[c] = fmaxf(mc[c], fmaxf(v[c][j].x, v[c][j].y));
      }
      const float mx = fmaxf(fmaxf(mc[0], mc[1]), fmaxf(mc[2], mc[3]));
      // exp(scale * (x - max)) as 2^(x * scale * log2(e) - max * scale * log2(e)): one packed
      // multiply-add per pair and one exponential per element; masked keys give 2^(-inf) = 0
      const float sl2 = p.scale * 1.4426950408889634f;
      const float2 k2 = splat2(sl2), nm2 = splat2(-mx * sl2);
      float2 sc[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        sc[c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 16; j++) {
          const float2 t = __ffma2_rn(v[c][j], k2, nm2);
          v[c][j].x = fast_exp2(t.x);
          v[c][j].y = fast_exp2(t.y);
          sc[c] = __fadd2_rn(sc[c], v[c][j]);
        }
      }
      const float sum = ((sc[0].x + sc[0].y) + (sc[1].x + sc[1].y)) + ((sc[2].x + sc[2].y) + (sc[3].x + sc[3].y));
      const float2 inv = splat2(1.0f / sum);
      // P as the A operand of the second product, over the item's Q and K tiles (both products
      // of the first kind have completed): k block = 64 keys = 16 KB, row r at 128 * r, its eight
      // 16-byte pieces permuted by r mod 8 (the 128-byte swizzle the tensor core expects)
      uint8_t* prow = smem + (size_t)s * AT_STAGE_BYTES + r * 128;
#pragma unroll
      for (int c = 0; c < 4; c++) {
#pragma unroll
        for (int j = 0; j < 16; j++) v[c][j] = __fmul2_rn(v[c][j], inv);
#pragma unroll
        for (int j = 0; j < 4; j++) {
          uint4 pk;
          __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&pk);
#pragma unroll
          for (int e = 0; e < 4; e++) h[e] = __float22bfloat162_rn(v[c][4 * j + e]);
          *reinterpret_cast<uint4*>(prow + (c >> 1) * AT_TILE_BYTES + ((((c & 1) * 4 + j) ^ (r & 7)) << 4)) = pk;
        }
      }
      // make the generic-proxy writes visible to the tensor core, then tell the MMA thread
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&pready_bar[g]));
      const int rlim = kPacked ? len : p.S;  // rows of the item that exist
      if (p.P != nullptr) {
        // the backward pass reads whole S x S blocks: rows that do not exist are stored as zeros
        if (kPacked && r >= rlim) {
#pragma unroll
          for (int c = 0; c < 4; c++)
#pragma unroll
            for (int j = 0; j < 16; j++) v[c][j] = make_float2(0.f, 0.f);
        }
        bf16* pg = p.P + zo * p.p_bo + zi * p.p_bi;
        if (p.fast_p) {  // S a multiple of 32: whole 32-column pieces only
          if (r < p.S) {
#pragma unroll
            for (int c = 0; c < 4; c++)
              if (c * 32 < p.S) store_row32_bf16(pg + (long long)r * p.S + c * 32, v[c]);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 4; c++)
            if (c * 32 < p.S) stage_store_bf16(stg, lane, v[c], pg, p.S, q * 32, c * 32, p.S, p.S, p.vec_ok_p);
        }
      }
      // context tile: 64 columns of this group's accumulator
      if (!mbar_wait(smem_u32(&ofull_bar[g]), use & 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      const uint32_t orow = tmem_base + ((uint32_t)(q * 32) << 16) + AT_O_COL + (uint32_t)g * 64;
      tc_ld32(orow, v[0]);
      tc_ld32(orow + 32, v[1]);
      tc_fence_before();
      bf16* cg = p.C + (kPacked ? p.cu[zo] * p.c_ld : zo * p.c_bo) + zi * p.c_bi;
      if (p.fast_c) {
        if (r < rlim) {
          store_row32_bf16(cg + (long long)r * p.c_ld, v[0]);
          store_row32_bf16(cg + (long long)r * p.c_ld + 32, v[1]);
        }
      } else {
        stage_store_bf16(stg, lane, v[0], cg, p.c_ld, q * 32, 0, rlim, 64, p.vec_ok_c);
        stage_store_bf16(stg, lane, v[1], cg, p.c_ld, q * 32, 32, rlim, 64, p.vec_ok_c);
      }
    }
    if (kPacked) zero_tail_rows(p.C, p.c_ld, p.heads * 64, p.rows);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AT_TMEM_COLS)
                 : "memory");
  }
}

// ---- forward for rows of 129..512 keys that stores the probabilities (single-kernel entry point) ----
// A work item is (sequence, head, tile of 128 queries); the keys come in blocks of 128.  The scores
// of a row do not fit tensor memory next to two context accumulators, so an item runs two passes over
// the key blocks: pass 1 forms the row maximum and the sum of exponentials (S = Q K_j^T only), pass 2
// forms the scores again, writes P_j = exp(.)/sum as bf16 and accumulates C += P_j V_j: probabilities
// that can be stored as they are.
// Each of the two softmax groups owns every second item of the CTA, whole: its own Q tile, ring of
// K / V tiles, score and context accumulators, P block, producer thread and MMA-issuing thread.  A
// thread owns one query row of its group's item through all key blocks, so nothing is exchanged
// between the groups, and the waits of one item (loads, the P hand-over, the last second product,
// the context store) are covered by the other item's arithmetic.  Measured on the earlier form, in
// which the two groups shared one item: 21 k cycles per item of which 8 k were exponentials.
constexpr int AL_THREADS = NUM_THREADS + 64;     // warps 10 and 11: MMA issuer and producer of group 1
constexpr int AL_RING = 3;                       // 16 KB tiles (a K block or a V block) per group
constexpr int AL_P_BYTES = 2 * AT_TILE_BYTES;    // P_j as an MMA operand: 32 KB
constexpr int AL_BARS_PER_GROUP = 4 + 2 * AL_RING + 6;
constexpr long long AL_GROUP_SKEW_CYCLES = 2000;

__global__ void __launch_bounds__(AL_THREADS, 1)
attn_fwd_long_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* q_smem = smem;                                        // [group] Q tile
  uint8_t* ring_smem = q_smem + 2 * AT_TILE_BYTES;               // [group][AL_RING] K or V tile
  uint8_t* p_smem = ring_smem + 2 * AL_RING * AT_TILE_BYTES;     // [group] P block
  uint8_t* staging = p_smem + 2 * AL_P_BYTES;
  uint64_t* bars = (uint64_t*)(staging + NUM_EPI_WARPS * AT_STAGING);
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * AL_BARS_PER_GROUP);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int g = 0; g < 2; g++) {
      uint64_t* b = bars + g * AL_BARS_PER_GROUP;
      for (int a = 0; a < 2 + 2 * AL_RING + 1; a++) mbar_init(smem_u32(&b[a]), 1);  // qfull, qempty, tfull[], tempty[], sfull
      mbar_init(smem_u32(&b[2 + 2 * AL_RING + 1]), AT_GROUP_WARPS);  // sempty
      mbar_init(smem_u32(&b[2 + 2 * AL_RING + 2]), AT_GROUP_WARPS);  // pready
      mbar_init(smem_u32(&b[2 + 2 * AL_RING + 3]), 1);               // pfree
      mbar_init(smem_u32(&b[2 + 2 * AL_RING + 4]), 1);               // ofull
      mbar_init(smem_u32(&b[2 + 2 * AL_RING + 5]), AT_GROUP_WARPS);  // oempty
    }
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmQ);
    prefetch_map(&tmK);
    prefetch_map(&tmV);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(AT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  const int nqt = (p.S + 127) >> 7;   // query tiles per (sequence, head); key blocks likewise
  const int nzh = p.items / nqt;      // (sequence, head) pairs
  // Keys at or beyond the sequence's length have probability 0: an item covers only the
  // ceil(len / 128) key blocks that hold valid keys, and a query tile that lies wholly in the
  // padding is not computed at all (its context rows, which nothing may depend on, are zeroed).
  // Every role derives the same counts from seq_lens.
  auto item_len = [&](int zo) {
    int len = p.seq_lens ? p.seq_lens[zo] : p.S;
    return min(max(len, 1), p.S);
  };
  const int n_my = ((int)blockIdx.x < p.items) ? (p.items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  // Which group this thread serves, and that group's barriers.  Running counts per group: ig items,
  // tt ring tiles, sp score products, pv second products; each barrier's phase is the parity of
  // the count it is used by.
  const int g = warp == 0 ? 0 : (warp == 1 ? 0 : (warp >= 10 ? 1 : (warp - 2) >> 2));
  uint64_t* gb = bars + g * AL_BARS_PER_GROUP;
  const uint32_t qfull = smem_u32(&gb[0]), qempty = smem_u32(&gb[1]);
  const uint32_t tfull0 = smem_u32(&gb[2]), tempty0 = smem_u32(&gb[2 + AL_RING]);
  const uint32_t sfull = smem_u32(&gb[2 + 2 * AL_RING]), sempty = smem_u32(&gb[2 + 2 * AL_RING + 1]);
  const uint32_t pready = smem_u32(&gb[2 + 2 * AL_RING + 2]), pfree = smem_u32(&gb[2 + 2 * AL_RING + 3]);
  const uint32_t ofull = smem_u32(&gb[2 + 2 * AL_RING + 4]), oempty = smem_u32(&gb[2 + 2 * AL_RING + 5]);
  uint8_t* my_q = q_smem + g * AT_TILE_BYTES;
  uint8_t* my_ring = ring_smem + (size_t)g * AL_RING * AT_TILE_BYTES;
  uint8_t* my_p = p_smem + (size_t)g * AL_P_BYTES;
  // Tiles of an item in the order the MMA thread uses them: pass 1: K_0 .. K_{n-1}; pass 2: K_0, then
  // (K_j, V_{j-1}) for j = 1 .. n-1, then V_{n-1} (the scores of block j are issued before the second
  // product of block j - 1, which has to wait for that block's probabilities).

  if ((warp == 0 || warp == 11) && !p.starve && elect_one()) {
    // ------------------------------- TMA producer of group g -------------------------------
    bool ok = true;
    uint32_t tt = 0, ig = 0;
    for (int i = g; i < n_my && ok; i += 2) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int qt = w / nzh, zh = w - qt * nzh;  // query tile slowest: tiles that may be padding come last
      const int zo = zh / p.heads, zi = zh - zo * p.heads;
      const int len = item_len(zo);
      if (qt * 128 >= len) continue;
      const int nkb = (len + 127) >> 7;
      if (!mbar_wait(qempty, (ig & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      ig++;
      int c[4];
      c[0] = 0; c[p.q_perm[0]] = qt * 128; c[p.q_perm[1]] = zi; c[p.q_perm[2]] = zo;
      mbar_expect_tx(qfull, AT_TILE_BYTES);
      tma_load_4d(smem_u32(my_q), &tmQ, qfull, c[0], c[1], c[2], c[3]);
      for (int idx = 0; idx < 3 * nkb; idx++, tt++) {
        // which block, and K or V
        int j = idx;
        bool is_v = false;
        if (idx >= nkb) {
          const int k = idx - nkb;
          if (k == 0) j = 0;
          else if (k == 2 * nkb - 1) { j = nkb - 1; is_v = true; }
          else if (k & 1) j = (k + 1) >> 1;
          else { j = (k >> 1) - 1; is_v = true; }
        }
        const uint32_t slot = tt % AL_RING, round = tt / AL_RING;
        if (!mbar_wait(tempty0 + slot * 8, (round & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        const uint32_t fb = tfull0 + slot * 8;
        mbar_expect_tx(fb, AT_TILE_BYTES);
        const int* perm = is_v ? p.v_perm : p.k_perm;
        c[0] = 0; c[1] = 0; c[2] = 0; c[3] = 0;
        c[perm[0]] = j * 128; c[perm[1]] = zi; c[perm[2]] = zo;
        tma_load_4d(smem_u32(my_ring + (size_t)slot * AT_TILE_BYTES), is_v ? &tmV : &tmK, fb, c[0], c[1], c[2], c[3]);
      }
    }
    if (!ok || *abort_flag) {  // give the copies in flight time to land before the CTA leaves
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 4000000ll) {}
    }
  } else if ((warp == 1 || warp == 10) && elect_one()) {
    // ------------------------------- MMA issuer of group g -------------------------------
    bool ok = true;
    const uint32_t hi = (uint32_t)(make_smem_desc(0, 16) >> 32);
    const uint32_t lbo_mn_lo = (uint32_t)make_smem_desc(0, 64 * BK * 2);
    const uint32_t p_lo = (uint32_t)make_smem_desc(smem_u32(my_p), 16);
    const uint32_t q_lo = (uint32_t)make_smem_desc(smem_u32(my_q), 16);
    const uint32_t s_tmem = tmem_base + (uint32_t)g * 128, o_tmem = tmem_base + AT_O_COL + (uint32_t)g * 64;
    uint32_t tt = 0, sp = 0, pv = 0, ig = 0;
    if (g == 1) {
      // The two groups do the same work at the same pace: started together they would want the
      // exponential unit at the same moments and leave it idle at the same moments.  Half a block
      // period of head start for group 0 keeps them out of step.
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < AL_GROUP_SKEW_CYCLES) {}
    }
    for (int i = g; i < n_my && ok; i += 2) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int qt = w / nzh, zh = w - qt * nzh;
      const int len = item_len(zh / p.heads);
      if (qt * 128 >= len) continue;
      const int nkb = (len + 127) >> 7;
      if (!mbar_wait(qfull, ig & 1, abort_flag, p.status)) { ok = false; break; }
      auto issue_scores = [&]() -> bool {  // S = Q K^T with the K tile in ring position tt
        const uint32_t slot = tt % AL_RING, round = tt / AL_RING;
        if (!mbar_wait(tfull0 + slot * 8, round & 1, abort_flag, p.status)) return false;
        if (!mbar_wait(sempty, (sp & 1) ^ 1, abort_flag, p.status)) return false;
        tc_fence_after();
        const uint32_t k_lo = (uint32_t)make_smem_desc(smem_u32(my_ring + (size_t)slot * AT_TILE_BYTES), 16);
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; k++) {
          const uint64_t ad = ((uint64_t)hi << 32) | (q_lo + k * (UMMA_K * 2 / 16));
          const uint64_t bd = ((uint64_t)hi << 32) | (k_lo + k * (UMMA_K * 2 / 16));
          tc_mma(s_tmem, ad, bd, p.idesc_s, k > 0 ? 1u : 0u);
        }
        tc_commit(sfull);
        tc_commit(tempty0 + slot * 8);  // the K tile is free once the product has completed
        tt++; sp++;
        return true;
      };
      auto issue_pv = [&](int j) -> bool {  // C (+)= P_j V_j with the V tile in ring position tt
        const uint32_t slot = tt % AL_RING, round = tt / AL_RING;
        if (!mbar_wait(pready, pv & 1, abort_flag, p.status)) return false;
        if (j == 0 && !mbar_wait(oempty, (ig & 1) ^ 1, abort_flag, p.status)) return false;
        if (!mbar_wait(tfull0 + slot * 8, round & 1, abort_flag, p.status)) return false;
        tc_fence_after();
        const uint32_t sv = smem_u32(my_ring + (size_t)slot * AT_TILE_BYTES);
        const uint32_t v_lo = lbo_mn_lo | ((sv & 0x3FFFFu) >> 4);
#pragma unroll
        for (int kb = 0; kb < 2; kb++)
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; k++) {
            const uint64_t ad = ((uint64_t)hi << 32) | (p_lo + kb * (AT_TILE_BYTES / 16) + k * (UMMA_K * 2 / 16));
            const uint64_t bd = ((uint64_t)hi << 32) | (v_lo + kb * (AT_TILE_BYTES / 2 / 16) + k * (UMMA_K * 128 / 16));
            tc_mma(o_tmem, ad, bd, p.idesc_o, (j > 0 || kb > 0 || k > 0) ? 1u : 0u);
          }
        tc_commit(pfree);
        tc_commit(tempty0 + slot * 8);
        tt++; pv++;
        return true;
      };
      for (int j = 0; j < nkb && ok; j++) ok = issue_scores();  // pass 1
      if (ok) ok = issue_scores();                                 // pass 2
      for (int j = 1; j < nkb && ok; j++) {
        ok = issue_scores();
        if (ok && j == nkb - 1) tc_commit(qempty);  // the last product that reads Q has been issued
        if (ok) ok = issue_pv(j - 1);
      }
      if (ok && nkb == 1) tc_commit(qempty);
      if (ok) ok = issue_pv(nkb - 1);
      if (ok) tc_commit(ofull);
      ig++;
    }
    if (!ok || *abort_flag) {
      tc_commit(sfull);
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (warp >= 2 && warp < 2 + NUM_EPI_WARPS) {
    // ------------------------------- softmax group g -------------------------------
    const int q = warp & 3;
    uint8_t* stg = staging + (size_t)(warp - 2) * AT_STAGING;
    const int r = q * 32 + lane;
    const float sl2 = p.scale * 1.4426950408889634f;
    const float2 k2 = splat2(sl2);
    bool ok = true;
    uint32_t sp = 0, pv = 0, ig = 0;
    const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)g * 128;
    const uint32_t orow = tmem_base + ((uint32_t)(q * 32) << 16) + AT_O_COL + (uint32_t)g * 64;
    for (int i = g; i < n_my && ok; i += 2) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int qt = w / nzh, zh = w - qt * nzh;
      const int zo = zh / p.heads, zi = zh - zo * p.heads;
      const int len = item_len(zo);
      float2 v[4][16];
      bf16* cg = p.C + zo * p.c_bo + zi * p.c_bi + (long long)qt * 128 * p.c_ld;
      bf16* pg = p.P + zo * p.p_bo + zi * p.p_bi + (long long)qt * 128 * p.S;
      if (qt * 128 >= len) {
        // a query tile in the padding: zero context rows (finite, so that masked reads stay harmless)
#pragma unroll
        for (int e = 0; e < 16; e++) v[0][e] = make_float2(0.f, 0.f);
        stage_store_bf16(stg, lane, v[0], cg, p.c_ld, q * 32, 0, p.S - qt * 128, 64, p.vec_ok_c);
        stage_store_bf16(stg, lane, v[0], cg, p.c_ld, q * 32, 32, p.S - qt * 128, 64, p.vec_ok_c);
        for (int n0 = 0; n0 < p.S; n0 += 32)
          stage_store_bf16(stg, lane, v[0], pg, p.S, q * 32, n0, p.S - qt * 128, p.S, p.vec_ok_p);
        continue;
      }
      const int nkb = (len + 127) >> 7;
      // reads the group's next score block into v, masks it; returns its row maximum
      auto load_block = [&](int j, float& bm) -> bool {
        if (!mbar_wait(sfull, sp & 1, abort_flag, p.status)) return false;
        sp++;
        tc_fence_after();
        tc_ld128(trow, v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sempty);
        float mc[4];
#pragma unroll
        for (int c = 0; c < 4; c++) {
          mc[c] = -INFINITY;
          const int k0 = j * 128 + c * 32;
          if (k0 + 32 > len) {
#pragma unroll
            for (int e = 0; e < 16; e++) {
              if (k0 + 2 * e >= len) v[c][e].x = -INFINITY;
              if (k0 + 2 * e + 1 >= len) v[c][e].y = -INFINITY;
            }
          }
#pragma unroll
          for (int e = 0; e < 16; e++) mc[c] = fmaxf(mc[c], fmaxf(v[c][e].x, v[c][e].y));
        }
        bm = fmaxf(fmaxf(mc[0], mc[1]), fmaxf(mc[2], mc[3]));
        return true;
      };
      // pass 1: running maximum of the raw scores and running sum
      // of 2^((s - max) * scale * log2 e)
      float mr = -INFINITY, l = 0.f;
      for (int j = 0; j < nkb && ok; j++) {
        float bm;
        if (!load_block(j, bm)) { ok = false; break; }
        const float mn = fmaxf(mr, bm);
        if (mn != -INFINITY) {
          const float2 nm2 = splat2(-mn * sl2);
          float2 sc[4];
#pragma unroll
          for (int c = 0; c < 4; c++) {
            sc[c] = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 16; e++) {
              const float2 a = __ffma2_rn(v[c][e], k2, nm2);
              sc[c] = __fadd2_rn(sc[c], make_float2(fast_exp2(a.x), fast_exp2(a.y)));
            }
          }
          const float bs = ((sc[0].x + sc[0].y) + (sc[1].x + sc[1].y)) + ((sc[2].x + sc[2].y) + (sc[3].x + sc[3].y));
          l = l * fast_exp2((mr - mn) * sl2) + bs;  // 2^(-inf) = 0 on the first valid block
        }
        mr = mn;
      }
      if (!ok) break;
      // mr is finite: at least one key of the row is valid
      const float2 nM2 = splat2(-mr * sl2);
      const float2 inv = splat2(1.0f / l);
      // pass 2
      for (int j = 0; j < nkb && ok; j++) {
        float bm;
        if (!load_block(j, bm)) { ok = false; break; }
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
          for (int e = 0; e < 16; e++) {
            const float2 a = __ffma2_rn(v[c][e], k2, nM2);
            const float2 ex = make_float2(fast_exp2(a.x), fast_exp2(a.y));
            v[c][e] = __fmul2_rn(ex, inv);
          }
        // the group's P block is free once its previous second product has read it
        if (!mbar_wait(pfree, (pv & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        pv++;
        uint8_t* prow = my_p + r * 128;
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
          for (int e4 = 0; e4 < 4; e4++) {
            uint4 pk;
            __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&pk);
#pragma unroll
            for (int e = 0; e < 4; e++) h[e] = __float22bfloat162_rn(v[c][4 * e4 + e]);
            *reinterpret_cast<uint4*>(prow + (c >> 1) * AT_TILE_BYTES + ((((c & 1) * 4 + e4) ^ (r & 7)) << 4)) = pk;
          }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(pready);
        if (pg != nullptr) {
          if (p.fast_p) {
            if (qt * 128 + r < p.S) {
#pragma unroll
              for (int c = 0; c < 4; c++)
                if (j * 128 + c * 32 < p.S) store_row32_bf16(pg + (long long)r * p.S + j * 128 + c * 32, v[c]);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 4; c++)
              if (j * 128 + c * 32 < p.S)
                stage_store_bf16(stg, lane, v[c], pg, p.S, q * 32, j * 128 + c * 32, p.S - qt * 128, p.S, p.vec_ok_p);
          }
        }
      }
      if (!ok) break;
      // key blocks past the length: their probabilities are 0
      if (pg != nullptr && nkb * 128 < p.S) {
        float2 zr[16];
#pragma unroll
        for (int e = 0; e < 16; e++) zr[e] = make_float2(0.f, 0.f);
        for (int n0 = nkb * 128; n0 < p.S; n0 += 32)
          stage_store_bf16(stg, lane, zr, pg, p.S, q * 32, n0, p.S - qt * 128, p.S, p.vec_ok_p);
      }
      // context tile: the row's 64 columns
      if (!mbar_wait(ofull, ig & 1, abort_flag, p.status)) { ok = false; break; }
      ig++;
      tc_fence_after();
      tc_ld32(orow, v[0]);
      tc_ld32(orow + 32, v[1]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(oempty);
      if (p.fast_c) {
        if (qt * 128 + r < p.S) {
          store_row32_bf16(cg + (long long)r * p.c_ld, v[0]);
          store_row32_bf16(cg + (long long)r * p.c_ld + 32, v[1]);
        }
      } else {
        stage_store_bf16(stg, lane, v[0], cg, p.c_ld, q * 32, 0, p.S - qt * 128, 64, p.vec_ok_c);
        stage_store_bf16(stg, lane, v[1], cg, p.c_ld, q * 32, 32, p.S - qt * 128, 64, p.vec_ok_c);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AT_TMEM_COLS)
                 : "memory");
  }
}

// ---- forward for rows of 129..512 keys, no probabilities stored -----------------------------------
// A work item is (sequence, head, tile of 128 queries).  Tensor memory holds the scores of a whole row
// (four blocks of 128 keys), so they are formed once: all sixteen softmax warps read them twice, first for
// the row maximum, then for the exponentials, and the context accumulates over columns whose scores have
// been used up (block 0 when there are four blocks, else the upper half of the unused block 3).
// A thread owns a quarter of one query row's scores in every key block; the quarters exchange maximum and
// sum through shared memory.  P_j goes to one of two shared-memory blocks as the second product's operand.
//   warp 0: TMA producer (Q tile, ring of K and V tiles: K_0 .. K_{n-1}, V_0 .. V_{n-1})
//   warp 1: MMA issuer: the next item's scores are issued behind this item's last second product, so they
//           are ready when the softmax warps have stored the context
//   warps 2-17: softmax; packed batches: warps 18, 19 clear the last V tile's rows beyond the sequence
// Bound by the exponential unit (16 a clock: 1024 cycles per block) and the passes around it.
// 16 sequences x 16 heads x 512 keys: 59.5 us with two groups of warps on items of their own and the scores
// formed twice; 49.5 us in this form with eight softmax warps (two per scheduler do not cover the
// tensor-memory reads and the fences); 48.3 us with sixteen, 46.2 with elected copying and issuing threads
// (64 x 12 x 256 keys 48.8, 12 x 16 x 384 24.2, 21 x 12 x 232 20.7).
// In steps of BERT-Large at 16 x (256..512) keys, packed tiles dealt out longest first: 56.8 -> 52.1 us a layer.
// The row's maximum is the reference of the exponentials, so that the largest probability is exactly 1 in bf16 and
// no context exceeds the largest value.  A form with two groups of warps that read the scores once, relative to the
// largest of a row's first 32, took 42.6 us (64 x 12 x 256 keys 40.6); its context was up to 1.27 times as far from
// float64 (a key of weight 0.3 past the first 32) and overflowed where values are large.
constexpr int AR_RING = 8;
constexpr int AR_TABLE = 256;  // items of a block described in shared memory; any beyond are read from memory
constexpr int AR_WARPS = 16;  // softmax warps: four per TMEM lane quarter
constexpr int AR_THREADS = 64 + 32 * AR_WARPS;

// 16 consecutive accumulator columns of this lane's row
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
// Hand-over between the four warps of a lane quarter (pair_sync for more partners).
__device__ __forceinline__ bool quad_sync(volatile int* flags, int me, int seq, int lane, volatile int* abort_flag, int* status) {
  __syncwarp();
  int ok = 1;
  if (lane == 0) {
    __threadfence_block();
    flags[me] = seq;
    const long long t0 = now_cycles();
    uint32_t spins = 0;
    const int first = me & ~3;
    while (flags[first] < seq || flags[first + 1] < seq || flags[first + 2] < seq || flags[first + 3] < seq) {
      if ((++spins & 255u) == 0u) {
        if (*abort_flag) { ok = 0; break; }
        if (now_cycles() - t0 > *reinterpret_cast<volatile long long*>(abort_flag + 1)) {
          *abort_flag = 1;
          atomicOr(status, ST_WAIT_TIMEOUT);
          ok = 0;
          break;
        }
      }
    }
    __threadfence_block();
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  return ok != 0;
}

template <bool kPacked>
__global__ void __launch_bounds__(AR_THREADS + (kPacked ? 32 * CLEAR_WARPS : 0), 1)
attn_fwd_rows_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* ring_smem = smem + AT_TILE_BYTES;                  // Q first
  uint8_t* p_smem = ring_smem + AR_RING * AT_TILE_BYTES;      // two blocks of P, 32 KB each
  float* xch = (float*)(p_smem + 4 * AT_TILE_BYTES);          // [2][AR_WARPS][32] maxima, sums
  int4* table = (int4*)(xch + 2 * AR_WARPS * 32);             // [AR_TABLE] items of this block
  volatile int* xflag = (volatile int*)(table + AR_TABLE);
  uint64_t* bars = (uint64_t*)(xflag + AR_WARPS);
  const uint32_t qfull = smem_u32(&bars[0]), qempty = smem_u32(&bars[1]);
  const uint32_t tfull0 = smem_u32(&bars[2]), tempty0 = smem_u32(&bars[2 + AR_RING]);
  const uint32_t sfull = smem_u32(&bars[2 + 2 * AR_RING]);
  const uint32_t pready0 = smem_u32(&bars[3 + 2 * AR_RING]), pfree0 = smem_u32(&bars[5 + 2 * AR_RING]);  // [2] each
  const uint32_t ofull = smem_u32(&bars[7 + 2 * AR_RING]), oempty = smem_u32(&bars[8 + 2 * AR_RING]);
  const uint32_t clean0 = smem_u32(&bars[9 + 2 * AR_RING]);  // [AR_RING]
  uint32_t* tmem_slot = (uint32_t*)(bars + 9 + 3 * AR_RING);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(qfull, 1); mbar_init(qempty, 1); mbar_init(sfull, 1); mbar_init(ofull, 1);
    mbar_init(oempty, AR_WARPS);
    for (int s = 0; s < AR_RING; s++) {
      mbar_init(tfull0 + 8 * s, 1);
      mbar_init(tempty0 + 8 * s, 1 + (kPacked ? CLEAR_WARPS : 0));
      mbar_init(clean0 + 8 * s, CLEAR_WARPS);
    }
    for (int b = 0; b < 2; b++) { mbar_init(pready0 + 8 * b, AR_WARPS); mbar_init(pfree0 + 8 * b, 1); }
    for (int i = 0; i < AR_WARPS; i++) xflag[i] = 0;
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmQ);
    prefetch_map(&tmK);
    prefetch_map(&tmV);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(AT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  // Items: packed batches list the query tiles that exist, those of the longest sequences first, so that
  // dealing them out leaves the CTAs level; otherwise the query tile is the slow index.
  const int nzh = p.items / ((p.S + 127) >> 7);
  const int n_items = kPacked ? p.rows[2] * p.heads : p.items;
  const int n_my = (int)blockIdx.x < n_items ? (n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  auto describe = [&](int i) -> int4 {  // {first row of the sequence, its length, sequence, query tile and head}
    const int w = (int)blockIdx.x + i * (int)gridDim.x;
    int zo, zi, qt;
    if (kPacked) {
      const int e = w / p.heads;
      zi = w - e * p.heads;
      zo = p.order[e] >> 3;
      qt = p.order[e] & 7;
    } else {
      qt = w / nzh;
      zo = (w - qt * nzh) / p.heads;
      zi = (w - qt * nzh) - zo * p.heads;
    }
    const int len = p.seq_lens ? p.seq_lens[zo] : p.S;
    return make_int4(kPacked ? p.cu[zo] : zo * p.S, min(max(len, 1), p.S), zo, qt << 24 | zi);
  };
  // Every role needs these words at the start of every item, and read from memory one after another they held up each
  // item by 0.7 us (64 sequences x 12 heads x 256 keys: 50.0 us without lengths, 58.6 with).  So all are fetched once;
  // a block of a single item has nothing to gain (5 x 12 x 256: 8.5 us, 9.0 by way of the table).
  const int listed = n_my > 1 ? min(n_my, AR_TABLE) : 0;
  if (listed) {
    for (int i = threadIdx.x; i < listed; i += blockDim.x) table[i] = describe(i);
    __syncthreads();
  }
  auto item = [&](int i) -> int4 { return i < listed ? table[i] : describe(i); };
  // column of the context accumulator, and the key block it lies in
  auto o_block = [](int n) { return n == 4 ? 0 : 3; };
  auto o_col = [](int n) { return n == 4 ? 0u : 448u; };

  if (warp == 0 && !p.starve && elect_one()) {
    // ------------------------------- TMA producer -------------------------------
    bool ok = true;
    uint32_t tt = 0, ig = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int4 it = item(i);
      const int len = it.y, zi = it.w & 0xffffff, qt = it.w >> 24;
      if (qt * 128 >= len) continue;
      const int n = (len + 127) >> 7;
      const int row0 = kPacked ? it.x : 0, zseq = kPacked ? 0 : it.z;
      if (!mbar_wait(qempty, (ig & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      ig++;
      int c[4];
      c[0] = 0; c[p.q_perm[0]] = row0 + qt * 128; c[p.q_perm[1]] = zi; c[p.q_perm[2]] = zseq;
      mbar_expect_tx(qfull, AT_TILE_BYTES);
      tma_load_4d(smem_u32(smem), &tmQ, qfull, c[0], c[1], c[2], c[3]);
      for (int k = 0; k < 2 * n; k++, tt++) {
        const bool is_v = k >= n;
        const uint32_t slot = tt % AR_RING, round = tt / AR_RING;
        if (!mbar_wait(tempty0 + 8 * slot, (round & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        mbar_expect_tx(tfull0 + 8 * slot, AT_TILE_BYTES);
        const int* perm = is_v ? p.v_perm : p.k_perm;
        c[0] = 0; c[perm[0]] = row0 + (is_v ? k - n : k) * 128; c[perm[1]] = zi; c[perm[2]] = zseq;
        tma_load_4d(smem_u32(ring_smem + (size_t)slot * AT_TILE_BYTES), is_v ? &tmV : &tmK, tfull0 + 8 * slot, c[0], c[1], c[2], c[3]);
      }
    }
    if (!ok || *abort_flag) {  // give the copies in flight time to land before the CTA leaves
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 4000000ll) {}
    }
  } else if (warp == 1 && elect_one()) {
    // ------------------------------- MMA issuer -------------------------------
    bool ok = true;
    const uint32_t hi = (uint32_t)(make_smem_desc(0, 16) >> 32);
    const uint32_t lbo_mn_lo = (uint32_t)make_smem_desc(0, 64 * BK * 2);
    const uint32_t q_lo = (uint32_t)make_smem_desc(smem_u32(smem), 16);
    uint32_t tt = 0, pv = 0, ig = 0;  // ring tiles, second products, items
    uint32_t cleaned = 0;             // parity of every slot's clean barrier
    int n_prev = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int4 it = item(i);
      const int len = it.y;
      if ((it.w >> 24) * 128 >= len) continue;
      const int n = (len + 127) >> 7;
      if (!mbar_wait(qfull, ig & 1, abort_flag, p.status)) { ok = false; break; }
      auto scores = [&](int j) -> bool {  // S_j = Q K_j^T
        const uint32_t pos = tt + j, slot = pos % AR_RING;
        if (!mbar_wait(tfull0 + 8 * slot, (pos / AR_RING) & 1, abort_flag, p.status)) return false;
        tc_fence_after();
        const uint32_t k_lo = (uint32_t)make_smem_desc(smem_u32(ring_smem + (size_t)slot * AT_TILE_BYTES), 16);
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; k++) {
          const uint64_t ad = ((uint64_t)hi << 32) | (q_lo + k * (UMMA_K * 2 / 16));
          const uint64_t bd = ((uint64_t)hi << 32) | (k_lo + k * (UMMA_K * 2 / 16));
          tc_mma(tmem_base + j * 128, ad, bd, p.idesc_s, k > 0 ? 1u : 0u);
        }
        tc_commit(tempty0 + 8 * slot);
        return true;
      };
      // The scores of the item before have been read (its P blocks were waited for below); only the block
      // its context lies in has to wait until that context has been read.
      const int held = n_prev ? o_block(n_prev) : -1;
      for (int j = 0; j < n && ok; j++)
        if (j != held) ok = scores(j);
      if (ok && n_prev && !mbar_wait(oempty, (ig & 1) ^ 1, abort_flag, p.status)) ok = false;
      if (ok && held >= 0 && held < n) ok = scores(held);
      if (!ok) break;
      tc_commit(sfull);
      tc_commit(qempty);
      tt += n;
      for (int j = 0; j < n; j++, pv++, tt++) {  // C (+)= P_j V_j
        const uint32_t slot = tt % AR_RING, b = pv & 1;
        const bool edge = kPacked && (j + 1) * 128 > len;
        if (!mbar_wait(pready0 + 8 * b, (pv >> 1) & 1, abort_flag, p.status) ||
            !mbar_wait(edge ? clean0 + 8 * slot : tfull0 + 8 * slot, edge ? (cleaned >> slot) & 1 : (tt / AR_RING) & 1, abort_flag,
                       p.status)) { ok = false; break; }
        if (edge) cleaned ^= 1u << slot;
        tc_fence_after();
        const uint32_t p_lo = (uint32_t)make_smem_desc(smem_u32(p_smem + b * 2 * AT_TILE_BYTES), 16);
        const uint32_t v_lo = lbo_mn_lo | ((smem_u32(ring_smem + (size_t)slot * AT_TILE_BYTES) & 0x3FFFFu) >> 4);
#pragma unroll
        for (int kb = 0; kb < 2; kb++)
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; k++) {
            const uint64_t ad = ((uint64_t)hi << 32) | (p_lo + kb * (AT_TILE_BYTES / 16) + k * (UMMA_K * 2 / 16));
            const uint64_t bd = ((uint64_t)hi << 32) | (v_lo + kb * (AT_TILE_BYTES / 2 / 16) + k * (UMMA_K * 128 / 16));
            tc_mma(tmem_base + o_col(n), ad, bd, p.idesc_o, (j > 0 || kb > 0 || k > 0) ? 1u : 0u);
          }
        tc_commit(pfree0 + 8 * b);
        tc_commit(tempty0 + 8 * slot);
      }
      if (ok) tc_commit(ofull);
      ig++;
      n_prev = n;
    }
    if (!ok || *abort_flag) {  // make sure no MMA is still writing tensor memory before it is freed
      tc_commit(sfull);
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (kPacked && warp >= 2 + AR_WARPS) {
    // ------------------------------- clearing of rows beyond the sequence -------------------------------
    bool ok = true;
    uint32_t tt = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int len = item(i).y, n = (len + 127) >> 7;
      for (int k = 0; k < 2 * n; k++, tt++) {
        const uint32_t slot = tt % AR_RING;
        if (!mbar_wait(tfull0 + 8 * slot, (tt / AR_RING) & 1, abort_flag, p.status)) { ok = false; break; }
        if (k == 2 * n - 1 && len < n * 128) {
          clear_tile_rows(ring_smem + (size_t)slot * AT_TILE_BYTES, len - (n - 1) * 128, 128, threadIdx.x - AR_THREADS);
          clear_done(clean0 + 8 * slot, lane);
        }
        if (lane == 0) mbar_arrive(tempty0 + 8 * slot);
      }
    }
  } else if (warp >= 2) {
    // ------------------------------- softmax warps -------------------------------
    const int q = warp & 3, part = (warp - 2) >> 2;  // columns part * 32 .. of every key block
    const int me = q * 4 + part;
    const int r = q * 32 + lane;
    const float sl2 = p.scale * 1.4426950408889634f;
    const float2 k2 = splat2(sl2);
    const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16);
    float* xsum = xch + AR_WARPS * 32;
    bool ok = true;
    uint32_t pv = 0, ig = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int4 it = item(i);
      const int row0 = it.x, len = it.y, zi = it.w & 0xffffff, qt = it.w >> 24;
      const int rlim = kPacked ? len : p.S;  // rows of the sequence that exist
      bf16* crow = p.C + (long long)(row0 + qt * 128 + r) * p.c_ld + zi * p.c_bi + part * 16;
      const bool row_ok = qt * 128 + r < rlim;
      if (qt * 128 >= len) {
        // a query tile in the padding: zero context rows (finite, so that masked reads stay harmless)
        if (row_ok)
          for (int e = 0; e < 2; e++) *reinterpret_cast<uint4*>(crow + 8 * e) = make_uint4(0, 0, 0, 0);
        continue;
      }
      const int n = (len + 127) >> 7;
      if (!mbar_wait(sfull, ig & 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      uint32_t s[32];
      auto load = [&](int j) {  // this thread's 32 scores of block j, keys beyond the sequence at -inf
        tc_ld32_issue(trow + j * 128 + part * 32, s);
        tc_ld32_wait(s);
        const int k0 = j * 128 + part * 32;
        if (k0 + 32 > len) {
#pragma unroll
          for (int e = 0; e < 32; e++)
            if (k0 + e >= len) s[e] = 0xff800000u;
        }
      };
      // pass 1: the row's maximum
      float mx = -INFINITY;
      for (int j = 0; j < n; j++) {
        load(j);
        float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          m0 = fmaxf(m0, __uint_as_float(s[e]));
          m1 = fmaxf(m1, __uint_as_float(s[e + 1]));
          m2 = fmaxf(m2, __uint_as_float(s[e + 2]));
          m3 = fmaxf(m3, __uint_as_float(s[e + 3]));
        }
        mx = fmaxf(mx, fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)));
      }
      xch[me * 32 + lane] = mx;
      if (!quad_sync(xflag, me, (int)ig * 2 + 1, lane, abort_flag, p.status)) { ok = false; break; }
#pragma unroll
      for (int o = 0; o < 4; o++) mx = fmaxf(mx, xch[(q * 4 + o) * 32 + lane]);  // finite: one key is valid
      // pass 2: exponentials, their sum, and P_j
      const float2 nm2 = splat2(-mx * sl2);
      float2 l0 = make_float2(0.f, 0.f);
      for (int j = 0; j < n; j++, pv++) {
        load(j);
#pragma unroll
        for (int e = 0; e < 16; e++) {
          const float2 a = __ffma2_rn(make_float2(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), k2, nm2);
          const float2 ea = make_float2(fast_exp2(a.x), fast_exp2(a.y));
          l0 = __fadd2_rn(l0, ea);
          const __nv_bfloat162 pa = __float22bfloat162_rn(ea);
          s[e] = *reinterpret_cast<const uint32_t*>(&pa);
        }
        const uint32_t b = pv & 1;
        if (!mbar_wait(pfree0 + 8 * b, ((pv >> 1) & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        uint8_t* prow = p_smem + (b * 2 + (part >> 1)) * AT_TILE_BYTES + r * 128;
#pragma unroll
        for (int c = 0; c < 4; c++)
          *reinterpret_cast<uint4*>(prow + ((((part & 1) * 4 + c) ^ (r & 7)) << 4)) = make_uint4(s[4 * c], s[4 * c + 1], s[4 * c + 2], s[4 * c + 3]);
        tc_fence_before();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(pready0 + 8 * b);
      }
      if (!ok) break;
      xsum[me * 32 + lane] = l0.x + l0.y;
      if (!quad_sync(xflag, me, (int)ig * 2 + 2, lane, abort_flag, p.status)) { ok = false; break; }
      float sum = 0.f;
#pragma unroll
      for (int o = 0; o < 4; o++) sum += xsum[(q * 4 + o) * 32 + lane];
      if (p.lse && part == 0 && row_ok) p.lse[zi * p.lse_ld + row0 + qt * 128 + r] = mx * sl2 + log2f(sum);
      // the context: 16 of the row's 64 columns
      if (!mbar_wait(ofull, ig & 1, abort_flag, p.status)) { ok = false; break; }
      ig++;
      tc_fence_after();
      uint32_t v[16];
      tc_ld16(trow + o_col(n) + part * 16, v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(oempty);
      if (row_ok) {
        const float2 il = splat2(1.0f / sum);
#pragma unroll
        for (int e = 0; e < 2; e++) {
          uint4 o;
          __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
          for (int t = 0; t < 4; t++)
            h[t] = __float22bfloat162_rn(__fmul2_rn(make_float2(__uint_as_float(v[8 * e + 2 * t]), __uint_as_float(v[8 * e + 2 * t + 1])), il));
          *reinterpret_cast<uint4*>(crow + 8 * e) = o;
        }
      }
    }
    if (kPacked && warp < 2 + NUM_EPI_WARPS) zero_tail_rows(p.C, p.c_ld, p.heads * 64, p.rows);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AT_TMEM_COLS)
                 : "memory");
  }
}

// ---- backward ---------------------------------------------------------------------------------------
// Per (sequence, head) item, with P the saved probabilities and dC the gradient of the context:
//   dV = P^T dC,  dP = dC V^T,  dS = P o (dP - rowsum(dP o P)) * scale,  dQ = dS K,  dK = dS^T Q.
// The same roles as the forward kernel.  One shared-memory stage holds the item's Q, K, V, dC and
// P tiles, every tile as 128-byte-swizzled rows indexed by position, which serves both operand
// forms: rows as the m/n index with k contiguous, or rows as the k index with m/n contiguous.
// dS (bf16) overwrites P once the first two products have completed.  A softmax group's thread
// owns row r of its item: query r of dP, dS and dQ, key r of dK and dV.  Tensor memory per group:
// dP in 128 columns, later reused by dQ and dK, and dV in 64.
constexpr int AB_STAGE_BYTES = 6 * AT_TILE_BYTES;  // Q, K, V, dC, P (two tiles): 96 KB
constexpr uint32_t AB_GROUP_COLS = 192;

struct AttnBwdParams {
  int S, heads, items;
  float scale;
  const int* seq_lens;  // with cu / rows: packed rows, as in the forward kernels
  const int* cu;
  const int* rows;
  bf16* dQKV;         // element (b, i, which, h, e) at dQKV + b * g_bo + i * g_ld + which * H + h * 64 + e
  long long g_ld, g_bo, H;
  int vec_ok;
  int q_perm[3], k_perm[3], v_perm[3], c_perm[3], p_perm[3];
  long long wait_limit;
  int starve;         // test hook, as in the forward kernels
  int* status;
  uint32_t idesc_dv, idesc_dp, idesc_dq, idesc_dk;
};

__global__ void __launch_bounds__(NUM_THREADS + 32 * CLEAR_WARPS, 1)
attn_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmC,
                const __grid_constant__ CUtensorMap tmP, const AttnBwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* staging = smem + 2 * AB_STAGE_BYTES;
  uint64_t* bars = (uint64_t*)(staging + NUM_EPI_WARPS * AT_STAGING);
  uint64_t* full_bar = bars;           // [2] the item's tiles have landed (stage = group = item parity)
  uint64_t* empty_bar = bars + 2;      // [2] every product of the item has read them
  uint64_t* dpfull_bar = bars + 4;     // [2] dV and dP complete
  uint64_t* dsready_bar = bars + 6;    // [2] dS in shared memory, dP read by the whole group
  uint64_t* gfull_bar = bars + 8;      // [2] dQ and dK complete
  uint64_t* accfree_bar = bars + 10;   // [2] the group has read dQ, dK, dV of its item
  uint64_t* clean_bar = bars + 12;     // [2] packed: the rows of the item's tiles beyond the sequence are zero
  uint32_t* tmem_slot = (uint32_t*)(bars + 14);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int a = 0; a < 2; a++) {
      mbar_init(smem_u32(&full_bar[a]), 1);
      mbar_init(smem_u32(&empty_bar[a]), 1 + (p.cu ? CLEAR_WARPS : 0));
      mbar_init(smem_u32(&dpfull_bar[a]), 1);
      mbar_init(smem_u32(&dsready_bar[a]), AT_GROUP_WARPS);
      mbar_init(smem_u32(&gfull_bar[a]), 1);
      mbar_init(smem_u32(&accfree_bar[a]), AT_GROUP_WARPS);
      mbar_init(smem_u32(&clean_bar[a]), CLEAR_WARPS);
    }
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmQ);
    prefetch_map(&tmK);
    prefetch_map(&tmV);
    prefetch_map(&tmC);
    prefetch_map(&tmP);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(AT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  const int n_my = ((int)blockIdx.x < p.items) ? (p.items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  auto item_len = [&](int i) {  // valid keys of this block's item i
    return p.seq_lens ? min(max(p.seq_lens[((int)blockIdx.x + i * (int)gridDim.x) / p.heads], 1), p.S) : p.S;
  };

  if (warp == 0 && !p.starve && elect_one()) {
    // ------------------------------- TMA producer -------------------------------
    bool ok = true;
    int issued = 0;
    for (int i = 0; i < n_my && ok; i++) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int zo = w / p.heads, zi = w - zo * p.heads;
      const uint32_t s = (uint32_t)i & 1, round = (uint32_t)i >> 1;
      if (!mbar_wait(smem_u32(&empty_bar[s]), (round & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      const uint32_t fb = smem_u32(&full_bar[s]);
      mbar_expect_tx(fb, AB_STAGE_BYTES);
      const uint32_t base = smem_u32(smem + (size_t)s * AB_STAGE_BYTES);
      const int row0 = p.cu ? p.cu[zo] : 0, zseq = p.cu ? 0 : zo;
      int c[4];
      c[0] = 0; c[p.q_perm[0]] = row0; c[p.q_perm[1]] = zi; c[p.q_perm[2]] = zseq;
      tma_load_4d(base, &tmQ, fb, c[0], c[1], c[2], c[3]);
      c[0] = 0; c[p.k_perm[0]] = row0; c[p.k_perm[1]] = zi; c[p.k_perm[2]] = zseq;
      tma_load_4d(base + AT_TILE_BYTES, &tmK, fb, c[0], c[1], c[2], c[3]);
      c[0] = 0; c[p.v_perm[0]] = row0; c[p.v_perm[1]] = zi; c[p.v_perm[2]] = zseq;
      tma_load_4d(base + 2 * AT_TILE_BYTES, &tmV, fb, c[0], c[1], c[2], c[3]);
      c[0] = 0; c[p.c_perm[0]] = row0; c[p.c_perm[1]] = zi; c[p.c_perm[2]] = zseq;
      tma_load_4d(base + 3 * AT_TILE_BYTES, &tmC, fb, c[0], c[1], c[2], c[3]);
      // P: two tiles of 64 keys, each 128 query rows of 128 bytes
      c[p.p_perm[0]] = 0; c[p.p_perm[1]] = zi; c[p.p_perm[2]] = zo;
      c[0] = 0;
      tma_load_4d(base + 4 * AT_TILE_BYTES, &tmP, fb, c[0], c[1], c[2], c[3]);
      c[0] = 64;
      tma_load_4d(base + 5 * AT_TILE_BYTES, &tmP, fb, c[0], c[1], c[2], c[3]);
      issued = i + 1;
    }
    if (!ok || *abort_flag) {
      const int n = issued < 2 ? issued : 2;
      for (int k = 0; k < n; k++) {
        const int j = issued - 1 - k;
        const uint32_t fb = smem_u32(&full_bar[j & 1]);
        const long long t0 = now_cycles();
        while (!mbar_try_wait(fb, (uint32_t)(j >> 1) & 1) && now_cycles() - t0 < 200000000ll) {}
      }
    }
  } else if (warp == 1 && elect_one()) {
    // ------------------------------- MMA issuer -------------------------------
    bool ok = true;
    const uint32_t hi = (uint32_t)(make_smem_desc(0, 16) >> 32);
    const uint32_t lbo_k = (uint32_t)make_smem_desc(0, 16);            // k-contiguous operand
    const uint32_t lbo_mn1 = (uint32_t)make_smem_desc(0, 8192);        // rows = k, one 64-wide m/n block
    const uint32_t lbo_mn2 = (uint32_t)make_smem_desc(0, AT_TILE_BYTES);  // two 64-wide blocks 16 KB apart
    auto addr16 = [](uint32_t a) { return (a & 0x3FFFFu) >> 4; };
    auto mma_k128 = [&](uint32_t d_tmem, uint32_t a_lo, uint32_t a_kb, uint32_t a_ks, uint32_t b_lo,
                        uint32_t b_kb, uint32_t b_ks, uint32_t idesc) {  // contraction over 128 = 2 x 4 x 16
      uint32_t accum = 0;
#pragma unroll
      for (int kb = 0; kb < 2; kb++)
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const uint64_t ad = ((uint64_t)hi << 32) | (a_lo + kb * a_kb + k * a_ks);
          const uint64_t bd = ((uint64_t)hi << 32) | (b_lo + kb * b_kb + k * b_ks);
          tc_mma(d_tmem, ad, bd, idesc, accum);
          accum = 1;
        }
    };
    constexpr uint32_t KS_K = UMMA_K * 2 / 16;      // 16 k values of a k-contiguous tile, in 16-byte units
    constexpr uint32_t KS_MN = UMMA_K * 128 / 16;   // 16 k rows of a row-is-k tile
    constexpr uint32_t KB_MN = 8192 / 16;           // 64 k rows
    constexpr uint32_t KB_K = AT_TILE_BYTES / 16;   // next 64-wide k block of a two-tile operand
    auto second_products = [&](int j) {  // dQ = dS K and dK = dS^T Q of item j
      const uint32_t g = (uint32_t)j & 1;
      const uint32_t base = smem_u32(smem + (size_t)g * AB_STAGE_BYTES);
      const uint32_t ds = addr16(base + 4 * AT_TILE_BYTES);
      const uint32_t acc = tmem_base + g * AB_GROUP_COLS;
      mma_k128(acc, lbo_k | ds, KB_K, KS_K, lbo_mn1 | addr16(base + AT_TILE_BYTES), KB_MN, KS_MN, p.idesc_dq);
      mma_k128(acc + 64, lbo_mn2 | ds, KB_MN, KS_MN, lbo_mn1 | addr16(base), KB_MN, KS_MN, p.idesc_dk);
      tc_commit(smem_u32(&gfull_bar[g]));
      tc_commit(smem_u32(&empty_bar[g]));
    };
    uint32_t cleaned = 0;  // parity of every stage's clean barrier
    for (int i = 0; i < n_my && ok; i++) {
      const uint32_t g = (uint32_t)i & 1, use = (uint32_t)i >> 1;
      const bool edge = p.cu && item_len(i) < 128;
      if (!mbar_wait(smem_u32(edge ? &clean_bar[g] : &full_bar[g]), edge ? (cleaned >> g) & 1 : use & 1, abort_flag, p.status)) {
        ok = false;
        break;
      }
      if (edge) cleaned ^= 1u << g;
      if (!mbar_wait(smem_u32(&accfree_bar[g]), (use & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      const uint32_t base = smem_u32(smem + (size_t)g * AB_STAGE_BYTES);
      const uint32_t acc = tmem_base + g * AB_GROUP_COLS;
      const uint32_t dc = addr16(base + 3 * AT_TILE_BYTES);
      // dV = P^T dC: both operands with rows = query index = k
      mma_k128(acc + 128, lbo_mn2 | addr16(base + 4 * AT_TILE_BYTES), KB_MN, KS_MN, lbo_mn1 | dc, KB_MN, KS_MN,
               p.idesc_dv);
      // dP = dC V^T: both operands k-contiguous, contraction over the head width
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const uint64_t ad = ((uint64_t)hi << 32) | ((lbo_k | dc) + k * KS_K);
        const uint64_t bd = ((uint64_t)hi << 32) | ((lbo_k | addr16(base + 2 * AT_TILE_BYTES)) + k * KS_K);
        tc_mma(acc, ad, bd, p.idesc_dp, k > 0 ? 1u : 0u);
      }
      tc_commit(smem_u32(&dpfull_bar[g]));
      if (i > 0) {
        const uint32_t g1 = (uint32_t)(i - 1) & 1, use1 = (uint32_t)(i - 1) >> 1;
        if (!mbar_wait(smem_u32(&dsready_bar[g1]), use1 & 1, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        second_products(i - 1);
      }
    }
    if (ok && n_my > 0) {
      const uint32_t g1 = (uint32_t)(n_my - 1) & 1, use1 = (uint32_t)(n_my - 1) >> 1;
      if (mbar_wait(smem_u32(&dsready_bar[g1]), use1 & 1, abort_flag, p.status)) {
        tc_fence_after();
        second_products(n_my - 1);
      } else {
        ok = false;
      }
    }
    if (!ok || *abort_flag) {
      tc_commit(smem_u32(&dpfull_bar[0]));
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (warp >= 2 + NUM_EPI_WARPS) {
    // ------------------------------- clearing of rows beyond the sequence -------------------------------
    for (int i = 0; i < n_my && p.cu; i++) {
      const int len = item_len(i);
      const uint32_t s = (uint32_t)i & 1;
      if (!mbar_wait(smem_u32(&full_bar[s]), (i >> 1) & 1, abort_flag, p.status)) break;
      if (len < 128) {
        for (int t = 0; t < 4; t++)  // Q, K, V, dC
          clear_tile_rows(smem + (size_t)s * AB_STAGE_BYTES + t * AT_TILE_BYTES, len, 128, threadIdx.x - NUM_THREADS);
        clear_done(smem_u32(&clean_bar[s]), lane);
      }
      if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }
  } else if (warp >= 2) {
    // ------------------------------- softmax-backward groups -------------------------------
    const int q = warp & 3;
    const int g = (warp - 2) >> 2;
    uint8_t* stg = staging + (size_t)(warp - 2) * AT_STAGING;
    const int r = q * 32 + lane;
    bool ok = true;
    for (int i = g; i < n_my && ok; i += 2) {
      const int w = (int)blockIdx.x + i * (int)gridDim.x;
      const int zo = w / p.heads, zi = w - zo * p.heads;
      const uint32_t use = (uint32_t)i >> 1;
      if (!mbar_wait(smem_u32(&dpfull_bar[g]), use & 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
      float2 v[4][16];  // row r of dP
      const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)g * AB_GROUP_COLS;
#pragma unroll
      for (int c = 0; c < 4; c++) tc_ld32(trow + c * 32, v[c]);
      // row r of P (and then of dS): two 128-byte halves, 16-byte pieces permuted by r mod 8
      uint8_t* prow = smem + (size_t)g * AB_STAGE_BYTES + 4 * AT_TILE_BYTES + r * 128;
      float2 dl[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        dl[c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const uint4 pk = *reinterpret_cast<const uint4*>(prow + (c >> 1) * AT_TILE_BYTES +
                                                           ((((c & 1) * 4 + j) ^ (r & 7)) << 4));
          dl[c] = __ffma2_rn(v[c][4 * j], bf162_to_f2(pk.x), dl[c]);
          dl[c] = __ffma2_rn(v[c][4 * j + 1], bf162_to_f2(pk.y), dl[c]);
          dl[c] = __ffma2_rn(v[c][4 * j + 2], bf162_to_f2(pk.z), dl[c]);
          dl[c] = __ffma2_rn(v[c][4 * j + 3], bf162_to_f2(pk.w), dl[c]);
        }
      }
      const float delta = ((dl[0].x + dl[0].y) + (dl[1].x + dl[1].y)) + ((dl[2].x + dl[2].y) + (dl[3].x + dl[3].y));
      const float2 nd = splat2(-delta), sc2 = splat2(p.scale);
#pragma unroll
      for (int c = 0; c < 4; c++) {
#pragma unroll
        for (int j = 0; j < 4; j++) {
          uint8_t* piece = prow + (c >> 1) * AT_TILE_BYTES + ((((c & 1) * 4 + j) ^ (r & 7)) << 4);
          const uint4 pk = *reinterpret_cast<const uint4*>(piece);
          const uint32_t pw[4] = {pk.x, pk.y, pk.z, pk.w};
          uint4 out;
          __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const float2 t = __fmul2_rn(__fadd2_rn(v[c][4 * j + e], nd), sc2);
            h[e] = __float22bfloat162_rn(__fmul2_rn(t, bf162_to_f2(pw[e])));
          }
          *reinterpret_cast<uint4*>(piece) = out;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&dsready_bar[g]));
      const int rlim = p.cu ? item_len(i) : p.S;  // rows of the item that exist
      bf16* gq = p.dQKV + (p.cu ? p.cu[zo] * p.g_ld : zo * p.g_bo) + zi * 64;
      // dV (complete since dP was): key r, 64 columns
      tc_ld32(trow + 128, v[0]);
      tc_ld32(trow + 160, v[1]);
      // (32-byte row stores straight from registers were slower here, 58 against 54 us: three 128-byte pieces per row)
      stage_store_bf16(stg, lane, v[0], gq + 2 * p.H, p.g_ld, q * 32, 0, rlim, 64, p.vec_ok);
      stage_store_bf16(stg, lane, v[1], gq + 2 * p.H, p.g_ld, q * 32, 32, rlim, 64, p.vec_ok);
      if (!mbar_wait(smem_u32(&gfull_bar[g]), use & 1, abort_flag, p.status)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 4; c++) tc_ld32(trow + c * 32, v[c]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&accfree_bar[g]));
      stage_store_bf16(stg, lane, v[0], gq, p.g_ld, q * 32, 0, rlim, 64, p.vec_ok);
      stage_store_bf16(stg, lane, v[1], gq, p.g_ld, q * 32, 32, rlim, 64, p.vec_ok);
      stage_store_bf16(stg, lane, v[2], gq + p.H, p.g_ld, q * 32, 0, rlim, 64, p.vec_ok);
      stage_store_bf16(stg, lane, v[3], gq + p.H, p.g_ld, q * 32, 32, rlim, 64, p.vec_ok);
    }
    if (p.cu) zero_tail_rows(p.dQKV, p.g_ld, p.g_ld, p.rows);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AT_TMEM_COLS)
                 : "memory");
  }
}

// ---- backward for rows of 129..512 keys -----------------------------------------------------------
// The probabilities are formed again from the scores and the forward's row sums (lse), so they never
// reach memory: with P, dP and dS as [S, S] matrices in HBM the backward of a layer of 16 x 16 heads x
// 512 keys took 184 us in four batched products and a softmax pass.
//   P = 2^(scale log2e S - lse),  dS = P o (dP - delta) scale,  delta = rowsum(dC o C)
// Two kernels of the same form.  kQ = false: an item is (sequence, head, tile of 128 keys), the loop
// runs over query tiles and accumulates dV += P^T dC and dK += dS^T Q.  kQ = true: an item is a tile of
// 128 queries, the loop runs over key tiles and accumulates dQ += dS K.  The second forms S and dP once
// more (2 of 7 products) and in return needs no sums across CTAs: same bits on every run.
// The rows of dS sum to zero: the key bias' gradient is nothing but such sums, and in dQ they multiply the keys'
// common part.  With delta from the context, which was rounded to bf16 (and so were the probabilities it was formed
// from), they do not (the first update of a BERT-Large layer's projection bias was off by 0.165 of its mean, 0.15
// allowed).  So kQ = true runs first, adds up what is left, rest = rowsum(P o (dP - delta)), and beside dS K
// accumulates P K: dQ = dS K - scale rest P K is the product with the corrected dS.  It leaves rest (by half rows)
// for kQ = false, which adds it to delta.
//   warp 0: TMA producer (the item's two fixed tiles, a ring of three pairs of loop tiles)
//   warp 1: one thread issues S and dP of a pair, then the accumulating products of the pair before
//   warps 2-9: two warps per TMEM lane quarter, 64 columns each; a thread owns half a query row.
//   warps 10, 11: clear the rows of the tiles that lie beyond the sequence
// Tensor memory: S 128 columns, dP 128, accumulators 2 x 64.  Bound by the serial chain of a pair
// (products, tensor-memory reads, exponentials, P and dS to shared memory): the products of the next
// pair run while this one is worked on.
constexpr int BL_RING = 3;
constexpr uint32_t BL_ACC_COL = 256;

struct AttnBwdLongParams {
  int S, heads, items;
  float scale;
  const int* seq_lens;
  const int* cu;
  const int* rows;
  const int* order;
  const float* lse;
  float* delta;       // [3][heads][ld]: delta, then the two halves' corrections
  long long ld;       // rows of one head in lse and delta
  bf16* dQKV;
  long long g_ld, H;
  int q_perm[3], k_perm[3], v_perm[3], c_perm[3];
  long long wait_limit;
  int starve;
  int* status;
  uint32_t idesc_s, idesc_kv, idesc_q;
};

template <bool kQ>
__global__ void __launch_bounds__(NUM_THREADS + 32 * CLEAR_WARPS, 1)
attn_bwd_long_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmC,
                     const AttnBwdLongParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // fixed tiles: K, V of the item (kQ: Q, dC); ring stage: Q, dC of a query tile (kQ: K, V of a key tile)
  uint8_t* ring_smem = smem + 2 * AT_TILE_BYTES;
  uint8_t* p_smem = ring_smem + BL_RING * 2 * AT_TILE_BYTES;   // P
  uint8_t* ds_smem = p_smem + 2 * AT_TILE_BYTES;               // dS
  float* xch = (float*)(ds_smem + 2 * AT_TILE_BYTES);          // kQ: [2][NUM_EPI_WARPS][32] sums of half rows
  volatile int* xflag = (volatile int*)(xch + 2 * NUM_EPI_WARPS * 32);
  uint64_t* bars = (uint64_t*)(xflag + NUM_EPI_WARPS);
  uint64_t* rfull_bar = bars;                    // [BL_RING]
  uint64_t* rempty_bar = bars + BL_RING;         // [BL_RING]
  uint64_t* misc = bars + 2 * BL_RING;
  const uint32_t ffull = smem_u32(&misc[0]), fempty = smem_u32(&misc[1]);    // fixed tiles
  const uint32_t sfull = smem_u32(&misc[2]), sempty = smem_u32(&misc[3]);    // S and dP of a pair
  const uint32_t pready = smem_u32(&misc[4]), pfree = smem_u32(&misc[5]);    // P and dS in shared memory
  const uint32_t accfull = smem_u32(&misc[6]), accempty = smem_u32(&misc[7]);
  // the rows of these tiles beyond the sequence are zero: fixed tiles, [BL_RING]
  const uint32_t fclean = smem_u32(&misc[8]), rclean0 = smem_u32(&misc[9]);
  uint32_t* tmem_slot = (uint32_t*)(misc + 9 + BL_RING);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < BL_RING; s++) {
      mbar_init(smem_u32(&rfull_bar[s]), 1);
      mbar_init(smem_u32(&rempty_bar[s]), 1 + CLEAR_WARPS);
      mbar_init(rclean0 + 8 * s, CLEAR_WARPS);
    }
    mbar_init(ffull, 1); mbar_init(fempty, 1 + CLEAR_WARPS); mbar_init(fclean, CLEAR_WARPS);
    mbar_init(sfull, 1); mbar_init(sempty, NUM_EPI_WARPS);
    mbar_init(pready, NUM_EPI_WARPS); mbar_init(pfree, 1);
    mbar_init(accfull, 1); mbar_init(accempty, NUM_EPI_WARPS);
    for (int i = 0; i < NUM_EPI_WARPS; i++) xflag[i] = 0;
    *abort_flag = 0;
    *reinterpret_cast<volatile long long*>(abort_flag + 1) = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && elect_one()) {
    prefetch_map(&tmQ);
    prefetch_map(&tmK);
    prefetch_map(&tmV);
    prefetch_map(&tmC);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(AT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();
  // items as in the forward kernel: packed batches list the tiles that exist, longest sequences first
  const int nt = (p.S + 127) >> 7, nzh = p.items / nt;
  const int n_items = p.cu ? p.rows[2] * p.heads : p.items;
  auto decode = [&](int w, int& zo, int& zi, int& tile) {
    if (p.cu) {
      const int e = w / p.heads;
      zi = w - e * p.heads;
      zo = p.order[e] >> 3;
      tile = p.order[e] & 7;
    } else {
      tile = w / nzh;
      zo = (w - tile * nzh) / p.heads;
      zi = (w - tile * nzh) - zo * p.heads;
    }
  };
  auto item_len = [&](int zo) {
    int len = p.cu ? p.seq_lens[zo] : p.S;
    return min(max(len, 1), p.S);
  };
  auto row_base = [&](int zo) { return p.cu ? p.cu[zo] : zo * p.S; };

  if (warp == 0 && !p.starve && elect_one()) {
    // ------------------------------- TMA producer -------------------------------
    bool ok = true;
    uint32_t rt = 0, ni = 0;
    auto load = [&](const CUtensorMap* map, const int (&perm)[3], uint32_t dst, uint32_t bar, int row, int zi) {
      int c[4] = {0, 0, 0, 0};
      c[perm[0]] = row; c[perm[1]] = zi;
      tma_load_4d(dst, map, bar, c[0], c[1], c[2], c[3]);
    };
    for (int w = (int)blockIdx.x; w < n_items && ok; w += (int)gridDim.x) {
      int zo, zi, tile;
      decode(w, zo, zi, tile);
      const int len = item_len(zo), row0 = row_base(zo);
      const int n = (len + 127) >> 7;
      if (!mbar_wait(fempty, (ni & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
      ni++;
      mbar_expect_tx(ffull, 2 * AT_TILE_BYTES);
      const uint32_t f0 = smem_u32(smem);
      load(kQ ? &tmQ : &tmK, kQ ? p.q_perm : p.k_perm, f0, ffull, row0 + tile * 128, zi);
      load(kQ ? &tmC : &tmV, kQ ? p.c_perm : p.v_perm, f0 + AT_TILE_BYTES, ffull, row0 + tile * 128, zi);
      for (int t = 0; t < n; t++, rt++) {
        const uint32_t slot = rt % BL_RING, round = rt / BL_RING;
        if (!mbar_wait(smem_u32(&rempty_bar[slot]), (round & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        const uint32_t fb = smem_u32(&rfull_bar[slot]);
        mbar_expect_tx(fb, 2 * AT_TILE_BYTES);
        const uint32_t r0 = smem_u32(ring_smem + (size_t)slot * 2 * AT_TILE_BYTES);
        load(kQ ? &tmK : &tmQ, kQ ? p.k_perm : p.q_perm, r0, fb, row0 + t * 128, zi);
        load(kQ ? &tmV : &tmC, kQ ? p.v_perm : p.c_perm, r0 + AT_TILE_BYTES, fb, row0 + t * 128, zi);
      }
    }
    if (!ok || *abort_flag) {  // give the copies in flight time to land before the CTA leaves
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 4000000ll) {}
    }
  } else if (warp == 1 && elect_one()) {
    // ------------------------------- MMA issuer -------------------------------
    bool ok = true;
    const uint32_t hi = (uint32_t)(make_smem_desc(0, 16) >> 32);
    const uint32_t lbo_k = (uint32_t)make_smem_desc(0, 16);               // k-contiguous operand
    const uint32_t lbo_mn1 = (uint32_t)make_smem_desc(0, 8192);           // rows = k, one 64-wide m/n block
    const uint32_t lbo_mn2 = (uint32_t)make_smem_desc(0, AT_TILE_BYTES);  // two 64-wide blocks 16 KB apart
    auto addr16 = [](uint32_t a) { return (a & 0x3FFFFu) >> 4; };
    constexpr uint32_t KS_K = UMMA_K * 2 / 16, KS_MN = UMMA_K * 128 / 16;
    constexpr uint32_t KB_MN = 8192 / 16, KB_K = AT_TILE_BYTES / 16;
    auto mma_k128 = [&](uint32_t d_tmem, uint32_t a_lo, uint32_t a_kb, uint32_t a_ks, uint32_t b_lo, uint32_t idesc,
                        bool first) {  // contraction over 128 = 2 x 4 x 16, B with rows = k
#pragma unroll
      for (int kb = 0; kb < 2; kb++)
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const uint64_t ad = ((uint64_t)hi << 32) | (a_lo + kb * a_kb + k * a_ks);
          const uint64_t bd = ((uint64_t)hi << 32) | (b_lo + kb * KB_MN + k * KS_MN);
          tc_mma(d_tmem, ad, bd, idesc, (first && kb == 0 && k == 0) ? 0u : 1u);
        }
    };
    auto mma_k64 = [&](uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr) {  // both operands k-contiguous
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const uint64_t ad = ((uint64_t)hi << 32) | ((lbo_k | addr16(a_addr)) + k * KS_K);
        const uint64_t bd = ((uint64_t)hi << 32) | ((lbo_k | addr16(b_addr)) + k * KS_K);
        tc_mma(d_tmem, ad, bd, p.idesc_s, k > 0 ? 1u : 0u);
      }
    };
    const uint32_t f0 = smem_u32(smem), pa = addr16(smem_u32(p_smem)), da = addr16(smem_u32(ds_smem));
    uint32_t rt = 0, np = 0, ni = 0;  // score pairs (= ring tiles), accumulated pairs, items
    uint32_t cleaned = 0;             // parity of every slot's clean barrier, the fixed tiles' behind them
    for (int w = (int)blockIdx.x; w < n_items && ok; w += (int)gridDim.x) {
      int zo, zi, tile;
      decode(w, zo, zi, tile);
      const int len = item_len(zo);
      const int n = (len + 127) >> 7;
      auto landed = [&](uint32_t full, uint32_t parity, uint32_t clean, uint32_t bit, bool edge) -> bool {
        if (!mbar_wait(edge ? clean : full, edge ? (cleaned >> bit) & 1 : parity, abort_flag, p.status)) return false;
        if (edge) cleaned ^= 1u << bit;
        return true;
      };
      if (!landed(ffull, ni & 1, fclean, BL_RING, (tile + 1) * 128 > len)) { ok = false; break; }
      auto accumulate = [&](int t) -> bool {  // the accumulating products of pair t of this item
        if (!mbar_wait(pready, np & 1, abort_flag, p.status)) return false;
        if (t == 0 && !mbar_wait(accempty, (ni & 1) ^ 1, abort_flag, p.status)) return false;
        tc_fence_after();
        const uint32_t slot = np % BL_RING;
        const uint32_t r0 = smem_u32(ring_smem + (size_t)slot * 2 * AT_TILE_BYTES);
        const uint32_t acc = tmem_base + BL_ACC_COL;
        if (kQ) {
          mma_k128(acc, lbo_k | da, KB_K, KS_K, lbo_mn1 | addr16(r0), p.idesc_q, t == 0);       // dQ += dS K
          mma_k128(acc + 64, lbo_k | pa, KB_K, KS_K, lbo_mn1 | addr16(r0), p.idesc_q, t == 0);  // and P K
        } else {
          mma_k128(acc, lbo_mn2 | pa, KB_MN, KS_MN, lbo_mn1 | addr16(r0 + AT_TILE_BYTES), p.idesc_kv, t == 0);  // dV += P^T dC
          mma_k128(acc + 64, lbo_mn2 | da, KB_MN, KS_MN, lbo_mn1 | addr16(r0), p.idesc_kv, t == 0);             // dK += dS^T Q
        }
        tc_commit(pfree);
        tc_commit(smem_u32(&rempty_bar[slot]));
        np++;
        return true;
      };
      for (int t = 0; t < n && ok; t++, rt++) {
        const uint32_t slot = rt % BL_RING, round = rt / BL_RING;
        if (!landed(smem_u32(&rfull_bar[slot]), round & 1, rclean0 + 8 * slot, slot, (t + 1) * 128 > len)) { ok = false; break; }
        if (!mbar_wait(sempty, (rt & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t r0 = smem_u32(ring_smem + (size_t)slot * 2 * AT_TILE_BYTES);
        mma_k64(tmem_base, kQ ? f0 : r0, kQ ? r0 : f0);                                   // S = Q K^T
        mma_k64(tmem_base + 128, (kQ ? f0 : r0) + AT_TILE_BYTES, (kQ ? r0 : f0) + AT_TILE_BYTES);  // dP = dC V^T
        tc_commit(sfull);
        if (t > 0) ok = accumulate(t - 1);
      }
      if (ok) ok = accumulate(n - 1);
      if (ok) {
        tc_commit(accfull);
        tc_commit(fempty);
      }
      ni++;
    }
    if (!ok || *abort_flag) {
      // make sure no MMA is still writing tensor memory before it is freed
      tc_commit(sfull);
      const long long t0 = now_cycles();
      while (now_cycles() - t0 < 2000000ll) {}
    }
  } else if (warp >= 2 + NUM_EPI_WARPS) {
    // ------------------------------- clearing of rows beyond the sequence -------------------------------
    bool ok = true;
    uint32_t rt = 0, ni = 0;
    auto clear = [&](uint32_t full, uint32_t parity, uint32_t clean, uint32_t empty, uint8_t* tiles, int r0) -> bool {
      if (!mbar_wait(full, parity, abort_flag, p.status)) return false;
      if (r0 < 128) {
        for (int t = 0; t < 2; t++) clear_tile_rows(tiles + t * AT_TILE_BYTES, r0, 128, threadIdx.x - NUM_THREADS);
        clear_done(clean, lane);
      }
      if (lane == 0) mbar_arrive(empty);
      return true;
    };
    for (int w = (int)blockIdx.x; w < n_items && ok; w += (int)gridDim.x) {
      int zo, zi, tile;
      decode(w, zo, zi, tile);
      const int len = item_len(zo);
      const int n = (len + 127) >> 7;
      ok = clear(ffull, ni & 1, fclean, fempty, smem, len - tile * 128);
      ni++;
      for (int t = 0; t < n && ok; t++, rt++) {
        const uint32_t slot = rt % BL_RING;
        ok = clear(smem_u32(&rfull_bar[slot]), (rt / BL_RING) & 1, rclean0 + 8 * slot, smem_u32(&rempty_bar[slot]),
                   ring_smem + (size_t)slot * 2 * AT_TILE_BYTES, len - t * 128);
      }
    }
  } else if (warp >= 2) {
    // ------------------------------- softmax-backward warps -------------------------------
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int r = q * 32 + lane;
    const float sl2 = p.scale * 1.4426950408889634f;
    const float2 k2 = splat2(sl2), sc2 = splat2(p.scale);
    const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16);
    bool ok = true;
    uint32_t sp = 0, ni = 0;
    uint8_t* prow = p_smem + half * AT_TILE_BYTES + r * 128;
    uint8_t* drow = ds_smem + half * AT_TILE_BYTES + r * 128;
    for (int w = (int)blockIdx.x; w < n_items && ok; w += (int)gridDim.x) {
      int zo, zi, tile;
      decode(w, zo, zi, tile);
      const int len = item_len(zo);
      const int n = (len + 127) >> 7;
      const long long row0 = row_base(zo);
      float2 rest = make_float2(0.f, 0.f);
      for (int t = 0; t < n && ok; t++) {
        const int qrow = (kQ ? tile : t) * 128 + r, key0 = (kQ ? t : tile) * 128 + half * 64;
        // a row beyond the sequence gets probability 2^-inf = 0 everywhere
        float nl = -INFINITY, nd = 0.f;
        if (qrow < len) {
          nl = -p.lse[zi * p.ld + row0 + qrow];
          const float* dl = p.delta + zi * p.ld + row0 + qrow;
          nd = kQ ? -dl[0] : -(dl[0] + (dl[p.heads * p.ld] + dl[2 * p.heads * p.ld]));
        }
        const float2 nl2 = splat2(nl), nd2 = splat2(nd);
        if (!mbar_wait(sfull, sp & 1, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        uint32_t s0[32], s1[32], d0[32], d1[32];
        tc_ld32_issue(trow + half * 64, s0);
        tc_ld32_issue(trow + half * 64 + 32, s1);
        tc_ld32_issue(trow + 128 + half * 64, d0);
        tc_ld32_issue(trow + 128 + half * 64 + 32, d1);
        tc_ld32_wait(s0);
        tc_ld32_wait(s1);
        tc_ld32_wait(d0);
        tc_ld32_wait(d1);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sempty);
        // P and dS as bf16 pairs, kept in the registers of S and dP
        auto work = [&](uint32_t (&s)[32], uint32_t (&d)[32], int k0) {
          const bool edge = k0 + 32 > len;
#pragma unroll
          for (int j = 0; j < 16; j++) {
            const float2 a = __ffma2_rn(make_float2(__uint_as_float(s[2 * j]), __uint_as_float(s[2 * j + 1])), k2, nl2);
            float2 pr = make_float2(fast_exp2(a.x), fast_exp2(a.y));
            if (edge) {
              if (k0 + 2 * j >= len) pr.x = 0.f;
              if (k0 + 2 * j + 1 >= len) pr.y = 0.f;
            }
            const float2 dp = __fadd2_rn(make_float2(__uint_as_float(d[2 * j]), __uint_as_float(d[2 * j + 1])), nd2);
            const float2 pd = __fmul2_rn(dp, pr);
            if (kQ) rest = __fadd2_rn(rest, pd);
            const __nv_bfloat162 ds = __float22bfloat162_rn(__fmul2_rn(pd, sc2));
            const __nv_bfloat162 pb = __float22bfloat162_rn(pr);
            s[j] = *reinterpret_cast<const uint32_t*>(&pb);
            d[j] = *reinterpret_cast<const uint32_t*>(&ds);
          }
        };
        work(s0, d0, key0);
        work(s1, d1, key0 + 32);
        // the accumulating products of the pair before have read P and dS
        if (!mbar_wait(pfree, (sp & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
        sp++;
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const int u0 = (c ^ (r & 7)) << 4, u1 = ((4 + c) ^ (r & 7)) << 4;
          *reinterpret_cast<uint4*>(prow + u0) = make_uint4(s0[4 * c], s0[4 * c + 1], s0[4 * c + 2], s0[4 * c + 3]);
          *reinterpret_cast<uint4*>(prow + u1) = make_uint4(s1[4 * c], s1[4 * c + 1], s1[4 * c + 2], s1[4 * c + 3]);
          *reinterpret_cast<uint4*>(drow + u0) = make_uint4(d0[4 * c], d0[4 * c + 1], d0[4 * c + 2], d0[4 * c + 3]);
          *reinterpret_cast<uint4*>(drow + u1) = make_uint4(d1[4 * c], d1[4 * c + 1], d1[4 * c + 2], d1[4 * c + 3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(pready);
      }
      if (!ok) break;
      float total = rest.x + rest.y;
      if (kQ) {  // the row's other half
        if (tile * 128 + r < len) p.delta[(1 + half) * p.heads * p.ld + zi * p.ld + row0 + tile * 128 + r] = total;
        float* x = xch + (ni & 1) * NUM_EPI_WARPS * 32;  // a partner may still read the item before
        x[(half * 4 + q) * 32 + lane] = total;
        if (!pair_sync(xflag, half * 4 + q, (half ^ 1) * 4 + q, (int)ni + 1, lane, abort_flag, p.status)) { ok = false; break; }
        total += x[((half ^ 1) * 4 + q) * 32 + lane];
      }
      // the item's gradients: row r of its tile
      if (!mbar_wait(accfull, ni & 1, abort_flag, p.status)) { ok = false; break; }
      ni++;
      tc_fence_after();
      float2 v0[16], v1[16];
      const uint32_t acol = BL_ACC_COL + (kQ ? half * 32 : half * 64);
      tc_ld32(trow + acol, v0);
      tc_ld32(trow + acol + (kQ ? 64 : 32), v1);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(accempty);
      if (tile * 128 + r < len) {
        bf16* g = p.dQKV + (row0 + tile * 128 + r) * p.g_ld + zi * 64;
        if (kQ) {
          const float2 off = splat2(-p.scale * total);
#pragma unroll
          for (int j = 0; j < 16; j++) v0[j] = __ffma2_rn(v1[j], off, v0[j]);
          store_row32_bf16(g + half * 32, v0);
        } else {
          g += half ? p.H : 2 * p.H;  // the first accumulator is dV, the second dK
          store_row32_bf16(g, v0);
          store_row32_bf16(g + 32, v1);
        }
      }
    }
    if (kQ && p.cu) zero_tail_rows(p.dQKV, p.g_ld, p.g_ld, p.rows);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AT_TMEM_COLS)
                 : "memory");
  }
}

// delta[h][row] = sum over the head's 64 columns of dC o C.  Eight lanes share a head's row.
__global__ void __launch_bounds__(256)
attn_delta_kernel(const bf16* __restrict__ c, const bf16* __restrict__ dc, float* __restrict__ delta, int rows, int heads,
                  long long ld, const int* __restrict__ rows_dev) {
  pdl_begin();
  if (rows_dev) rows = min(rows, rows_dev[0]);
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  const long long unit = i >> 3;  // (row, head)
  const long long row = unit / heads;
  const int h = (int)(unit - row * heads);
  float s = 0.f;
  if (row < rows) {
    float a[8], b[8];
    VecT<bf16>::load(c + unit * 64 + (i & 7) * 8, a);
    VecT<bf16>::load(dc + unit * 64 + (i & 7) * 8, b);
#pragma unroll
    for (int e = 0; e < 8; e++) s = fmaf(a[e], b[e], s);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((i & 7) == 0 && row < rows) delta[h * ld + row] = s;
}

}  // namespace

static std::atomic<long long> g_attn_launches{0};
static std::atomic<int> g_attn_starve{0};
void attn_starve_next(int on) { g_attn_starve.store(on ? 1 : 0); }
long long attn_launches() { return g_attn_launches.load(); }

namespace {
// per-device facts and one-time kernel attributes (a process may drive several GPUs)
struct AttnDevice {
  int num_sms = 0, smem_optin = 0;
  bool attr_fwd[2] = {false, false}, attr_rows[2] = {false, false}, attr_long = false;
  bool attr_bwd = false, attr_bwd_kv = false, attr_bwd_q = false;
};
constexpr int kMaxDevices = 64;
AttnDevice g_adev[kMaxDevices];
std::mutex g_adev_mu;
AttnDevice* attn_device(char* err) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    snprintf(err, 256, "attention: no CUDA device");
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_adev_mu);
  AttnDevice& a = g_adev[dev];
  if (a.num_sms == 0) {
    cudaDeviceGetAttribute(&a.num_sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&a.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (a.num_sms <= 0) { snprintf(err, 256, "attention: no CUDA device"); return nullptr; }
  }
  return &a;
}
// opts a kernel in to the large dynamic shared memory size once per device
template <typename K>
int attn_opt_in(K kernel, bool* done, int smem_optin, char* err) {
  std::lock_guard<std::mutex> lock(g_adev_mu);
  if (*done) return 0;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
  if (e != cudaSuccess) { snprintf(err, 256, "attention: cudaFuncSetAttribute: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  *done = true;
  return 0;
}
}  // namespace

int attn_fwd_launch(const void* qkv, void* probs, void* ctx, const int* seq_lens, int B, int S, int A, int d,
                    float scale, int* status, cudaStream_t st, char* err, const int* cu, const int* rows, float* lse,
                    const int* order) {
  // the test hook is used up by this call even if an argument check below rejects it
  const bool starve = g_attn_starve.exchange(0) != 0;
  AttnDevice* adev = attn_device(err);
  if (!adev) return MSLT_ERR_CUDA;
  const int num_sms = adev->num_sms, smem_optin = adev->smem_optin;
  if (d != 64 || S < 1 || S > 512 || B < 1 || A < 1 || !status) {
    snprintf(err, 256, "attention: the fused kernel needs head width 64 and 1 <= S <= 512");
    return MSLT_ERR_ARG;
  }
  const bool long_rows = S > 128;  // several key blocks per row: the two-pass kernel
  const long long H = (long long)A * d;
  AttnParams p;
  memset(&p, 0, sizeof(p));
  p.S = S; p.heads = A; p.items = B * A * (long_rows ? (S + 127) / 128 : 1); p.scale = scale; p.seq_lens = seq_lens;
  p.cu = cu; p.rows = rows; p.order = order;
  p.lse = lse; p.lse_ld = (long long)B * S;
  if ((cu && (!seq_lens || !rows || (long_rows && !order))) || (cu && long_rows && probs) || (lse && (!long_rows || probs))) {
    snprintf(err, 256, "attention: packed rows need lengths and row counts; long packed rows store no probabilities");
    return MSLT_ERR_ARG;
  }
  p.P = (bf16*)probs; p.p_bo = (long long)A * S * S; p.p_bi = (long long)S * S;
  p.C = (bf16*)ctx; p.c_ld = H; p.c_bo = (long long)S * H; p.c_bi = d;
  p.vec_ok_p = (S % 8 == 0 && ((uintptr_t)probs & 15) == 0) ? 1 : 0;
  p.vec_ok_c = (H % 8 == 0 && ((uintptr_t)ctx & 15) == 0) ? 1 : 0;
  p.fast_c = row_fast(ctx, H);
  p.fast_p = (probs != nullptr && S % 32 == 0) ? row_fast(probs, S) : 0;
  p.wait_limit = WAIT_LIMIT_CYCLES;
  p.status = status;
  if (starve) {  // armed by mslt_debug_starve_next_attention
    p.starve = 1;
    p.wait_limit = 40000000ll;  // about 20 ms
  }
  // fp32 accumulate, bf16 x bf16; scores: both operands k-contiguous, N = 128; context: V row-contiguous, N = 64
  p.idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
  p.idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
  const bf16* base = (const bf16*)qkv;
  // packed rows: one long run of rows, a sequence being an offset into it
  const long long mrows = cu ? (long long)B * S : S, mbo = cu ? 0 : (long long)S * 3 * H;
  const int mseqs = cu ? 1 : B;
  MapVal mq, mk, mv;
  int rc = get_map(base, mrows, d, 3 * H, 1, mbo, d, A, mseqs, BM, &mq, err);
  if (rc) return rc;
  rc = get_map(base + H, mrows, d, 3 * H, 1, mbo, d, A, mseqs, BM, &mk, err);
  if (rc) return rc;
  // V: the short kernel reads it as two boxes of 64 keys with the head width contiguous; the long
  // one as one box of 128 key rows, which are the same bytes in shared memory
  if (long_rows) rc = get_map(base + 2 * H, mrows, d, 3 * H, 1, mbo, d, A, mseqs, BM, &mv, err);
  else rc = get_map(base + 2 * H, d, mrows, 1, 3 * H, mbo, d, A, mseqs, 64, &mv, err);
  if (rc) return rc;
  for (int i = 0; i < 3; i++) { p.q_perm[i] = mq.perm[i]; p.k_perm[i] = mk.perm[i]; p.v_perm[i] = mv.perm[i]; }
  if (long_rows && probs == nullptr) {
    const size_t smem_rows = (size_t)(1 + AR_RING + 4) * AT_TILE_BYTES + 2 * AR_WARPS * 32 * 4 + AR_TABLE * 16 + 1024 + 512;
    if ((int)smem_rows > smem_optin) { snprintf(err, 256, "attention: not enough shared memory"); return MSLT_ERR_CUDA; }
    const auto kernel = cu ? attn_fwd_rows_kernel<true> : attn_fwd_rows_kernel<false>;
    rc = attn_opt_in(kernel, &adev->attr_rows[cu != nullptr], smem_optin, err);
    if (rc) return rc;
    launch_pdl(kernel, p.items < num_sms ? p.items : num_sms, AR_THREADS + (cu ? 32 * CLEAR_WARPS : 0), smem_rows, st, mq.map, mk.map, mv.map, p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
    g_attn_launches++;
    return 0;
  }
  if (long_rows) {
    const size_t smem_long = 2 * (size_t)AT_TILE_BYTES + 2 * (size_t)AL_RING * AT_TILE_BYTES + 2 * (size_t)AL_P_BYTES +
                             NUM_EPI_WARPS * AT_STAGING + 1024 + 512;
    if ((int)smem_long > smem_optin) { snprintf(err, 256, "attention: not enough shared memory"); return MSLT_ERR_CUDA; }
    rc = attn_opt_in(attn_fwd_long_kernel, &adev->attr_long, smem_optin, err);
    if (rc) return rc;
    const int grid_long = p.items < num_sms ? p.items : num_sms;
    launch_pdl(attn_fwd_long_kernel, grid_long, AL_THREADS, smem_long, st, mq.map, mk.map, mv.map, p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
    g_attn_launches++;
    return 0;
  }
  const size_t smem_bytes = (size_t)AT_STAGES * AT_STAGE_BYTES + NUM_EPI_WARPS * AT_STAGING + 1024 + 256;
  if ((int)smem_bytes > smem_optin) { snprintf(err, 256, "attention: not enough shared memory"); return MSLT_ERR_CUDA; }
  const auto kernel = cu ? attn_fwd_kernel<true> : attn_fwd_kernel<false>;
  rc = attn_opt_in(kernel, &adev->attr_fwd[cu != nullptr], smem_optin, err);
  if (rc) return rc;
  const int grid = p.items < num_sms ? p.items : num_sms;
  launch_pdl(kernel, grid, NUM_THREADS + (cu ? 32 * CLEAR_WARPS : 0), smem_bytes, st, mq.map, mk.map, mv.map, p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  g_attn_launches++;
  return 0;
}

int attn_bwd_launch(const void* qkv, const void* probs, const void* dctx, void* dqkv, int B, int S, int A, int d,
                    float scale, int* status, cudaStream_t st, char* err, const int* seq_lens, const int* cu,
                    const int* rows) {
  // the test hook is used up by this call even if an argument check below rejects it
  const bool starve = g_attn_starve.exchange(0) != 0;
  AttnDevice* adev = attn_device(err);
  if (!adev) return MSLT_ERR_CUDA;
  const int num_sms = adev->num_sms, smem_optin = adev->smem_optin;
  if (d != 64 || S < 8 || S > 128 || S % 8 || B < 1 || A < 1 || !status || !qkv || !probs || !dctx || !dqkv) {
    snprintf(err, 256, "attention backward: the fused kernel needs head width 64 and S a multiple of 8 in [8, 128]");
    return MSLT_ERR_ARG;
  }
  const long long H = (long long)A * d;
  AttnBwdParams p;
  memset(&p, 0, sizeof(p));
  p.S = S; p.heads = A; p.items = B * A; p.scale = scale;
  p.dQKV = (bf16*)dqkv; p.g_ld = 3 * H; p.g_bo = (long long)S * 3 * H; p.H = H;
  p.vec_ok = ((uintptr_t)dqkv & 15) == 0 ? 1 : 0;
  p.wait_limit = WAIT_LIMIT_CYCLES;
  p.status = status;
  if (starve) {  // armed by mslt_debug_starve_next_attention
    p.starve = 1;
    p.wait_limit = 40000000ll;  // about 20 ms
  }
  // fp32 accumulate, bf16 x bf16, M = 128; bit 15 / 16: A / B operand with rows = k index
  const uint32_t common = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);
  p.idesc_dv = common | (1u << 15) | (1u << 16) | ((uint32_t)(64 >> 3) << 17);
  p.idesc_dp = common | ((uint32_t)(128 >> 3) << 17);
  p.idesc_dq = common | (1u << 16) | ((uint32_t)(64 >> 3) << 17);
  p.idesc_dk = common | (1u << 15) | (1u << 16) | ((uint32_t)(64 >> 3) << 17);
  const bf16* base = (const bf16*)qkv;
  const long long mrows = cu ? (long long)B * S : S;
  const int mseqs = cu ? 1 : B;
  p.seq_lens = seq_lens; p.cu = cu; p.rows = rows;
  MapVal mq, mk, mv, mc, mp;
  int rc = get_map(base, mrows, d, 3 * H, 1, cu ? 0 : (long long)S * 3 * H, d, A, mseqs, BM, &mq, err);
  if (rc) return rc;
  rc = get_map(base + H, mrows, d, 3 * H, 1, cu ? 0 : (long long)S * 3 * H, d, A, mseqs, BM, &mk, err);
  if (rc) return rc;
  rc = get_map(base + 2 * H, mrows, d, 3 * H, 1, cu ? 0 : (long long)S * 3 * H, d, A, mseqs, BM, &mv, err);
  if (rc) return rc;
  rc = get_map(dctx, mrows, d, H, 1, cu ? 0 : (long long)S * H, d, A, mseqs, BM, &mc, err);
  if (rc) return rc;
  rc = get_map(probs, S, S, S, 1, (long long)A * S * S, (long long)S * S, A, B, BM, &mp, err);
  if (rc) return rc;
  for (int i = 0; i < 3; i++) {
    p.q_perm[i] = mq.perm[i]; p.k_perm[i] = mk.perm[i]; p.v_perm[i] = mv.perm[i];
    p.c_perm[i] = mc.perm[i]; p.p_perm[i] = mp.perm[i];
  }
  const size_t smem_bytes = (size_t)2 * AB_STAGE_BYTES + NUM_EPI_WARPS * AT_STAGING + 1024 + 256;
  if ((int)smem_bytes > smem_optin) { snprintf(err, 256, "attention: not enough shared memory"); return MSLT_ERR_CUDA; }
  rc = attn_opt_in(attn_bwd_kernel, &adev->attr_bwd, smem_optin, err);
  if (rc) return rc;
  const int grid = p.items < num_sms ? p.items : num_sms;
  launch_pdl(attn_bwd_kernel, grid, NUM_THREADS + 32 * CLEAR_WARPS, smem_bytes, st, mq.map, mk.map, mv.map, mc.map, mp.map, p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  g_attn_launches++;
  return 0;
}

int attn_bwd_long_launch(const void* qkv, const void* ctx, const void* dctx, const float* lse, float* delta,
                         void* dqkv, int B, int S, int A, float scale, int* status, cudaStream_t st, char* err,
                         const int* seq_lens, const int* cu, const int* rows, const int* order) {
  const bool starve = g_attn_starve.exchange(0) != 0;
  AttnDevice* adev = attn_device(err);
  if (!adev) return MSLT_ERR_CUDA;
  if (S < 1 || S > 512 || B < 1 || A < 1 || !status || !lse || !delta || (seq_lens && !cu) ||
      (cu && (!seq_lens || !rows || !order))) {
    snprintf(err, 256, "attention backward: bad arguments");
    return MSLT_ERR_ARG;
  }
  const long long H = (long long)A * 64, T = (long long)B * S;
  AttnBwdLongParams p;
  memset(&p, 0, sizeof(p));
  p.S = S; p.heads = A; p.items = B * A * ((S + 127) / 128); p.scale = scale;
  p.seq_lens = seq_lens; p.cu = cu; p.rows = rows; p.order = order; p.lse = lse; p.delta = delta; p.ld = T;
  p.dQKV = (bf16*)dqkv; p.g_ld = 3 * H; p.H = H;
  p.wait_limit = starve ? 40000000ll : WAIT_LIMIT_CYCLES;
  p.starve = starve ? 1 : 0;
  p.status = status;
  const uint32_t common = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);
  p.idesc_s = common | ((uint32_t)(128 >> 3) << 17);
  p.idesc_kv = common | (1u << 15) | (1u << 16) | ((uint32_t)(64 >> 3) << 17);
  p.idesc_q = common | (1u << 16) | ((uint32_t)(64 >> 3) << 17);
  const bf16* base = (const bf16*)qkv;
  MapVal mq, mk, mv, mc;
  int rc = get_map(base, T, 64, 3 * H, 1, 0, 64, A, 1, BM, &mq, err);
  if (!rc) rc = get_map(base + H, T, 64, 3 * H, 1, 0, 64, A, 1, BM, &mk, err);
  if (!rc) rc = get_map(base + 2 * H, T, 64, 3 * H, 1, 0, 64, A, 1, BM, &mv, err);
  if (!rc) rc = get_map(dctx, T, 64, H, 1, 0, 64, A, 1, BM, &mc, err);
  if (rc) return rc;
  for (int i = 0; i < 3; i++) {
    p.q_perm[i] = mq.perm[i]; p.k_perm[i] = mk.perm[i]; p.v_perm[i] = mv.perm[i]; p.c_perm[i] = mc.perm[i];
  }
  const size_t smem = (size_t)(2 + 2 * BL_RING + 4) * AT_TILE_BYTES + 2 * NUM_EPI_WARPS * 32 * 4 + 1024 + 512;
  if ((int)smem > adev->smem_optin) { snprintf(err, 256, "attention: not enough shared memory"); return MSLT_ERR_CUDA; }
  rc = attn_opt_in(attn_bwd_long_kernel<false>, &adev->attr_bwd_kv, adev->smem_optin, err);
  if (!rc) rc = attn_opt_in(attn_bwd_long_kernel<true>, &adev->attr_bwd_q, adev->smem_optin, err);
  if (rc) return rc;
  const int grid = p.items < adev->num_sms ? p.items : adev->num_sms;
  launch_pdl(attn_delta_kernel, (unsigned)((T * A * 8 + 255) / 256), 256, 0, st, (const bf16*)ctx, (const bf16*)dctx,
             delta, (int)T, A, T, rows);
  launch_pdl(attn_bwd_long_kernel<true>, grid, NUM_THREADS + 32 * CLEAR_WARPS, smem, st, mq.map, mk.map, mv.map, mc.map, p);
  launch_pdl(attn_bwd_long_kernel<false>, grid, NUM_THREADS + 32 * CLEAR_WARPS, smem, st, mq.map, mk.map, mv.map, mc.map, p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { snprintf(err, 256, "attention: launch failed: %s", cudaGetErrorString(e)); return MSLT_ERR_CUDA; }
  g_attn_launches += 3;
  return 0;
}

}  // namespace mslt
