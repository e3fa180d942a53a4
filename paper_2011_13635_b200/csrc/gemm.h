// Dense contraction with the step's fused epilogue; see mslt_gemm_desc in mslt.h.
//   D[z][m][n] = epilogue(alpha * sum_k A[z](m,k) * B[z](n,k))
// dtype 0: fp32 on the CUDA cores (gemm_f32.cu), or on the tensor cores after a split (gemm_f32x3.cu);
// dtype 1: bf16 on tcgen05 (gemm_tc.cu; gemm_tc_small.cu where the output has few tiles).
#pragma once
#include <cuda_runtime.h>

#include "../../include/mslt.h"

namespace mslt {

// Enqueues the contraction on `st`.  `status` is a device word that a tensor-core kernel ORs an
// error bit into when one of its bounded waits runs out.  Returns 0, or a negative mslt_status
// with a message in `err` (at least 256 bytes).
// rows (dtype 1 only, may be null): device count <= M, or <= K with rows_are_k, of the rows that hold
// anything; work is cut to it (row results beyond it are not written).  b_static: B is written by neither
// of the two kernels before this one in the stream (weights inside a step), so it may be read early.
// parts (one fp32 output of all rows, not accumulated, alpha its only epilogue): the splits of k leave a result each, M * ldd elements after the one before,
// instead of adding to one; in: how many there is room for (kMaxParts are used at most), out: their number.  The caller
// adds them in order.
constexpr int kMaxParts = 8;
int gemm_launch(const mslt_gemm_desc& d, int* status, cudaStream_t st, char* err, const int* rows = nullptr,
                int rows_are_k = 0, bool b_static = false, int* parts = nullptr);

int gemm_f32_launch(const mslt_gemm_desc& d, cudaStream_t st, char* err, bool b_static);
// The same on the tensor cores (gemm_f32x3.cu), for products without a batch: each operand has first been
// split into three bf16 planes (launch_split3; n elements of the operand's storage, 6 n bytes of planes).
// wide: device word, zeroed beforehand, that a split raises for a value the planes cannot stand for; the products
// that are given it then read the operands themselves.
// accepts: layouts the kernel takes; wins: whether it is estimated to be faster as well; planes_ready: bit 0 / 1 =
// the planes of A / B exist already.
void launch_split3(const float* x, void* planes, long long n, int* wide, cudaStream_t st);
bool gemm_f32x3_accepts(const mslt_gemm_desc& d);
bool gemm_f32x3_wins(const mslt_gemm_desc& d, int planes_ready);
int gemm_f32x3_launch(const mslt_gemm_desc& d, const void* planes_a, const void* planes_b, const int* wide, int* status,
                      cudaStream_t st, char* err);
int gemm_simt_launch(const mslt_gemm_desc& d, cudaStream_t st, char* err);
int gemm_tc_launch(const mslt_gemm_desc& d, int* status, cudaStream_t st, char* err, const int* rows, int rows_are_k,
                   bool b_static, int* parts, int room);
// Shares of its rows that a product may turn out to have where only the device knows; one alone where the host does.
struct Fills {
  int n;
  double share[3];
  static int of(int rows, double share) { const int r = (int)(share * rows); return r < 1 ? 1 : r; }
};
constexpr Fills kFull = {1, {1.}}, kUnknownFill = {3, {0.4, 0.7, 1.}};
// The form for few tiles (gemm_tc_small.cu): split count and estimated time (the mean over fills), 0 where it does not apply.
int gemm_tc_small_plan(const mslt_gemm_desc& d, int num_sms, const Fills& fills, double* t);
int gemm_tc_small_launch(const mslt_gemm_desc& d, int splits, bool early, int* status, cudaStream_t st, char* err,
                         const int* rows, bool starve);

// Test hook: the next tensor-core launch gets a producer that issues no copies and a wait limit of
// about 20 ms, so that its first wait runs out and the give-up path is exercised.
void gemm_tc_starve_next(int on);
// Measurement hook: 0 = automatic tiling, 1 = one CTA per tile, 2 = CTA pairs wherever possible.
void gemm_tc_set_variant(int variant);

// Fused attention forward (attn_tc.cu) for bf16, head width 64 and at most 512 keys per row:
//   probs[b,h,i,:] = softmax over valid keys j < seq_lens[b] of scale * q_i . k_j,  ctx = probs * v.
// qkv is the fused projection [B*S, 3*A*d] (queries, keys, values; head h in columns h*d..);
// probs ([B, A, S, S], may be null: not written) and ctx ([B*S, A*d]) are outputs.  `status` as for
// gemm_launch.  Returns 0 or a negative mslt_status with a message in `err`.
// cu (with rows, both device): the batch is packed, sequence b holds rows cu[b] .. cu[b] + len - 1 of
// qkv and ctx (allocated for B*S rows); rows = {rows in use, rounded up, query tiles}: ctx between the
// first two is zeroed.  order (more than 128 keys): 8 * sequence + tile of every query tile.
// probs then still are [B, A, S, S], with zero rows where there is no query.
// lse (more than 128 keys): [A, B*S] by row, log2 of the row's sum of exponentials, for the backward.
int attn_fwd_launch(const void* qkv, void* probs, void* ctx, const int* seq_lens, int B, int S, int A, int d,
                    float scale, int* status, cudaStream_t st, char* err, const int* cu = nullptr,
                    const int* rows = nullptr, float* lse = nullptr, const int* order = nullptr);
// Its backward: dqkv ([B*S, 3*A*d], queries | keys | values like qkv) from the saved probabilities
// and the gradient of the context dctx ([B*S, A*d]); S a multiple of 8.
//   dV = P^T dC,  dP = dC V^T,  dS = P o (dP - rowsum(dP o P)) * scale,  dQ = dS K,  dK = dS^T Q
int attn_bwd_launch(const void* qkv, const void* probs, const void* dctx, void* dqkv, int B, int S, int A, int d,
                    float scale, int* status, cudaStream_t st, char* err, const int* seq_lens = nullptr,
                    const int* cu = nullptr, const int* rows = nullptr);
// The backward for 129 to 512 keys: no stored probabilities, they are formed again from lse.  ctx is the
// forward's output, delta [3, A, B*S] scratch (per row and head: sum of dctx o ctx).  Without cu every
// sequence has S rows.  Three launches.
int attn_bwd_long_launch(const void* qkv, const void* ctx, const void* dctx, const float* lse, float* delta,
                         void* dqkv, int B, int S, int A, float scale, int* status, cudaStream_t st, char* err,
                         const int* seq_lens, const int* cu, const int* rows, const int* order);
long long attn_launches();
// Test hook like gemm_tc_starve_next, for the next attention launch (forward or backward).
void attn_starve_next(int on);

// The form of the last contraction that this thread launched, for tests (mslt_debug_last_gemm_form).
struct GemmForm { int kernel, tile_m, tile_n, k_blocks, splits; };
extern thread_local GemmForm g_gemm_form;

// Kernels launched by the GEMM front end since the library was loaded (for launch accounting).
int64_t gemm_launches();

// The same in fp32 (attn_f32.cu), S a multiple of 8 up to 128, rows not packed.  probs may be null in the
// forward; the backward needs it, and the context.
int attn_f32_fwd_launch(const float* qkv, float* probs, float* ctx, const int* seq_lens, int B, int S, int A, float scale,
                        cudaStream_t st, char* err);
int attn_f32_bwd_launch(const float* qkv, const float* probs, const float* ctx, const float* dctx, float* dqkv,
                        const int* seq_lens, int B, int S, int A, float scale, cudaStream_t st, char* err);

}  // namespace mslt
