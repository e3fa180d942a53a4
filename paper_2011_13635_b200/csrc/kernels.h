// Host-side launchers of the fused memory-bound kernels (kernels.cu).
// `bf` selects the activation type: true = bf16, false = float.  All pointers are device
// pointers; every launcher only enqueues work on `st`.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mslt {

struct AdamChunk {
  int64_t offset;  // element offset into the parameter arena (multiple of 4)
  int32_t count;   // elements in this chunk (multiple of 4)
  float decay;     // 1 for matrices and tables, 0 for vectors
  int32_t tensor;  // index of the tensor the chunk belongs to (LAMB sums its norms per tensor)
  int32_t pad_;
};
struct AdamHyper {
  float lr, beta1, beta2, eps, weight_decay;
  float omb1, omb2;  // 1 - beta, formed in double on the host
  float bc1, bc2;    // bias corrections 1 / (1 - beta^t), or 1: filled on the device
};

// Packed batches.  A batch whose sequences have lengths is kept without its padding: sequence b holds
// rows cu[b] .. cu[b + 1] - 1 of every activation, rows_dev (device) = {rows in use, the same rounded up
// to a tile of 128}.  The launchers below then get the allocated row count for their grid and work on the
// rows in use only; null = every row.
void launch_ln_fwd(bool bf, const void* z, const float* gamma, const float* beta, void* y,
                   float* stats, int rows, int H, float eps, cudaStream_t st, const int* rows_dev = nullptr, bool early = false);
// segments / type: segment ids and the two-row segment table, or null (no segment term).  rows = B * S.
// Packed: ptok (and pseg) receive the token id (segment) of every packed row, -1 past the last.
void launch_embed_ln(bool bf, const int* tokens, const int* segments, const void* word, const void* pos,
                     const void* type, const float* gamma, const float* beta, void* y, void* zstash,
                     float* stats, int rows, int S, int H, int V, float eps, int* status, cudaStream_t st,
                     const int* cu = nullptr, const int* rows_dev = nullptr, int* ptok = nullptr, int* pseg = nullptr);
void launch_ln_bwd(bool bf, const void* dy, const void* z, const float* stats, const float* gamma,
                   void* dz, float* dgamma, float* dbeta, float* dbias, int rows, int H, cudaStream_t st,
                   const int* rows_dev = nullptr, const void* gelu_u = nullptr);
void launch_softmax_fwd(bool bf, const void* sc, void* p, const int* seq_lens, int rows, int S,
                        int rows_per_seq, float scale, cudaStream_t st);
void launch_softmax_bwd(bool bf, void* dp, const void* p, int rows, int S, float scale,
                        cudaStream_t st);
// what a call zeroes before it starts: 16-byte vectors
struct ZeroRanges {
  void* p[8];
  int64_t vecs[8];
  int n;
  void add(void* q, int64_t bytes) {
    p[n] = q;
    vecs[n++] = (bytes + 15) / 16;
  }
};
// Opens a call: zeroes the ranges, scalars[0 .. 3] = {status, filled slots, 1 / filled slots, loss} and scalars[8], then
// checks the slots and forms rowsrc / rowlabel (positions null: not).  cu, rows, order (outputs, with
// seq_lens): the packed layout; rows[2] = number of 128-row tiles and order = 8 * sequence + tile of each,
// longest sequences first (S <= 512).
void launch_step_prepare(const ZeroRanges& zr, int* scalars, const int* positions, const int* labels, const int* seq_lens,
                         int B, int S, int P, int V, int* rowsrc, int* rowlabel, cudaStream_t st, int* cu = nullptr,
                         int* rows = nullptr, int* order = nullptr);
// out [B, S, H] from packed rows; zero past a sequence's length
void launch_unpack_rows(bool bf, const void* x, const int* cu, void* out, int B, int S, int H, cudaStream_t st);
// fp32 rows of pitch ldi to dense rows of V (a strided device copy took 91 us for 720 x 30522, this 30)
void launch_copy_rows(const float* in, int64_t ldi, float* out, int R, int V, cudaStream_t st);
void launch_gather_rows(bool bf, const void* x, const int* rowsrc, void* out, int R, int H,
                        cudaStream_t st);
void launch_scatter_rows(bool bf, const void* d, const int* rowsrc, void* dx, int B, int P, int H,
                         cudaStream_t st);
// The rows' gradient from the slots' (rows without a slot: zero), the loss from the slots' nll, and the bias
// corrections bc[2] of the step that follows the *t taken so far.
struct HeadScalars {
  const float *nll, *inv_n;
  float* loss;
  int R;
  const int* t;
  float* bc;
  float beta1, beta2;
  int bias_correction;
};
void launch_head_dx(bool bf, const void* d, const int* rowsrc, void* dx, int B, int P, int S, int H, const int* cu,
                    const int* rows_dev, const HeadScalars& hs, cudaStream_t st);
// logits fp32 [R, ldl]; dlogits (activation type) [R, ldd] or null; ldl >= ldd, both multiples of 8
void launch_cross_entropy(bool bf, const float* logits, int64_t ldl, const int* rowlabel,
                          const float* inv_n, void* dlogits, int64_t ldd, float* nll, int R, int V,
                          cudaStream_t st);
void launch_loss_reduce(const float* nll, int R, const float* inv_n, float* loss, cudaStream_t st);
// out[n] += sum over rows; N a multiple of the 16-byte vector width, out has room for N floats
void launch_colsum(bool bf, const void* x, int64_t ld, int rows, int N, float* out,
                   cudaStream_t st, const int* rows_dev = nullptr);
// The embedding gradients without hot-row atomics and with run-to-run identical bits: counting sort
// of the rows by token id, one block per token id, batch sum per position.  Needs H / (16 bytes of
// activation) <= 1024 column threads and V <= 262144.  Scratch: counts [ceil(T/256) * V], total [V],
// start [V], rank [T], order [T], blocksum [1024], hot [2 + 3 * 2048] (ints), partial [2048 * H] (floats);
// needs T <= 65536 and H / (16-byte vector) <= 256.  counts and hot[0 .. 1] are zeroed beforehand.
void launch_embed_grad_sorted(bool bf, const void* dz, const int* tokens, float* dword, float* dpos, int B, int S,
                              int H, int V, int* counts, int* total, int* start, int* rank, int* order,
                              int* blocksum, int* hot, float* partial, cudaStream_t st, const int* cu = nullptr,
                              const int* rows_dev = nullptr);
// t_dev: step count in device memory (incremented here); bc_dev: the bias corrections of this step, formed by
// launch_head_dx or launch_bias_correction
void launch_bias_correction(const int* t_dev, float* bc_dev, float beta1, float beta2, int bias_correction, cudaStream_t st);
void launch_adam(const AdamChunk* chunks, int n_chunks, float* w, const float* g, float* m, float* v,
                 void* wb, const AdamHyper& h, int* t_dev, const float* bc_dev, cudaStream_t st);
// LAMB on the same chunk table: the Adam direction r = m_hat / (sqrt(v_hat) + eps) + decay * w is
// scaled per tensor by ||w|| / ||r|| (1 when either norm is 0).  Two kernels: the first updates m and
// v and sums w^2 and r^2 of every tensor into norms[2 * tensor] / [2 * tensor + 1] (zeroed beforehand);
// the second forms r again from the new moments and applies the step. 
void launch_lamb(const AdamChunk* chunks, int n_chunks, float* w, const float* g, float* m, float* v,
                 void* wb, const AdamHyper& h, int* t_dev, const float* bc_dev, float* norms, cudaStream_t st);
// Next-sentence-prediction head.  prepare: rowsrc[b] = b * S (first tokens) and inv_n = 1 / (number of
// labels in {0, 1}, or *total_valid when given).  head: two-way classifier on the pooled rows, loss
// added to *loss, gradients of the classifier added to dwn [2,H] / dbn [2], and dup [B,H] = gradient
// at the pooler's pre-activation (tanh derivative included).
void launch_nsp_prepare(const int* labels, int B, int S, int* rowsrc, float* inv_n, const int* total_valid,
                        cudaStream_t st, const int* cu = nullptr);
void launch_nsp_head(bool bf, const void* pooled, const float* wn, const float* bn, const int* labels,
                     const float* inv_n, void* dup, float* dwn, float* dbn, float* loss, int B, int H,
                     cudaStream_t st);
void launch_tanh(bool bf, const void* x, void* y, int64_t n, cudaStream_t st);
// dtype[seg[t], :] += dz[t, :] for the two-row segment table
void launch_type_grad(bool bf, const void* dz, const int* segments, float* dtype, int rows, int H,
                      cudaStream_t st, const int* rows_dev = nullptr);
// data-parallel steps: the loss normaliser becomes 1 / *total_valid (0 when that count is 0)
void launch_override_inv_n(const int* total_valid, float* inv_n, cudaStream_t st);
void launch_sum_parts(const float* src, int64_t stride, int parts, void* dst, int64_t n, cudaStream_t st);
void launch_f32_to_bf16(const float* src, void* dst, int64_t n, cudaStream_t st);

}  // namespace mslt
