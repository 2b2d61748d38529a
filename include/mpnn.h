/*
 * mpnn.h -- C ABI of the message-passing surrogate kernels in libdem.so.
 *
 * The surrogate is a learned stand-in for the DEM force evaluation over a
 * stride of time steps: a message-passing network over the particle
 * neighbour graph that predicts each particle's mean linear and angular
 * acceleration over the stride.  This header exposes its building blocks;
 * the network, its training loop and the DEM fallback are assembled by the
 * Python module paper_2507_12610_gb300/surrogate.py.  The paper has no
 * learned component; these entry points are the project's own.
 *
 * Conventions: every pointer is a DEVICE pointer unless stated; matrices are
 * row-major; bf16 is IEEE bfloat16 stored as uint16_t; `stream` is a
 * cudaStream_t (NULL = legacy default stream).  Calls enqueue work and return
 * without waiting (except mpnn_graph, which reads the edge count back); they
 * return DEM_OK (0), DEM_ERR_INVALID (1) for bad sizes or NULL pointers,
 * DEM_ERR_CAPACITY (2) if the edge buffers are too small, or DEM_ERR_CUDA (4)
 * if a launch fails.  No call allocates device memory.  Every sum is taken in
 * a fixed order: results do not depend on the launch shape or on timing.
 */
#ifndef MPNN_H_
#define MPNN_H_

#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* C[M][N] (fp32) = A[M][K] (bf16) * B, B given transposed as Bt[N][K] (bf16),
 * then, by `epi`: 0 plain, 1 + bias[N] (fp32), 2 relu(+ bias).  If Cb is not
 * NULL the result is also written as bf16 to Cb[M][N].  With `accumulate`
 * nonzero, C += A * B (epi must be 0).  Tensor cores (mma m16n8k16, bf16
 * inputs, fp32 accumulation).  Requires M % 64 == 0, N % 64 == 0, K % 16 == 0. */
int mpnn_gemm(int64_t M, int64_t N, int64_t K, const uint16_t* A, const uint16_t* Bt,
              float* C, uint16_t* Cb, const float* bias, int32_t epi, int32_t accumulate,
              void* stream);

/* As mpnn_gemm (epi 0) with the k range split in `splits` parts whose partial
 * products go to work[splits][M][N] (caller-owned) and are then summed in
 * ascending part order; for long reductions (weight gradients). */
int mpnn_gemm_split(int64_t M, int64_t N, int64_t K, int32_t splits, const uint16_t* A,
                    const uint16_t* Bt, float* C, int32_t accumulate, float* work, void* stream);

/* Out[R][C] (bf16) = In[C][R] transposed. */
int mpnn_transpose_bf16(int64_t R, int64_t C, const uint16_t* in, uint16_t* out, void* stream);

/* fp32 -> bf16 (round to nearest even) of n values. */
int mpnn_to_bf16(int64_t n, const float* in, uint16_t* out, void* stream);

/* Neighbour graph: for each of n nodes at x (fp32 [n][3]) the nodes j != i
 * with |x_j - x_i| < cutoff, in ascending j: cnt[n] (work), off[n+1] (CSR
 * offsets, int64), nbr[E] (sender j), dst[E] (receiver i).  Writes the edge
 * count E to *n_edges_host (host pointer; the call waits for it) and returns
 * DEM_ERR_CAPACITY without writing edges if E > max_edges.  All pairs are
 * tested (O(n^2), tiled through shared memory). */
int mpnn_graph(int64_t n, const float* x, float cutoff, int64_t* cnt, int64_t* off,
               int32_t* nbr, int32_t* dst, int64_t max_edges, int64_t* n_edges_host,
               void* stream);

/* The same graph from cell lists (cells of edge `cutoff` over the nodes'
 * bounding box, 27 cells searched per node; O(n)), in ascending j per node.
 * work: device workspace of 2 (max_cells + 1) + 2 n int64 words + 1; box:
 * 6 floats of device memory (the bounding box, written).  The call waits for
 * the bounding box and the edge count.  Errors: DEM_ERR_INVALID (n < 1 or
 * n >= 2^24, non-finite positions, cutoff <= 0), DEM_ERR_CAPACITY (more than
 * max_cells cells, more than max_edges edges, or a node with more than 128
 * neighbours; nothing written then). */
int mpnn_graph_cells(int64_t n, const float* x, float cutoff, int64_t max_cells, int64_t* work,
                     float* box, int64_t* cnt, int64_t* off, int32_t* nbr, int32_t* dst,
                     int64_t max_edges, int64_t* n_edges_host, void* stream);

/* perm[k] = index of the reverse of edge k (the graph is symmetric); grouped
 * by off, perm lists the edges each node sends, in ascending receiver. */
int mpnn_reverse_edges(int64_t E, const int64_t* off, const int32_t* nbr, const int32_t* dst,
                       int32_t* perm, void* stream);

/* Network inputs, 16 bf16 columns per node / edge, column 7 = 1 (bias):
 * node i: v_i / vs, R_i w_i / vs, R_i / Rs - 1; edge (i <- j):
 * (x_j - x_i) / Rs, (|x_j - x_i| - R_i - R_j) / Rs, (v_j - v_i) / vs.  Rows
 * past n (up to npad) and past E (up to Epad) are zero.  x, v, w fp32 [n][3],
 * R fp32 [n]. */
int mpnn_features(int64_t n, int64_t npad, int64_t E, int64_t Epad, const int32_t* dst,
                  const int32_t* nbr, const float* x, const float* v, const float* w,
                  const float* R, float vs, float Rs, uint16_t* nf, uint16_t* ef, void* stream);

/* Message-layer input: row e of Out (bf16, width 2H + F + 16) =
 * [Hn[dst[e]], Hn[src[e]], Ef[e], 1, 0 x 15]; rows past E (up to Epad) zero. */
int mpnn_gather_edges(int64_t E, int64_t Epad, int32_t H, int32_t F, const int32_t* dst,
                      const int32_t* src, const uint16_t* Hn, const uint16_t* Ef, uint16_t* out,
                      void* stream);

/* Out[i] = [A[i] (bf16, WA columns), bf16(B[i]) (fp32, WB columns), 1, 0 x 15];
 * rows past n (up to npad) zero. */
int mpnn_concat_rows(int64_t n, int64_t npad, int32_t WA, int32_t WB, const uint16_t* A,
                     const float* B, uint16_t* out, void* stream);

/* h += u (fp32, n values) and hb = bf16(h). */
int mpnn_residual(int64_t n, float* h, const float* u, uint16_t* hb, void* stream);

/* Out[e] = In[idx[e]] (fp32 rows of width W); rows past E (up to Epad) zero. */
int mpnn_gather_rows(int64_t E, int64_t Epad, int32_t W, const int32_t* idx, const float* in,
                     float* out, void* stream);

/* Out[i][:] = sum over e in [off[i], off[i+1]) of In[e][:] (fp32, width W),
 * ascending e; rows past n (up to npad) zero. */
int mpnn_segment_sum(int64_t n, int64_t npad, int32_t W, const int64_t* off, const float* in,
                     float* out, void* stream);

/* As mpnn_segment_sum over columns [c0, c0 + W) of rows of width `stride`,
 * through perm when not NULL (In row perm[k] for k in the segment). */
int mpnn_segment_sum_cols(int64_t n, int64_t npad, int32_t W, int64_t stride, int32_t c0,
                          const int64_t* off, const int32_t* perm, const float* in, float* out,
                          void* stream);

/* As mpnn_segment_sum through perm. */
int mpnn_segment_sum_perm(int64_t n, int64_t npad, int32_t W, const int64_t* off,
                          const int32_t* perm, const float* in, float* out, void* stream);

/* ReLU backward: G[i] = 0 where Y[i] <= 0 (fp32, n values). */
int mpnn_relu_backward(int64_t n, const float* Y, float* G, void* stream);

/* The layers of the network of width 128 (surrogate.py) with their gathers,
 * concatenations, residuals and sums inside, bitwise equal to the calls above
 * in sequence.  npad is a multiple of 64, every pointer 16-byte aligned.
 * Weights are the transposed bf16 copies Wt[outputs][inputs].
 *
 * Encode: h = relu(nf Wn) (nf [npad][16]), hb = bf16(h), and p1 [npad][128] =
 * hb times the first 128 input rows (the receiver's) of the next round's
 * message layer Wm_next [128][400]. */
int mpnn_encode_nodes(int64_t n, int64_t npad, const uint16_t* nf, const uint16_t* Wn,
                      const uint16_t* Wm_next, float* h, uint16_t* hb, float* p1, void* stream);

/* The same, and *status (device, may be NULL) = DEM_OK. */
int mpnn_encode_nodes_checked(int64_t n, int64_t npad, const uint16_t* nf, const uint16_t* Wn,
                              const uint16_t* Wm_next, float* h, uint16_t* hb, float* p1,
                              int32_t* status, void* stream);

/* Edge states: eb [E][128] = bf16(relu(ef We)) (ef [E][16]). */
int mpnn_encode_edges(int64_t E, const uint16_t* ef, const uint16_t* We, uint16_t* eb,
                      void* stream);

/* One round's messages, relu([h_dst, h_nbr, e, 1] Wm), summed over the edges
 * each node receives, ascending: Mb [npad][128] bf16 (rows 0 .. n-1 written;
 * NaN if a bounded wait inside the kernel ran out).  eb: the edge states; p1:
 * from the node call before.  Optional mask [E][4]: the bits of the message
 * components > 0 (component c: word c / 32, bit c % 32). */
int mpnn_message_sums(int64_t n, int64_t E, const int64_t* off, const int32_t* nbr,
                      const int32_t* dst, const uint16_t* hb, const uint16_t* eb,
                      const uint16_t* Wm, const float* p1, uint16_t* Mb, uint32_t* mask,
                      void* stream);

/* The same, with the number of tries of each bounded wait (< 0: the library's,
 * 2^18; 0: every wait runs out at once) and a report: *status (device, may be
 * NULL) becomes DEM_ERR_TIMEOUT if a wait ran out and is left alone otherwise.
 * (The next layer's relu takes a NaN in Mb for 0: the status is what tells.) */
int mpnn_message_sums_checked(int64_t n, int64_t E, const int64_t* off, const int32_t* nbr,
                              const int32_t* dst, const uint16_t* hb, const uint16_t* eb,
                              const uint16_t* Wm, const float* p1, uint16_t* Mb, uint32_t* mask,
                              int32_t tries, int32_t* status, void* stream);

/* Node update: h += relu([hb_in, Mb, 1] Wu) (rows past n: plus nothing), hb =
 * bf16(h) (may be hb_in), then out = p1 for the next round (W_next the message
 * layer [128][400], out [npad][128]) or, with decode nonzero, the outputs
 * [hb, 1] W_next (W_next [64][144], out [npad][64]).  Optional mask [npad][4]:
 * the bits of the update components > 0. */
int mpnn_update_nodes(int64_t n, int64_t npad, const uint16_t* hb_in, const uint16_t* Mb,
                      const uint16_t* Wu, const uint16_t* W_next, int32_t decode, float* h,
                      uint16_t* hb, float* out, uint32_t* mask, void* stream);

/* The same; with decode, the outputs are NaN if *status (device, may be NULL) is
 * not DEM_OK. */
int mpnn_update_nodes_checked(int64_t n, int64_t npad, const uint16_t* hb_in, const uint16_t* Mb,
                              const uint16_t* Wu, const uint16_t* W_next, int32_t decode,
                              float* h, uint16_t* hb, float* out, uint32_t* mask,
                              const int32_t* status, void* stream);

/* Backward of the fused layers.  zb is the bf16 gradient of a layer's output
 * before its relu (zero where the relu cut it off); W the bf16 copies
 * W[inputs][outputs]; gradients of the states add up in the order of the calls
 * above in sequence (the same bits).  Pointers are 16-byte aligned.
 *
 * Decoder: dh [npad][128] = dyb [npad][64] times Wdec^T, and zb [npad][128] of
 * the last update layer (mask: its bits). */
int mpnn_grad_decode(int64_t npad, const uint16_t* dyb, const uint16_t* Wdec,
                     const uint32_t* mask, float* dh, uint16_t* zb, void* stream);

/* Update layer: dh += the state's part of zb Wu^T; dMb = the message sums' part. */
int mpnn_grad_update(int64_t npad, const uint16_t* zb, const uint16_t* Wu, float* dh,
                     uint16_t* dMb, void* stream);

/* Message layer: zm [E][128], the edge's gradient, is dMb[dst] where its mask bits
 * are set and 0 elsewhere; dX
 * [E][256] = the receiver's and sender's parts of it times Wm^T; de [E][128] the
 * edge state's, starting at 0 with `first`; with `last` it is not stored, and zeb
 * [E][128] = bf16(de) where eb > 0. */
int mpnn_grad_messages(int64_t E, const int32_t* dst, const uint16_t* dMb, const uint32_t* mask,
                       const uint16_t* Wm, const uint16_t* eb, int32_t first, int32_t last,
                       uint16_t* zm, float* dX, float* de, uint16_t* zeb, void* stream);

/* Nodes: dh = (dh + the sum of dX[e][0..128) over the edges received) + the sum of
 * dX[perm][128..256) over those sent; zb = bf16(dh) where the bits of mask are set
 * or, with mask NULL, where hb > 0. */
int mpnn_grad_nodes(int64_t n, int64_t npad, const int64_t* off, const int32_t* perm,
                    const float* dX, const uint32_t* mask, const uint16_t* hb, float* dh,
                    uint16_t* zb, void* stream);

/* Weights: G [kp][N] = [X0[idx0], X1[idx1], X2, 1]^T dZ over `rows` rows, of the
 * first `segments` (1 to 3) inputs of width 128 each; idx NULL: the row itself.
 * segments 0: X0 of width 16 alone, no constant.  N = 128 (one segment: or 64).
 * Rows of G past the inputs are zero.  The bits are those of mpnn_gemm_split over K
 * >= rows rows (zeros after `rows`, K % 16 == 0) in `splits` parts; work
 * [splits][kp][N], caller-owned. */
int mpnn_grad_weights(int64_t rows, int64_t K, int32_t segments, const uint16_t* X0,
                      const int32_t* idx0, const uint16_t* X1, const int32_t* idx1,
                      const uint16_t* X2, const uint16_t* dZ, int32_t N, int32_t kp,
                      int32_t splits, float* work, float* G, void* stream);

/* Adam step (bias-corrected, step t >= 1) on n fp32 parameters W with
 * moments m, v and gradient G.  Also writes the bf16 copy Wb (same layout,
 * may be NULL) and, if Wt is not NULL, the transposed bf16 copy of the
 * [rows][cols] matrix's first kin rows: Wt[cols][kin]. */
int mpnn_adam(int64_t n, float* W, float* m, float* v, const float* G, float lr, float beta1,
              float beta2, float eps, int64_t t, uint16_t* Wb, uint16_t* Wt, int32_t rows,
              int32_t cols, int32_t kin, void* stream);

/* out[0] = sum of (a - b)^2 over n values (in a fixed order), and
 * G = 2 (a - b) * scale. */
int mpnn_mse(int64_t n, const float* a, const float* b, float scale, float* G, float* out,
             void* stream);

#ifdef __cplusplus
}
#endif

#endif /* MPNN_H_ */
