// Tensor-core kernels of the surrogate network (mw3_mlp_tc.cu), for widths up to 256.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace mw3 {

constexpr int kMlpMaxLayers = 17;
constexpr int kMlpRows = 32;      // batch rows per CTA of the chain kernel

// Padded width: the neurons are the M dimension of the products (tiles of 128).
inline int mlp_tc_width(int width) { return width <= 128 ? 128 : (width <= 256 ? 256 : 0); }

struct MlpArgs {
  const float* X;                 // [.][nin] inputs, row idx[r] (or r) is batch row r
  const float* y;                 // targets (training)
  const int* idx;                 // row numbers of the batch, or nullptr
  long n;                         // batch rows of this launch
  long ntot;                      // rows of the whole batch (the loss is their mean)
  int nin, width, depth, wp;      // wp = mlp_tc_width(width)
  int woff[kMlpMaxLayers], boff[kMlpMaxLayers];   // flat offsets of W_l, b_l
  const float* p;                 // FP32 parameters (the biases)
  const __nv_bfloat16* ph;        // BF16 copy (the weights of the first and last layer)
  const unsigned char* Wf;        // [depth - 1] hidden weights W[o][i] as operands (o, K = i)
  const unsigned char* Wb;        // the same transposed: (i, K = o)
  // activations, gelu'(z) and dL/dz of every hidden layer (training): value (neuron n, row r) at
  // ((l ld + r) / 4 wp + n) 4 + r % 4, four rows of a neuron together, neurons next to each other
  float* H;
  float* D;
  float* G;
  long ld;                        // rows, a multiple of 128
  float* out;                     // [n]
  float* tpart;                   // [tile][row group][n_in + 3][wp] sums of the first and last layer
  double* lossp;                  // [tiles] sums of squared errors
  float* part;                    // [nsplit][pstride] partial gradients
  long pstride;                   // number of parameters rounded up to a multiple of 4
  int nsplit, rc;                 // batch splits of the weight gradients, rows per split
  int train;
  long wait_limit;                // polls of a bounded wait
  int* err;                       // [0] set on a wait that timed out
};

cudaError_t launch_mlp_chain(const MlpArgs& a, cudaStream_t st);
cudaError_t launch_mlp_dw(const MlpArgs& a, cudaStream_t st);
// Where the hidden weights sit in the flat parameters (hid0: offset of the second layer's W).
struct MlpShape {
  long hid0;
  int width, depth, wp;
};
// g[p] = sum of the partials in split order; with an update also one AdamW step on p and the
// BF16 copies (flat and operand form). A gradient from a wait that ran out is incomplete: once
// err[0] is set nothing is updated; err[1] is the number of the last update made.
struct MlpUpdate {
  float *p, *g, *m, *v;
  __nv_bfloat16* ph;
  const unsigned char* wmask;
  MlpShape shape;
  unsigned char *Wf, *Wb;
  float lr, b1, b2, eps, wd, c1, c2;
  int update;                     // its number, from 1 on; 0: the sum alone
  int* err;
};
cudaError_t launch_mlp_update(const float* part, int nsplit, long pstride, long nparam,
                              const MlpUpdate& u, cudaStream_t st);
// floats of MlpArgs::tpart for a batch of n rows
inline long mlp_tpart_size(long n, int n_in, int wp) {
  return (n + kMlpRows - 1) / kMlpRows * (kMlpRows / (8 * (wp / 128))) * (n_in + 3) * wp;
}
// CTAs of the weight-gradient launch per batch split
inline int mlp_dw_ctas(int depth, int wp) { return (depth - 1) * (wp / 128) * (wp / 128) + 1; }
cudaError_t launch_mlp_operands(const __nv_bfloat16* ph, const MlpShape& c, long nparam,
                                unsigned char* Wf, unsigned char* Wb, cudaStream_t st);
// loss[s] = (sum of lossp[s][0 .. tiles)) / n, tiles in order
cudaError_t launch_mlp_losses(const double* lossp, int steps, int tiles, double n, double* loss,
                              cudaStream_t st);

}  // namespace mw3
