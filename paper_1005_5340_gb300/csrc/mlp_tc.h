// Tensor-core path of the guess network (mlp_tc.cu), used by learn.cu.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace tddft {

constexpr int kMlpMaxIn = 12, kMlpMaxWidth = 256, kMlpMaxOut = 4;

// One network's operands and scratch, all inside one allocation of
// mlp_tc_bytes (256-byte aligned).
struct MlpTc {
  CUtensorMap map2, map2t;         // w2 and w2t in boxes of 64 x 256 rows
  int n_in = 0, width = 0, n_out = 0;
  const float *params = nullptr;   // the packed parameters
  __nv_bfloat16 *w2 = nullptr;     // [3][256][256] planes of W2
  __nv_bfloat16 *w2t = nullptr;    // [3][256][256] planes of W2^T
  float *w1 = nullptr;             // [2][256][12] W1 (float32; rounded to bf16)
  float *vec = nullptr;            // b1, b2, W3 (float32), W3 (rounded to bf16), b3: rows of 256
  float *w3_dw2 = nullptr;         // [4][256] W3 as dW2 takes it (infinite: see odd_w)
  int *odd_w = nullptr;            // [256] per unit: 1 its row of W2 has weights without planes,
                                   // 2 it has an infinite output weight
  int *err = nullptr;              // code of a wait that gave up (0: none), training steps
                                   // skipped since, 64-bit wait limit in ns (0: 2 s)
  float *part2 = nullptr, *part1 = nullptr;   // per-CTA partial gradients
  int64_t part_stride = 0;
};

// Whether a network takes this path, its scratch, and the set-up.
bool mlp_tc_fits(int n_in, int width, int n_out);
size_t mlp_tc_bytes(int64_t max_rows);
cudaError_t mlp_tc_init(MlpTc &tc, int n_in, int width, int n_out, int64_t max_rows,
                        const float *params, void *mem, cudaStream_t st);
// Y of rows of F; with H1 and H2 (float32 weights only) both hidden layers are
// stored for mlp_tc_backward.
cudaError_t mlp_tc_forward(cudaStream_t st, const MlpTc &tc, int64_t rows, const float *F,
                           float *H1, float *H2, float *Y, bool bf16);
// grad of sum dY . Y from the stored H1 and H2 (every entry written); dH1 is
// scratch of rows x width.
cudaError_t mlp_tc_backward(cudaStream_t st, const MlpTc &tc, int64_t rows, const float *F,
                            const float *dY, const float *H1, const float *H2, float *dH1,
                            float *grad);

}  // namespace tddft
