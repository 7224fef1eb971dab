// Float MLP stacks of few rows: forward and backward passes as one launch each (few_rows.cu).
#pragma once
#include "hbp_internal.h"

namespace hbp {

// Pre-LN or plain MLP stack, float, no shifted split.  Caches as hbp_forward leaves them otherwise: Y, rstd (pre-LN), ACT, DACT.
struct FewRows {
  int L = 0, d = 0, h = 0;
  int64_t N = 0;
  bool preln = false;
  float eps = 0.0f;
  const float *W1 = nullptr, *W2 = nullptr, *a = nullptr;
  int gate = HBP_GATE_ONE;
  const float* x0 = nullptr;
  float *x_all = nullptr, *Y = nullptr, *rstd = nullptr, *ACT = nullptr, *DACT = nullptr;
  // backward
  int k = 0;
  bool exact = false;  // (then k is not read)
  bool every = false;  // delta [L+1][N][d], else [N][d]
  const float* delta = nullptr;
  float* g_all = nullptr;
  bool resident = false;  // (few_rows_backward's: weights and gelu' stay in shared memory)
  float* dZ = nullptr;  // [L][N][h], or null: no parameter gradients follow
};
// Whether a stack is one that these serve faster than a launch per product.
bool few_rows_take(int64_t N, int d, int h);
// false (of either): nothing was launched (unaligned weights, more layers than fit shared memory or than gain); with *refused, because the
// device refuses the launch.
bool few_rows_forward(Launcher& lc, const FewRows& a, bool* refused);
bool few_rows_backward(Launcher& lc, const FewRows& a, bool* refused);

// Parameter gradients from the states g [L+1][N][d], what W1 was applied to y [L][N][d] (16-byte aligned) and the dZ of
// few_rows_backward; dW1, dW2 of any alignment.
void few_rows_wgrad(Launcher& lc, const FewRows& a, const float* g, const float* y, float* dW1, float* dW2);

}  // namespace hbp
