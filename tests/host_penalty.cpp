// The characteristic face penalty (add_penalty of paper_2011_02600_gb300/csrc/common.cuh) in FP32,
// compiled as host C++, at n nodes of a face with the normal along x, |a| = 1 and unit spacing.
// Built by tests/test_host_penalty.py.
#include <algorithm>
#include <cmath>

using std::max;
using std::min;
using std::sqrt;

#include "common.cuh"

static const float kAx[3] = {1.0f, 0.0f, 0.0f};

// v (3), s (6): the same at every node; mat: 1/(rho J), lambda/J, mu/J per node; out: rv (3), e (6) per node
extern "C" void host_penalty(int side, float gamma, const float* v, const float* s, const float* mat, int n,
                             float* out) {
  for (int t = 0; t < n; ++t) {
    for (int c = 0; c < 9; ++c) out[9 * t + c] = 0.0f;
    sbp::add_penalty<float>(side, 1, gamma, 1.0f, v, s, kAx, mat[3 * t], mat[3 * t + 1], mat[3 * t + 2], out + 9 * t,
                            out + 9 * t + 3);
  }
}
