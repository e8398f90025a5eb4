// The topography check the kernel runs (topography_within of paper_2011_02600_gb300/csrc/topo_check.h)
// compiled as host C++: the nodes of a dense FP64 metric array (10 fields [s][r][q], no padding) that
// are not within tol, and those where it disagrees with topography_deviation <= tol.  Built by
// tests/test_host_topography_within.py.
#include "topo_check.h"

extern "C" void host_topography_within(const double* jmet, int nq, int nr, int ns, double c, double tol, long long* far,
                                       long long* differ) {
  const long long plane = (long long)nq * nr;
  const sbp::Dims d{nq, nr, ns, nq, (int)plane, plane * ns};
  *far = *differ = 0;
  for (long long t = 0; t < plane * ns; ++t) {
    const bool in = sbp::topography_within(jmet, d.fs, c, tol, t);
    *far += !in;
    *differ += in != (sbp::topography_deviation(jmet, d, c, t) <= tol);
  }
}
