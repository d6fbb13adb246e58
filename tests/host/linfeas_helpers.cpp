// Host build of the projection's branch subproblem (linfeas_qp.cuh) for the
// CPU tests.  Plain C entry point for ctypes.
#define ACOPF_HD
#include <math.h>
#include <algorithm>
using std::fmax;
#include "../../paper_2310_13143_gb300/csrc/linfeas_qp.cuh"
using namespace acopf;

extern "C" void host_quot_kept(int n, const double* a, const double* b, double* out) {
  for (int i = 0; i < n; ++i) out[i] = quot_kept(a[i], b[i], 1.0 / b[i]);
}

// in: Y (gii bii gij bij gji bji gjj bjj), rho, 2 wR0, 2 wI0, bounds of w_i
// and w_j, y of the two ends (21 values per problem); out: w_i, w_j, wR, wI
extern "C" void host_lf_branch(int n, const double* in, double* out) {
  for (int b = 0; b < n; ++b) {
    const double* r = in + 21 * b;
    double c[kLfBranch];
    lf_constants(r, r[8], c);
    for (int k = 8; k < kLfBranch; ++k) c[k] = r[1 + k];
    lf_branch(r, c, r + 15, r + 18, out + 4 * b, lf_edges);
  }
}
