// Every array the kernels read of the operator, formed on the device from its compact source
// (T_x of every problem, T_y and its eigenvalues): tau K in both precisions, K in the solve
// basis, and the residual coefficients.  One upload of 24 bytes per x-row (2D: plus 32 per
// y-row) and one pass replace some twenty uploads of up to 68 bytes per unknown, which with
// the host loops that formed them took most of a 0.5 ms operator swap (127 x 127, n_t = 512).
#include <algorithm>

#include "pd_internal.h"

namespace pd {

__global__ void __launch_bounds__(256) k_operator(OperatorArgs o) {
  grid_dep_wait();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < o.nrx) {
    o.rxl[j] = o.tau * o.xlo[j];
    o.rxd[j] = fma(o.tau, o.xdiag[j], 1.0);
    o.rxu[j] = o.tau * o.xup[j];
  }
  if (o.mu && j < o.ny) {
    o.ryl[j] = o.tau * o.ylo[j];
    o.ryd[j] = o.tau * o.ydiag[j];
    o.ryu[j] = o.tau * o.yup[j];
  }
  if (j >= o.nbar) return;
  // 2D: row r of the stacked grid, x-coefficients of its problem r / nym
  const int64_t r = o.mu ? j / o.nx : 0;
  const int64_t i = o.mu ? (r / o.nym) * o.nx + (j - r * o.nx) : j;
  const double lo = o.xlo[i], up = o.xup[i], di = o.mu ? o.xdiag[i] + o.mu[r] : o.xdiag[i];
  const double tl = o.tau * lo, td = o.tau * di, tu = o.tau * up;
  o.klo[j] = lo;
  o.kdiag[j] = di;
  o.kup[j] = up;
  o.tlo_d[j] = tl;
  o.tdiag_d[j] = td;
  o.tup_d[j] = tu;
  if (o.tlo_f) {
    o.tlo_f[j] = (float)tl;
    o.tdiag_f[j] = (float)td;
    o.tup_f[j] = (float)tu;
    // T_x's row sum first (exact zeros stay zero), then the mode's eigenvalue; the couplings out
    // of a block do not exist
    const int64_t ix = j % o.nx;
    const double sl = ix > 0 ? lo : 0.0, su = ix + 1 < o.nx ? up : 0.0;
    const double e = (o.xdiag[i] + sl) + su;
    o.texc_f[j] = (float)(o.tau * (o.mu ? e + o.mu[r] : e));
  }
  if (o.mu) o.rdd[j] = fma(o.tau, o.xdiag[i], 1.0) + o.tau * o.ydiag[r];
}

void launch_operator(Ctx &c, const OperatorArgs &o) {
  const int64_t n = std::max(o.nbar, std::max(o.nrx, o.ny));
  c.launch("operator", (double)o.nbar * (o.tlo_f ? 60.0 : 48.0), [&] {
    pdl_launch(c.pdl, k_operator, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, c.stream, o);
  });
}

}  // namespace pd
