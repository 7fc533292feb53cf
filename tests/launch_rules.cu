// The host-side launch rules of lbm_launch.h behind a C interface, for the CPU tests.
#include "lbm_launch.h"

using namespace lbm;

// boxes: n triples nx, ny, nz; takes and candidates: kBatchModes flags each.  Returns
// the mode the set gets.
extern "C" int rule_batch_mix(int prec, int stencil, int n, const int* boxes, const double* tau, int* takes,
                              int* candidates) {
  BatchMix m{prec, stencil};
  for (int k = 0; k < n; ++k) m.add(boxes[3 * k], boxes[3 * k + 1], boxes[3 * k + 2], tau[k]);
  for (int k = 0; k < kBatchModes; ++k) {
    takes[k] = m.takes(k);
    candidates[k] = m.candidate(k);
  }
  return m.mode();
}
