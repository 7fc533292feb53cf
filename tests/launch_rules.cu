// The host-side launch rules of lbm_launch.h behind a C interface, for the CPU tests.
#include "lbm_launch.h"

using namespace lbm;

// boxes: n triples nx, ny, nz; slots: lattices of the set that run at a time, 0 a group of
// all; takes and candidates: kBatchModes flags each.  Returns the mode the set gets.
extern "C" int rule_batch_mix(int prec, int stencil, int n, const int* boxes, const double* tau, int slots,
                              int* takes, int* candidates) {
  BatchMix m{prec, stencil, slots, slots > 0 ? 16 : 0};
  for (int k = 0; k < n; ++k) m.add(boxes[3 * k], boxes[3 * k + 1], boxes[3 * k + 2], tau[k]);
  for (int k = 0; k < kBatchModes; ++k) {
    takes[k] = m.takes(k);
    candidates[k] = m.candidate(k);
  }
  return m.mode();
}

// passes: the lattice has the psi plane of the two passes; out: ok, aligned, items, grid,
// by, zc, density threads, collision threads
extern "C" void rule_row_plan(int prec, int nx, int ny, int nz, int sms, int passes, int* out) {
  const RowPlan r = row_plan(prec, nx, ny, nz, sms, passes != 0);
  const int v[8] = {r.ok, r.aligned, r.items, r.grid, r.cfg.by, r.cfg.zc, r.cfg.nd, r.cfg.nc};
  for (int k = 0; k < 8; ++k) out[k] = v[k];
}
extern "C" int rule_row_batch_rows(int prec, int stencil, int nx, int ny, int nz) {
  return row_batch_rows(prec, stencil, nx, ny, nz);
}
// out: slot, mcap, kd, threads of a CTA at most, density and collision warps of a batch CTA
extern "C" void rule_row_caps(int prec, int* out) {
  const RowCaps c = row_caps(prec);
  const int v[6] = {c.slot, c.mcap, c.kd, kRowThreads, kRowBatchDensityWarps, kRowBatchCollideWarps};
  for (int k = 0; k < 6; ++k) out[k] = v[k];
}

// the route of a default step (kind 5 or 6, launcher-chosen z chunk), with a psi plane
extern "C" int rule_step_route(int prec, int stencil, int unit_tau, int nx, int ny, int nz, int eager) {
  const RowPlan r = row_plan(prec, nx, ny, nz, 152, prec != kF16);
  LatticeDesc d{};
  d.nx = nx;
  d.ny = ny;
  d.nz = nz;
  d.plane = (long long)nx * ny * nz;
  d.omega = unit_tau ? 1.0 : 1.25;
  d.aux = prec == kF16 ? nullptr : &d;
  d.rows = r.ok && unit_tau && stencil == 4 ? &r : nullptr;
  TileCfg c{32, stencil == 4 ? 8 : 4, 0};
  c.kind = 5;
  c.eager = eager != 0;
  return step_route(prec, stencil, d, c);
}
extern "C" int rule_steps_per_graph(int route) { return steps_per_graph((StepRoute)route); }
