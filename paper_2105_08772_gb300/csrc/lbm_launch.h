// Host-side launch interface between the C-ABI (lbm_api.cu) and the kernel
// translation units (one per storage precision).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>

#include <vector>

#include "lbm_common.cuh"
#include "lbm_kernels.cuh"

namespace lbm {

// Step-kernel configuration.  kind 0: lattice_kernel (register loads), one CTA
// per (column, chunk of zchunk planes).  kind 1: lattice_async_kernel
// (cp.async stages, prefetch depth `depth`) on a persistent grid; zchunk 0
// lets the launcher choose the chunk, > 0 fixes it.  kind 4: lattice_chunk_kernel
// (16-byte row chunks), kind 5: the unit-tau moment kernel with row chunks, kind 6:
// the moment kernel with element copies; same grid rules.
// prepare = true launches nothing: it sets the kernel's shared-memory limit
// (and caches the occupancy), which must happen outside any stream capture.
struct TileCfg {
  int bx, by, zchunk;
  int kind = 0;
  int depth = 1;
  bool prepare = false;
  bool eager = false;   // the step is launched by itself, not captured for replays
};

// TMA tensor maps of both population buffers of one lattice (host side; kind 7):
// map[b][0] boxes XW x PY, map[b][k] XW x k wrapped rows (k = 1 .. R + 1),
// map[b][R + 2] 4 x PY (a 16-byte x apron), over the 4-D view (x, y, z,
// population) of buffer b
struct TmaMaps {
  int ok = 0;
  int bx = 0, by = 0;               // tile shape the boxes were encoded for
  const void* base[2] = {nullptr, nullptr};
  CUtensorMap map[2][kMaxTmaMaps];
};
// Encode the maps of one FP32 lattice for bx x by tiles of a stencil of radius R.
// Returns false (t->ok = 0) when the box or the lattice does not meet the TMA
// kernel's requirements or the driver's encoder is unavailable or refuses.
bool build_tma_maps(TmaMaps* t, const void* pop0, const void* pop1, int nx, int ny, int nz, int R, int bx,
                    int by);
// the TMA kernel's requirements on the box (kind 7)
inline bool tma_box_ok(int nx, int ny, int nz, int by) {
  return nx % 4 == 0 && nx >= 64 && ny % by == 0 && ny >= 2 * by && nz >= 3;
}
// tile shapes compiled for the register-load step kernel (E4 / wider stencils)
constexpr int kNumShapesE4 = 3;
constexpr int kShapesE4[kNumShapesE4][2] = {{32, 4}, {32, 8}, {64, 4}};
constexpr int kNumShapesWide = 2;
constexpr int kShapesWide[kNumShapesWide][2] = {{32, 4}, {32, 8}};
// (bx, by, depth) compiled for the pipelined step kernel (F32 / F64 storage)
constexpr int kNumAsyncE4 = 5;
constexpr int kAsyncE4[kNumAsyncE4][3] = {{32, 8, 1}, {32, 8, 2}, {32, 4, 1}, {32, 4, 2}, {64, 4, 1}};
constexpr int kNumAsyncWide = 2;
constexpr int kAsyncWide[kNumAsyncWide][3] = {{32, 4, 1}, {32, 8, 1}};

// Launch one step (mode kModeStep) or the field-observable pass (kModeObs)
// for a lattice of the given precision and stencil.  Returns
// cudaErrorInvalidValue for a configuration that is not compiled.
cudaError_t launch_lattice_f64(int stencil, int mode, const LatticeDesc& d, TileCfg cfg,
                               const ObsArgs& oa, cudaStream_t s);
cudaError_t launch_lattice_f32(int stencil, int mode, const LatticeDesc& d, TileCfg cfg,
                               const ObsArgs& oa, cudaStream_t s);
cudaError_t launch_lattice_f16(int stencil, int mode, const LatticeDesc& d, TileCfg cfg,
                               const ObsArgs& oa, cudaStream_t s);

inline cudaError_t launch_lattice(int prec, int stencil, int mode, const LatticeDesc& d,
                                  TileCfg cfg, const ObsArgs& oa, cudaStream_t s) {
  switch (prec) {
    case kF64: return launch_lattice_f64(stencil, mode, d, cfg, oa, s);
    case kF32: return launch_lattice_f32(stencil, mode, d, cfg, oa, s);
    case kF16: return launch_lattice_f16(stencil, mode, d, cfg, oa, s);
  }
  return cudaErrorInvalidValue;
}

// dynamic shared memory of the pipelined kernel: (R + 1 + depth) population
// stages and 2R + 1 psi planes of the padded (bx + 2R) x (by + 2R) tile
constexpr size_t async_smem_bytes(size_t elem, int R, int bx, int by, int depth) {
  return elem * (size_t)(bx + 2 * R) * (by + 2 * R) * ((R + 1 + depth) * Q + 2 * R + 1);
}
// dynamic shared memory of the chunked kernel: (R + 1 + depth) stages of
// 19 x (by + 2R) rows of bx + 8 elements, psi ring of 2R + 1 padded planes
constexpr size_t chunk_smem_bytes(size_t elem, int R, int bx, int by, int depth) {
  return elem * ((size_t)(R + 1 + depth) * Q * (by + 2 * R) * (bx + 8) +
                 (size_t)(2 * R + 1) * (bx + 2 * R) * (by + 2 * R));
}
// (bx, by, depth) compiled for the chunked step kernel (kind 4)
constexpr int kNumChunkE4 = 5;
constexpr int kChunkE4[kNumChunkE4][3] = {{32, 8, 1}, {32, 8, 2}, {32, 4, 1}, {32, 4, 2}, {64, 4, 1}};
constexpr int kNumChunkWide = 1;
constexpr int kChunkWide[kNumChunkWide][3] = {{32, 4, 1}};

// staged left of a tile by the chunked copies: one 16-byte chunk, at least 4
constexpr int chunk_apron(size_t stored) { return 16 / (int)stored > 4 ? 16 / (int)stored : 4; }
// dynamic shared memory of the unit-tau moment kernel: 1 + depth stages of the
// stored type (rows of bx + 2 apron), psi ring of 2R + 2 padded planes in the
// arithmetic type
// (FP32 32 x 8 E4 tiles pad each staged row by 4 floats: see MomentShape::XWS)
constexpr size_t moment_smem_bytes(size_t stored, size_t arith, int R, int bx, int by, int depth) {
  return stored * (size_t)(1 + depth) * Q * (by + 2 * R) *
             (bx + 2 * chunk_apron(stored) + ((stored == 4 && bx == 32 && by == 8 && R == 1) ? 4 : 0)) +
         arith * (size_t)(2 * R + 2) * (bx + 2 * R) * (by + 2 * R);
}
// (bx, by, depth) compiled for the moment kernel (kind 5; tau = 1, else the
// chunked kernel of the same shape runs)
constexpr int kNumMomentE4 = 5;
constexpr int kMomentE4[kNumMomentE4][3] = {{32, 8, 1}, {32, 8, 2}, {32, 4, 1}, {32, 4, 2}, {64, 4, 1}};
constexpr int kNumMomentWide = 1;
constexpr int kMomentWide[kNumMomentWide][3] = {{32, 4, 1}};

// the moment kernel with element copies (kind 6): 1 + depth stages of 19 padded
// planes of the stored type, psi ring of 2R + 2 padded planes
constexpr size_t moment_elem_smem_bytes(size_t stored, size_t arith, int R, int bx, int by, int depth) {
  return ((size_t)(1 + depth) * Q * stored + (size_t)(2 * R + 2) * arith) * (bx + 2 * R) * (by + 2 * R);
}

// kind 6 runs 2 CTAs per SM (228 KB of shared memory, 1 KB reserved per CTA)
constexpr bool moment_elem_two_per_sm(size_t elem, int R, int bx, int by, int depth) {
  return 2 * (moment_elem_smem_bytes(elem, elem, R, bx, by, depth) + 1024) <= 228 * 1024;
}

constexpr size_t kMaxSmemPerCta = 227 * 1024;   // opt-in limit of one CTA on sm_103

// ---------------------------------------------------------------- row kernel
// The whole-row step (lbm_kernels_row.cuh) behind tile kinds 5 and 6 with a
// launcher-chosen z chunk at tau = 1.  One CTA of at most kRowThreads threads and
// nearly all of an SM's shared memory per SM: 128 registers a thread.  Versions whose
// plane loop spilled 16 bytes and more were 10 to 40% slower (L1 is some 20 KB beside
// that much shared memory).  The FP16 kernels and the FP32 one for aligned rows spill
// nothing; a few words still spill in the FP32 ones for any rows (12 bytes) and for
// batches (aligned rows 24 bytes, any rows 52).
constexpr int kRowThreads = 512;

// How one launch cuts a lattice.
struct RowCfg {
  int by, zc;    // rows and planes of an item
  int nd, nc;    // density and collision threads (multiples of 32)
};

// Capacities of a row CTA: elements of a population's slot, interior nodes, packed
// operands per density thread.  A padded node takes 19 staged populations and 2R + 2
// psi values, an interior node R + 2 planes of 4 moments (R = 1); both fill the SM at the
// tiles that the plan takes most (14 to 16 rows of 64 to 96 nodes, 4 to 8 of 128 to
// 256).
struct RowCaps { int slot, mcap, kd; };
constexpr RowCaps row_caps(int prec) {
  return prec == kF16 ? RowCaps{2336, 1920, 3} : RowCaps{1808, 1344, 3};
}

// Smaller boxes have no row plan: the two passes (F32) and the moment kernel (F16) start
// faster and have more in flight.  us, rows against the other: F32 aligned rows 64^3
// 11.4 / 9.8, 72^3 12.4 / 12.6, 96^3 22.1 / 26.2; unaligned 70x71x72 15.7 / 11.7, 97^3
// 31.3 / 27.3, 105^3 36.5 / 35.5, 113^3 43.9 / 48.3; F16 64^3 rows, 48^3 the moment
// kernel.  (row_pays leaves out more, by shape.)
constexpr long long row_min_nodes(int prec, bool aligned) {
  return prec == kF16 ? 190000 : aligned ? 350000 : 1200000;
}

struct RowPlan {
  bool ok;
  bool aligned;   // rows are whole 16-byte pieces
  int items, grid;
  RowCfg cfg;
};

// Whether a cut is expected to beat what the box runs otherwise.  Its time is that of
// row_plan, a start of 3 us (FP32), and at least the copies of each plane: 19 at 0.045 us
// each and their bytes at 54 per clock, several times as many where the blocks wrap
// around a short box in y (64x3x5000 67 us, the moment kernel 38).  One-row FP16 items
// (rows past 576 nodes, densities formed three times) count for a third more.  The
// others: the two passes (FP32 up to 1.5 million nodes, where the lattice has the psi
// plane for them: `passes`) 28 nodes a nanosecond (30 in a
// replayed graph, but two launches where steps are launched one by one: 64x64x100 13.2 us
// in rows, 13.5, and 13.7 against 18.6 launched singly); the moment kernel 27 (aligned
// rows), 23 (any rows; odd boxes), 22 in boxes that would take the two passes if they
// could (72^3 21.5 us, 452x30x30 21.2), in FP32 its last tile of a row counted whole.
// Measured on 456 boxes of 3 to 1389 rows and 3 to 31250 planes: the choice is 0.4% off
// the faster kernel on the mean, 13% at most; with the row kernel wherever it has a cut it
// was 9% on the mean and up to 3.5 times (us, row kernel / other: 33x3x20000 502 / 144,
// 449x80x80 142 / 108, 96x16x4461 240 / 194, F16 600x64x64 64.7 / 54.8).
inline bool row_pays(int prec, int nx, int ny, int nz, int sms, bool passes, const RowPlan& r, double plane,
                     double mem) {
  constexpr int R = 1;
  const double nodes = (double)nx * ny * nz;
  const int by = r.cfg.by, zc = r.cfg.zc, es = prec == kF16 ? 2 : 4;
  const int wraps = by + 2 * R <= ny && ny >= 3 * by ? 1 : (by + 2 * R <= 2 * ny ? 2 : 3);
  const double copies = 19.0 * (0.045 * wraps + (double)(by + 2 * R) * nx * es / 54.0 / 1900.0);
  const double rounds = (r.items + sms - 1) / sms;
  const double sm = rounds * ((zc + 2 * R) * (plane > copies ? plane : copies) + 0.3) + (prec == kF16 ? 0.0 : 3.0);
  const double a = sm * sm * sm, b = mem * mem * mem;
  double t = cbrt(sqrt(a * a + b * b));
  if (prec == kF16) {
    if (by == 1) t *= 1.35;
    return t < nodes / 27e3;
  }
  if (passes && nodes <= 1.5e6) return t < nodes / 28e3;
  const double rate = nodes <= 1.5e6 ? 22e3 : (r.aligned ? 27e3 : 23e3);
  return t < (double)((nx + 31) / 32 * 32) * ny * nz / rate;
}

// The cut with the least expected time, or ok = false where no item fits (rows too
// long) or the box is too small for the copies' wrap.
// An SM's time is its rounds of items times their planes (with the halo planes) times
// a plane's time: a latency (of the density warps, or of the collision warps' turns)
// and a share for each 64-node piece that the two kinds of warps handle.  Memory's
// time counts the populations once and, for boxes beyond L2, the halo planes that a
// chunk's two neighbours read at another time; large boxes also lose 2% a chunk (the
// more places of the 19 planes are walked at once: 192^3 in 4 chunks 171 us, in 5 183).
// The constants (microseconds) were
// fitted to 2300 measured cuts of 28 boxes, 24^3 to 256^3, odd and ragged ones among
// them: the plan's choice is within 4% of the best cut of each, but for two FP16 boxes
// (128^3 9%, 160^3 10%).  There is no plan where the other kernel is expected to be
// faster (row_pays).
inline RowPlan row_plan(int prec, int nx, int ny, int nz, int sms, bool passes) {
  constexpr int R = 1;   // E4 (E6 in rows: 256^3 730 us, the two passes 545)
  RowPlan best{false, false, 0, 0, {0, 0, 0, 0}};
  const int es = prec == kF16 ? 2 : 4, ve = 16 / es;
  const bool aligned = nx % ve == 0;
  if (prec == kF64 || (prec == kF16 && !aligned) || nx < 2 * R + 1 || ny < 2 * R + 1 || nz < 2 * R + 1) return best;
  if ((long long)nx * ny * nz < row_min_nodes(prec, aligned)) return best;
  const RowCaps caps = row_caps(prec);
  const double bytes = (double)nx * ny * nz * 38.0 * es;
  const double scale = (aligned ? 1.0 : 1.42) * (prec == kF16 ? 0.9 : 1.0);
  double best_t = 0.0, best_plane = 0.0, best_mem = 0.0;
  for (int by = 1; by <= ny; ++by) {
    const long long nodes = (long long)(by + 2 * R) * nx, inner = (long long)by * nx;
    if (nodes > caps.slot - 4 * ve || inner > caps.mcap) break;
    // a block's copy wraps in y at most once (aligned rows: four segments)
    if (aligned ? by + 2 * R > 3 * ny : by + 2 * R > ny + 1) break;
    const int wd = (int)((nodes + 63) / 64), wc = (int)((inner + 63) / 64);   // 64-node pieces
    const int nd = (wd + caps.kd - 1) / caps.kd, most = kRowThreads / 32 - 1 - nd;
    if (most < 1) break;
    const int turns = (wc + most - 1) / most;   // pieces a collision warp takes
    if (turns > 16) break;
    const int nc = (wc + turns - 1) / turns, cols = (ny + by - 1) / by;
    const double lat_d = 1.15 * scale, lat_c = 0.134 * turns * scale + 0.285;
    const double plane = (lat_d > lat_c ? lat_d : lat_c) + 0.0282 * (wd + 1.07 * wc) * scale;
    for (int chunks = 1, zc = nz;; chunks = (nz + zc - 2) / (zc - 1)) {   // the next with fewer planes
      zc = (nz + chunks - 1) / chunks;
      const long long items = (long long)cols * ((nz + zc - 1) / zc), rounds = (items + sms - 1) / sms;
      const double sm = rounds * ((zc + 2 * R) * plane + 0.3);
      double mem = bytes / 9e6;
      if (bytes > 2.3e8) mem = bytes / 6.55e6 * (1.0 + (bytes > 5e8 ? 1.0 : 2.0) * R / zc);
      if (bytes > 5e8 && prec == kF32) mem *= 1.0 + 0.02 * (chunks - 2);
      const double a = sm * sm * sm, b = mem * mem * mem, t = a * a + b * b;   // (sm^6 + mem^6): rises with the time
      if (!best.ok || t < best_t) {
        best_t = t;
        best_plane = plane;
        best_mem = mem;
        best = RowPlan{true, aligned, (int)items, (int)(items < sms ? items : sms), {by, zc, nd * 32, nc * 32}};
      }
      if (zc == 1) break;
    }
  }
  if (best.ok && !row_pays(prec, nx, ny, nz, sms, passes, best, best_plane, best_mem)) best.ok = false;
  return best;
}

// number of CTAs (= FieldPartial records) a kind-0 lattice launch uses
inline long long lattice_grid_ctas(const LatticeDesc& d, TileCfg cfg) {
  const long long tiles = (long long)((d.nx + cfg.bx - 1) / cfg.bx) * ((d.ny + cfg.by - 1) / cfg.by);
  return tiles * ((d.nz + cfg.zchunk - 1) / cfg.zchunk);
}

// Where the two-pass step (lbm_kernels_split.cuh) runs behind kinds 5 and 6, of the
// boxes that the row kernel leaves: always in FP64; in FP32 with E6, and with E8 at
// tau = 1; else up to 1.5 million nodes (the second pass's pull of the populations, or
// the extra planes, miss L2 beyond.  us, two passes against the old kernel's best z
// chunk, tau != 1: E4 64^3 12.0 / 14.8, 112^3 63.4 / 71.1, 120^3 77.9 / 73.3, 128^3
// 92.9 / 86.9, 256^3 701 / 585; E8 112^3 89.8 / 105, 128^3 130 / 126, 192^3 423 / 383;
// E6 128^3 95.6 / 114, 192^3 314 / 344).
inline bool split_applies(int prec, int stencil, bool unit_tau, long long nodes) {
  if (prec == kF64 || stencil == 6 || (stencil == 8 && unit_tau)) return true;
  return nodes <= 1500000;
}

// FP32 steps launched one by one, where a second launch costs more than the two passes
// gain: boxes with at most one plane of one tile for each SM (32 x 8 tiles, E6 and E8
// 32 x 4).  us a step over 100 launches, one launch against two: E4 8^3 to 32^3 6.2 /
// 8.2, 100x3x3 6.2 / 8.2, 48x48x12 8.2 / 8.2, tau 0.8 28^3 7.2 / 8.2; past the line
// 33^3 10.4 / 8.2, 3x100x100 14.7 / 8.2.  E6 and E8 gain in strips alone: 100x5x5 8.2 /
// 10.3, but 24^3 8.2 / 8.2 and a single step of 8^3 16.2 / 14.7.  (In a replayed graph
// the launches cost less and the two passes win: 8^3 4.1 / 2.8.)
inline bool eager_one_launch(int prec, int stencil, int nx, int ny, int nz) {
  const int by = stencil == 4 ? 8 : 4;
  const long long planes = (long long)((nx + 31) / 32) * ((ny + by - 1) / by) * nz;
  return prec == kF32 && planes <= 152 && (stencil == 4 || nx >= 64);
}

// What a step of this configuration runs: a tile kernel by its own name, or, behind
// kinds 5 and 6 with a launcher-chosen z chunk, the row kernel where the lattice has a
// plan (d.rows), the two passes where they are faster.
enum StepRoute : int { kRouteTile = 0, kRouteRow = 1, kRouteSplit = 2 };
inline StepRoute step_route(int prec, int stencil, const LatticeDesc& d, const TileCfg& c) {
  if ((c.kind != 5 && c.kind != 6) || c.zchunk != 0) return kRouteTile;
  const bool unit_tau = d.omega == 1.0;
  if (stencil == 4 && unit_tau && c.bx == 32 && c.by == 8 && d.rows) return kRouteRow;
  if (!d.aux || !split_applies(prec, stencil, unit_tau, d.plane)) return kRouteTile;
  return c.eager && eager_one_launch(prec, stencil, d.nx, d.ny, d.nz) ? kRouteTile : kRouteSplit;
}

// Steps of a captured graph: 128 kernels of it, since a lattice captures its graph anew
// after each initialisation (the storage shift is among the kernels' parameters).  us a
// step, initialisation and 128 steps, 128 steps of two passes a graph against 64: 16^3
// 8.2 / 6.3, 64^3 19.5 / 17.6, tau 0.8 96^3 58.7 / 56.9, FP64 32^3 18.6 / 16.6; a run of
// 2048 steps takes the same.
constexpr int steps_per_graph(StepRoute route) { return route == kRouteSplit ? 64 : 128; }

// The whole-row kernel (F32, F16; E4, tau = 1) where the lattice has a plan (d.rows);
// cudaErrorNotSupported (nothing launched) where it has not.
cudaError_t launch_row_any(int prec, const LatticeDesc& d, bool prepare, cudaStream_t s);

// ---------------------------------------------------------------- batches
struct BatchEntry;
struct BatchHeader;
// the tile every batch of this precision / stencil uses, and its launch;
// prepare readies the kernel outside capture and reports the grid it uses
// batch kernel modes: the pipelined kernel for lattices with mixed tau or all tau = 1,
// the moment kernel (all tau = 1) with row chunks (nx % 4 == 0, nx >= tile width + 8)
// or with element copies, the row kernel with all rows aligned or any rows
enum BatchMode : int { kBatchMixedTau = 0, kBatchUnitTau = 1, kBatchMoment = 2, kBatchMomentElem = 3,
                       kBatchRow = 4, kBatchRowAny = 5 };
constexpr int kBatchModes = 6;
constexpr bool batch_mode_row(int mode) { return mode == kBatchRow || mode == kBatchRowAny; }
// rows of a batch item of this box under the row kernel: as many as a CTA holds (all
// items of a launch share one split of the warps), evened out over the box; 0 where
// the row kernel does not take the box (or the storage or stencil)
constexpr int kRowBatchDensityWarps = 9, kRowBatchCollideWarps = 6;
inline int row_batch_rows(int prec, int stencil, int nx, int ny, int nz) {
  if (stencil != 4 || prec == kF64 || nx < 3 || ny < 3 || nz < 3) return 0;
  const RowCaps caps = row_caps(prec);
  const int ve = prec == kF16 ? 8 : 4;
  int most = (int)(((long long)kRowBatchDensityWarps * caps.kd * 64) / nx);
  if ((caps.slot - 4 * ve) / nx < most) most = (caps.slot - 4 * ve) / nx;
  most -= 2;
  if (caps.mcap / nx < most) most = caps.mcap / nx;
  if (ny - 1 < most) most = ny - 1;
  if (most < 1 || (prec == kF16 && nx % ve != 0)) return 0;
  const int cols = (ny + most - 1) / most;
  return (ny + cols - 1) / cols;
}
// (tile kernels only; the row kernel's items are whole rows)
inline TileCfg batch_tile(int prec, int stencil, int mode) {
  TileCfg t{32, (stencil == 4 && (prec != kF64 || mode == kBatchMomentElem)) ? 8 : 4, 0};
  t.kind = mode == kBatchMoment ? 5 : (mode == kBatchMomentElem ? 6 : 1);
  return t;
}
// whether the kernel of a batch mode takes a lattice
inline bool batch_mode_takes(int prec, int stencil, int mode, int nx, int ny, int nz, double tau) {
  if (mode == kBatchMixedTau) return prec != kF16;
  if (tau != 1.0) return false;
  switch (mode) {
    case kBatchUnitTau:
    case kBatchMomentElem: return prec != kF16;
    // (a tile's staged row, 16-byte chunks of the box's row, wraps in x at most once)
    case kBatchMoment: return nx % (prec == kF16 ? 8 : 4) == 0 && nx >= (prec == kF16 ? 48 : batch_tile(prec, stencil, mode).bx + 8);
    case kBatchRow: return nx % (prec == kF16 ? 8 : 4) == 0 && row_batch_rows(prec, stencil, nx, ny, nz) > 0;
    case kBatchRowAny: return prec == kF32 && row_batch_rows(prec, stencil, nx, ny, nz) > 0;
  }
  return false;
}
// items of one lattice in a batch launch of this mode, z chunks of zc planes; *rows as
// for BatchEntry::rows
inline long long batch_items(int prec, int stencil, int mode, int nx, int ny, int nz, int zc, int* rows) {
  const long long chunks = (nz + zc - 1) / zc;
  if (batch_mode_row(mode)) {
    *rows = row_batch_rows(prec, stencil, nx, ny, nz);
    return chunks * ((ny + *rows - 1) / *rows);
  }
  *rows = 0;
  const TileCfg t = batch_tile(prec, stencil, mode);
  return chunks * ((nx + t.bx - 1) / t.bx) * ((ny + t.by - 1) / t.by);
}
struct MixBox { int nx, ny, nz; };
// One z chunk for all lattices of a launch on `grid` resident CTAs, chosen like the
// single-lattice launcher's (fewest rounds x planes).
inline int common_zchunk(int prec, int stencil, int mode, const MixBox* b, int n, int grid) {
  const int R = stencil == 4 ? 1 : 2;
  int max_nz = 1, rows = 0;
  for (int k = 0; k < n; ++k) max_nz = b[k].nz > max_nz ? b[k].nz : max_nz;
  int best_zc = max_nz;
  long long best_cost = -1;
  for (int zc = 1; zc <= max_nz; ++zc) {
    long long items = 0;
    for (int k = 0; k < n; ++k) items += batch_items(prec, stencil, mode, b[k].nx, b[k].ny, b[k].nz, zc, &rows);
    const long long rounds = (items + grid - 1) / grid, cost = rounds * (zc + 2 * R);
    if (best_cost < 0 || cost <= best_cost) {
      best_cost = cost;
      best_zc = zc;
    }
  }
  return best_zc;
}
// Expected microseconds of a step of n lattices (E4, tau = 1), mode kBatchRow or
// kBatchRowAny.  An item takes 5 us to start (its table entry, its first copies), then
// each plane a latency and a share for each 64-node piece, as in row_plan with the
// batch's fixed warps, or its copies (see row_pays) where they take longer.
inline double batch_row_us(int prec, int mode, const MixBox* b, int n) {
  constexpr int sms = 152;
  const int zc = common_zchunk(prec, 4, mode, b, n, sms), es = prec == kF16 ? 2 : 4;
  const double scale = mode == kBatchRowAny ? 1.64 : 1.0;
  double total = 0.0, most = 0.0, mem = 0.0;
  long long items = 0;
  for (int k = 0; k < n; ++k) {
    int by = 0;
    const int z = b[k].nz < zc ? b[k].nz : zc, nx = b[k].nx, ny = b[k].ny;
    const long long it = batch_items(prec, 4, mode, nx, ny, b[k].nz, z, &by);
    const int cols = (ny + by - 1) / by, wd = ((by + 2) * nx + 63) / 64, wc = (by * nx + 63) / 64;
    const int turns = (wc + kRowBatchCollideWarps - 1) / kRowBatchCollideWarps;
    const int wraps = by + 2 <= ny && cols >= 3 ? 1 : (by + 2 <= 2 * ny ? 2 : 3);
    const double lat_d = 0.85 * scale, lat_c = 0.134 * turns * scale + 0.285;
    double plane = (lat_d > lat_c ? lat_d : lat_c) + 0.0365 * (wd + 1.07 * wc) * scale;
    const double copies = 19.0 * (0.0375 * wraps + (double)(by + 2) * nx * es / 54.0 / 1900.0);
    if (copies > plane) plane = copies;
    const double t = (z + 2) * plane + 5.0;
    total += it * t;
    items += it;
    most = t > most ? t : most;
    mem += (double)nx * ny * b[k].nz * 38.0 * es * 1.15 / 6.5e6;
  }
  double sm = total / items * ((items + sms - 1) / sms);
  if (most > sm) sm = most;
  return sqrt(sqrt(sm * sm * sm * sm + mem * mem * mem * mem));
}
// The same with a moment kernel (kBatchMoment, kBatchMomentElem) in z chunks of zc planes
// (0: common_zchunk): a tile's plane takes 1.25 us, or 0.85 (FP16 0.62) for each CTA that
// an SM holds at a time.
inline double batch_tile_us(int prec, int mode, const MixBox* b, int n, int zc) {
  constexpr int sms = 152;
  const int cap = mode == kBatchMomentElem ? 2 : (prec == kF16 ? 4 : 3), es = prec == kF16 ? 2 : 4;
  if (zc == 0) zc = common_zchunk(prec, 4, mode, b, n, sms * cap);
  const double over = mode == kBatchMomentElem ? 1.65 : (prec == kF16 ? 2.1 : 1.3);
  double planes = 0.0, mem = 0.0;
  long long items = 0;
  int deepest = 0, rows = 0;
  for (int k = 0; k < n; ++k) {
    const int z = b[k].nz < zc ? b[k].nz : zc;
    const long long it = batch_items(prec, 4, mode, b[k].nx, b[k].ny, b[k].nz, z, &rows);
    items += it;
    planes += (double)it * (z + 2);
    deepest = z + 2 > deepest ? z + 2 : deepest;
    mem += (double)b[k].nx * b[k].ny * b[k].nz * 38.0 * es * over / 6.5e6;
  }
  const long long per_sm = (items + sms - 1) / sms, rounds = (items + sms * cap - 1) / (sms * cap);
  const double share = (prec == kF16 ? 0.62 : 0.85) * (per_sm < cap ? per_sm : cap);
  const double plane = share > 1.25 ? share : 1.25;
  double sm = rounds * planes / items * plane;
  if (deepest * plane > sm) sm = deepest * plane;
  sm += 1.9;
  return sqrt(sqrt(sm * sm * sm * sm + mem * mem * mem * mem));
}
// The modes that take a set of lattices, and the one it gets.  The row kernel's few large
// items suit sets of large boxes (8 of 44^3 22 us a step, the moment kernel 39), the tile
// kernels' many small CTAs sets of small ones (48 of 16^3 16 us, the row kernel 33; 391 of
// 8^3 35, 114), so the two expected times decide, for the lattices that run at a time.
// Measured on 229 sets of 1 to 1389 lattices, 6^3 to 128^3 and flat ones, in groups and
// batches: the choice is 0.1% off the faster kernel on the mean, 7% at most.  (Never the
// row kernel below 190000 nodes in the whole set, where none was measured.)
struct BatchMix {
  int prec, stencil;
  int resident;       // lattices that run at a time (0: all)
  int tile_zchunk;    // z chunk of the tile kernels (0: common_zchunk)
  bool all[kBatchModes] = {true, true, true, true, true, true};
  double nodes = 0.0;
  std::vector<MixBox> boxes;
  void add(int nx, int ny, int nz, double tau) {
    for (int m = 0; m < kBatchModes; ++m) all[m] = all[m] && batch_mode_takes(prec, stencil, m, nx, ny, nz, tau);
    nodes += (double)nx * ny * nz;
    boxes.push_back(MixBox{nx, ny, nz});
  }
  bool takes(int mode) const { return mode >= 0 && mode < kBatchModes && all[mode]; }
  int tile_mode() const {
    for (int m : {kBatchMoment, kBatchMomentElem, kBatchMixedTau})
      if (all[m]) return m;
    return kBatchMoment;
  }
  int row_mode() const {   // -1: none
    if (nodes < 190000.0) return -1;
    return all[kBatchRow] ? kBatchRow : (all[kBatchRowAny] ? kBatchRowAny : -1);
  }
  int mode() const {
    const int row = row_mode(), tile = tile_mode();
    if (row < 0) return tile;
    std::vector<MixBox> now;   // as many as run at a time, spread over the set
    const size_t n = boxes.size(), m = resident > 0 && (size_t)resident < n ? (size_t)resident : n;
    for (size_t k = 0; k < m; ++k) now.push_back(boxes[k * n / m]);
    const double r = batch_row_us(prec, row, now.data(), (int)m);
    return r < batch_tile_us(prec, tile, now.data(), (int)m, tile_zchunk) ? row : tile;
  }
  // the modes that the batch autotuner times
  bool candidate(int m) const {
    if (!all[m]) return false;
    if (m == kBatchMixedTau) return tile_mode() == m;
    return batch_mode_row(m) ? m == row_mode() : true;
  }
};
cudaError_t launch_row_batch_any(int prec, bool aligned, const BatchEntry* table, const BatchHeader* hdr, int step,
                                 bool prepare, int* grid, cudaStream_t s);
cudaError_t launch_batch_f64(int stencil, int mode, const BatchEntry* table, const BatchHeader* hdr,
                             int step, bool prepare, int* grid, cudaStream_t s);
cudaError_t launch_batch_f32(int stencil, int mode, const BatchEntry* table, const BatchHeader* hdr,
                             int step, bool prepare, int* grid, cudaStream_t s);
cudaError_t launch_batch_f16(int stencil, int mode, const BatchEntry* table, const BatchHeader* hdr,
                             int step, bool prepare, int* grid, cudaStream_t s);
inline cudaError_t launch_batch(int prec, int stencil, int mode, const BatchEntry* table,
                                const BatchHeader* hdr, int step, bool prepare, int* grid, cudaStream_t s) {
  if (prec == kF64) return launch_batch_f64(stencil, mode, table, hdr, step, prepare, grid, s);
  if (prec == kF32) return launch_batch_f32(stencil, mode, table, hdr, step, prepare, grid, s);
  if (prec == kF16) return launch_batch_f16(stencil, mode, table, hdr, step, prepare, grid, s);
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------- io / init (lbm_io.cu)
struct DropInit {
  double cx, cy, cz, R, rho_in, rho_out, width;
};
cudaError_t launch_init_drop(int prec, const LatticeDesc& d, const DropInit& di, cudaStream_t s);
cudaError_t launch_init_rho(int prec, const LatticeDesc& d, const double* rho_dev, cudaStream_t s);
// write population plane i of the stored state from f_i(x, t) (device doubles)
cudaError_t launch_set_plane(int prec, const LatticeDesc& d, int i, const double* f_dev,
                             cudaStream_t s);
// read population plane i of the current f_i(x, t) into device doubles
cudaError_t launch_get_plane(int prec, const LatticeDesc& d, int i, double* f_dev, cudaStream_t s);

// ---------------------------------------------------------------- observables (lbm_obs.cu)
struct PointOut {
  double n_in, n_out, P_in, P_out;
};
// centre node, farthest corner and the +x half axis: n, P^yy, P^xx (Eq. (9))
cudaError_t launch_point_obs(int prec, int stencil, const LatticeDesc& d, PointOut* pts,
                             double* n_line, double* PT_line, double* PN_line, cudaStream_t s);

struct FinalizeArgs {
  const FieldPartial* partials;
  long long n_partials;
  const PointOut* pts;
  const double* PT_line;
  int line_len;
  long long volume;
  double contrast0;       // |rho_in - rho_out| of the initial state (0: no collapse test)
  int center[3];          // centre node (nx/2, ny/2, nz/2)
  int have_u_old;
  long long steps;
  double* dP_prev;        // device: previous Delta P (NaN if none); updated
  const int* err;         // device: set when a step kernel's bounded wait ran out
  void* obs_out;          // device lbm_obs
};
cudaError_t launch_finalize(const FinalizeArgs& a, cudaStream_t s);

}  // namespace lbm
