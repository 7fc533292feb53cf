// Launches of the row kernel (E4, tau = 1; F32 and F16), single lattices and batches:
// a translation unit of its own, it compiles longest.
#include "lbm_kernels_row.cuh"
#include "lbm_step_launch.h"

namespace lbm {

// Launched with programmatic serialisation (the next step's CTAs take over SM by SM:
// 128^3 58.5 -> 56.2 us, 64^3 17.8 -> 15.2 us when it came in).
template <int P, bool ALIGNED>
static cudaError_t launch_row_shape(const LatticeDesc& d, const RowPlan* r, cudaStream_t s) {
  using Sh = RowShape<P>;
  auto kern = lattice_row_kernel<Sh, ALIGNED>;
  if (!r)   // prepare
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
  // every other step walks the planes downwards: what the last step wrote last is
  // read first, from L2 (128^3 54.1 -> 53.1 us, 192^3 170.4 -> 169.5, 157^3 100.5 -> 101.5)
  const int flip = reinterpret_cast<uintptr_t>(d.src) > reinterpret_cast<uintptr_t>(d.dst);
  return launch_step_kernel(kern, r->grid, r->cfg.nd + r->cfg.nc + 32, Sh::smem_bytes, s, true, d, r->cfg, flip);
}

// The whole-row kernel by the lattice's plan; cudaErrorNotSupported (nothing launched)
// where it has none.  One CTA per SM.
template <int P>
static cudaError_t launch_row(const LatticeDesc& d, bool prepare, cudaStream_t s) {
  const RowPlan* r = static_cast<const RowPlan*>(d.rows);
  if (prepare) {
    cudaError_t e = launch_row_shape<P, true>(d, nullptr, s);
    if constexpr (P != kF16)
      if (e == cudaSuccess) e = launch_row_shape<P, false>(d, nullptr, s);
    return e;
  }
  if (!r || !r->ok) return cudaErrorNotSupported;
  if (r->aligned) return launch_row_shape<P, true>(d, r, s);
  if constexpr (P == kF16) return cudaErrorNotSupported;
  else return launch_row_shape<P, false>(d, r, s);
}

template <int P, bool ALIGNED>
static cudaError_t launch_row_batch(const BatchEntry* table, const BatchHeader* hdr, int step, bool prepare,
                                    int* grid, cudaStream_t s) {
  using Sh = RowShape<P>;
  auto kern = lattice_row_batch_kernel<Sh, ALIGNED>;
  static int sms = 0;
  if (prepare || sms == 0) {
    int dev = 0, n = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms = n;
  }
  if (grid) *grid = sms;
  if (prepare) return cudaSuccess;
  return launch_step_kernel(kern, sms, (1 + kRowBatchDensityWarps + kRowBatchCollideWarps) * 32, Sh::smem_bytes, s,
                            true, table, hdr, step);
}

cudaError_t launch_row_any(int prec, const LatticeDesc& d, bool prepare, cudaStream_t s) {
  return prec == kF16 ? launch_row<kF16>(d, prepare, s) : launch_row<kF32>(d, prepare, s);
}

cudaError_t launch_row_batch_any(int prec, bool aligned, const BatchEntry* table, const BatchHeader* hdr, int step,
                                 bool prepare, int* grid, cudaStream_t s) {
  if (prec == kF16 && aligned) return launch_row_batch<kF16, true>(table, hdr, step, prepare, grid, s);
  if (prec == kF32 && aligned) return launch_row_batch<kF32, true>(table, hdr, step, prepare, grid, s);
  if (prec == kF32) return launch_row_batch<kF32, false>(table, hdr, step, prepare, grid, s);
  return cudaErrorInvalidValue;
}

}  // namespace lbm
