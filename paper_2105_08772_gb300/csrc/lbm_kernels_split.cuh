// FP64 step in two passes: moments, then collision.
//
// The FP64 step is bound by its FP64 instructions: an SM issues one warp
// instruction every 19 clocks, a single warp one every 64 clocks whatever its
// active lanes (measured).  HBM is a tenth busy, so the step trades bytes for
// instructions: the first pass forms n, j and psi of every node ONCE (47
// instructions), where the tile kernels form psi again in every halo (1.3 times a
// 32 x 8 tile's nodes, 3 times again for a chunk of one plane); the second reads
// them back and collides (112).  One thread per node and no barrier: each pass is
// as parallel as the box has nodes, which is what small boxes lack most (32^3: a
// plane's densities in three chained turns before).
//
// The node's own n and j wait in planes 15 .. 18 of the population buffer being
// written: only their own thread reads them, before it stores the node's new
// populations there.  psi, which neighbours read, has a plane of its own (LatticeDesc::aux).
// Same operations as the other kernels, any tau and stencil: bitwise equal fields.
//
// Measured, us a step, moment kernel -> two passes: 100x3x3 15.2 -> 8.4 (a launch each
// and the chain of 47 and 112 instructions of a lone warp), 32^3 26.4 -> 13.5, 64^3
// 119 -> 87, 128^3 799 -> 651 (159 instructions a node at the rate above are 619).
#pragma once

#include "lbm_launch.h"
#include "lbm_math.cuh"

namespace lbm {

constexpr int kSplitMoments = 15;   // first of the four planes that hold n, jx, jy, jz between the passes

struct SplitNode {
  int x, y, z, node;
  __device__ __forceinline__ SplitNode(const LatticeDesc& d) {
    node = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    x = node % d.nx;
    const int r = node / d.nx;
    y = r % d.ny;
    z = r / d.ny;
  }
};

// population i of the node as it streams in
__device__ __forceinline__ double split_pull(const LatticeDesc& d, const SplitNode& t, int i) {
  const double* src = static_cast<const double*>(d.src) + i * d.plane;
  const int xx = wrap(t.x - cx(i), d.nx), yy = wrap(t.y - cy(i), d.ny), zz = wrap(t.z - cz(i), d.nz);
  return __ldg(src + ((long long)zz * d.ny + yy) * d.nx + xx);
}

static __global__ void __launch_bounds__(128) split_moments_kernel(LatticeDesc d) {
  step_grid_enter();
  const SplitNode t(d);
  if (t.node >= d.plane) return;
  double v[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) v[i] = split_pull(d, t, i);
  double dn, jx, jy, jz;
  moments(v, dn, jx, jy, jz);
  static_cast<double*>(d.aux)[t.node] = psi_of<double>(vadd(d.n0, dn), d.eos);
  double* m = static_cast<double*>(d.dst) + kSplitMoments * d.plane + t.node;
  m[0] = dn;
  m[d.plane] = jx;
  m[2 * d.plane] = jy;
  m[3 * d.plane] = jz;
}

template <int ST, bool UNIT>
__global__ void __launch_bounds__(128) split_collide_kernel(LatticeDesc d) {
  step_grid_enter();
  constexpr int R = stencil_radius<ST>();
  const SplitNode t(d);
  if (t.node >= d.plane) return;
  double* const out = static_cast<double*>(d.dst) + t.node;
  const double* m = out + kSplitMoments * d.plane;
  const double dn = m[0], jx = m[d.plane], jy = m[2 * d.plane], jz = m[3 * d.plane];
  int xo[2 * R + 1], yo[2 * R + 1], zo[2 * R + 1];
#pragma unroll
  for (int k = -R; k <= R; ++k) {
    xo[k + R] = wrap(t.x + k, d.nx);
    yo[k + R] = wrap(t.y + k, d.ny) * d.nx;
    zo[k + R] = wrap(t.z + k, d.nz) * d.ny * d.nx;
  }
  const double* psi = static_cast<const double*>(d.aux);
  auto at = [&](int dx, int dy, int dz) { return __ldg(psi + (zo[dz + R] + yo[dy + R] + xo[dx + R])); };
  double Fx, Fy, Fz;
  sc_force_at<double, ST>(at, at(0, 0, 0), d.eos.G, Fx, Fy, Fz);
  collide_nodes<double, UNIT, false>(
      dn, vadd(d.n0, dn), jx, jy, jz, Fx, Fy, Fz, d.omega, 1.0, [&](int i) { return split_pull(d, t, i); },
      [&](int i, double g) { out[i * d.plane] = g; });
}

}  // namespace lbm
