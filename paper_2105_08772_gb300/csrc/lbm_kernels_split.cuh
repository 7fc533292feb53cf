// The step in two passes: moments, then collision (FP64; FP32 where split_applies
// says so).
//
// The first pass forms n, j and psi of every node once and writes them (20 more bytes
// a node in FP32, 40 in FP64), the second reads them back, forms the force and
// collides.  One thread per node and no barrier: each pass is as parallel as the box
// has nodes, and no halo's densities are formed twice.
//
//  * FP64 is bound by its FP64 instructions: an SM issues one warp instruction every
//    19 clocks, a single warp one every 64 clocks whatever its active lanes
//    (measured), and HBM is a tenth busy.  47 and 112 of them a node here; the tile
//    kernels form psi again in every halo (1.3 times a 32 x 8 tile's nodes, 3 times
//    again for a chunk of one plane) and chain a plane's densities in turns.
//    Measured, us a step, moment kernel -> two passes: 100x3x3 15.2 -> 8.4, 32^3 26.4
//    -> 13.5, 64^3 119 -> 87, 128^3 799 -> 651 (159 instructions a node at the rate
//    above are 619).
//  * FP32 with E6 or E8: a 32 x 4 tile forms 2.25 times its nodes' densities; here
//    psi's 32 or 92 neighbours come through L1.  E6 16^3 6.2 -> 4.0, 64^3 18.7 -> 11.5,
//    256^3 660 -> 545; E8 64^3 20.4 -> 14.8, 192^3 325 both.
//  * FP32 with tau != 1: the collision needs the node's old populations, which the
//    second pass pulls again (from L2, where the box fits it) instead of staging R + 1
//    planes of them.  120x72x100 42.0 -> 36.4.
//  * small FP32 boxes: a tile kernel's few CTAs each walk planes in turn, here all nodes
//    are in flight at once.  16^3 4.3 -> 3.2, 41^3 8.2 -> 4.8, 56^3 10.3 -> 7.3.
//
// The node's own n and j wait in planes 15 .. 18 of the population buffer being
// written: only their own thread reads them, before it stores the node's new
// populations there.  psi, which neighbours read, has a plane of its own
// (LatticeDesc::aux).  Same operations as the other kernels: bitwise equal fields.
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
template <typename T>
__device__ __forceinline__ T split_pull(const LatticeDesc& d, const SplitNode& t, int i) {
  const T* src = static_cast<const T*>(d.src) + i * d.plane;
  const int xx = wrap(t.x - cx(i), d.nx), yy = wrap(t.y - cy(i), d.ny), zz = wrap(t.z - cz(i), d.nz);
  return __ldg(src + ((zz * d.ny + yy) * d.nx + xx));
}

template <typename T>
__global__ void __launch_bounds__(128) split_moments_kernel(LatticeDesc d) {
  step_grid_enter();
  const SplitNode t(d);
  if (t.node >= d.plane) return;
  T v[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) v[i] = split_pull<T>(d, t, i);
  T dn, jx, jy, jz;
  moments(v, dn, jx, jy, jz);
  static_cast<T*>(d.aux)[t.node] = psi_of<T>(vadd(dparam<T>(d.n0, d.n0f), dn), d.eos);
  T* m = static_cast<T*>(d.dst) + kSplitMoments * d.plane + t.node;
  m[0] = dn;
  m[d.plane] = jx;
  m[2 * d.plane] = jy;
  m[3 * d.plane] = jz;
}

template <typename T, int ST, bool UNIT>
__global__ void __launch_bounds__(128) split_collide_kernel(LatticeDesc d) {
  step_grid_enter();
  constexpr int R = stencil_radius<ST>();
  const SplitNode t(d);
  if (t.node >= d.plane) return;
  T* const out = static_cast<T*>(d.dst) + t.node;
  const T* m = out + kSplitMoments * d.plane;
  const T dn = m[0], jx = m[d.plane], jy = m[2 * d.plane], jz = m[3 * d.plane];
  T old[UNIT ? 1 : Q];
  if constexpr (UNIT) {
    old[0] = (T)0;   // tau = 1 keeps nothing of it
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) old[i] = split_pull<T>(d, t, i);
  }
  int xo[2 * R + 1], yo[2 * R + 1], zo[2 * R + 1];
#pragma unroll
  for (int k = -R; k <= R; ++k) {
    xo[k + R] = wrap(t.x + k, d.nx);
    yo[k + R] = wrap(t.y + k, d.ny) * d.nx;
    zo[k + R] = wrap(t.z + k, d.nz) * d.ny * d.nx;
  }
  const T* psi = static_cast<const T*>(d.aux);
  auto at = [&](int dx, int dy, int dz) { return __ldg(psi + (zo[dz + R] + yo[dy + R] + xo[dx + R])); };
  T Fx, Fy, Fz;
  sc_force_at<T, ST>(at, at(0, 0, 0), Coupling<T>(d.eos), Fx, Fy, Fz);
  collide_nodes<T, UNIT, false>(
      dn, vadd(dparam<T>(d.n0, d.n0f), dn), jx, jy, jz, Fx, Fy, Fz, dparam<T>(d.omega, d.omegaf), (T)1,
      [&](int i) { return old[UNIT ? 0 : i]; }, [&](int i, T g) { out[i * d.plane] = g; });
}

}  // namespace lbm
