// Fused Shan-Chen step and field-observable kernels (templated; included by
// one translation unit per storage precision).
//
// One time step of Sec. II, Eq. (3):
//   pull      f_i(x, t) = f*_i(x - xi_i, t - 1)                 (streaming)
//   moments   n = sum_i f_i, j = sum_i xi_i f_i
//   force     F = -G c_s^2 psi(x) sum_a W_a psi(x + xi_a) xi_a   Eq. (8)
//   velocity  u = (j + F/2) / n                                  Eq. (7)
//   collide   f*_i = f_i - (f_i - f_i^eq)/tau + F_i              Eqs. (4)-(6)
//   store     f*_i(x, t) at x (read by the next step's pull).
//
// The force needs psi at the stencil neighbours, i.e. the density of the
// neighbours at the same time step.  A CTA owns a BX x BY column of the box
// and marches through a chunk of z planes.  For each plane it pulls the 19
// populations of the tile plus an R-node xy halo, forms n and psi there and
// keeps them in a ring of 2R+1 psi planes in shared memory; the tile's own
// pulled populations are parked in shared memory until the plane is
// collided R planes later.  Density and psi never touch HBM: every step
// moves 19 loads + 19 stores per node, the halo re-reads hit L2.  Two
// population buffers alternate (the halo reads of one CTA may not race with
// another CTA's in-place writes).
#pragma once

#include "lbm_common.cuh"
#include "lbm_math.cuh"

namespace lbm {

// per-CTA reduction record of the field-observable pass
struct FieldPartial {
  double mass;        // sum n
  double wsum;        // sum (n - n_out)
  double wd[3];       // sum (n - n_out) d_alpha (minimum image about the centre)
  double du;          // sum_x sum_alpha |u - u_old|
  double max_u;       // max |u|
  double bad;         // count of non-finite or non-positive densities
};

struct ObsArgs {
  const double* n_out;     // device scalar: density at the farthest corner
  void* u_old;             // velocity snapshot, 3 planes (double for F64, float otherwise)
  int have_u_old;          // 0 right after an init: skip the delta-u sum
  FieldPartial* partials;  // one record per CTA
  double* rho_out;         // optional full density field (doubles), may be null
  double* u_out;           // optional full velocity field (3 planes of doubles), may be null
  int write_u_old;         // 1: replace the snapshot by the current velocity
};

template <int P, int ST, int BX, int BY>
struct StepShape {
  using T = typename Storage<P>::T;
  static constexpr int R = stencil_radius<ST>();
  static constexpr int PX = BX + 2 * R;
  static constexpr int PY = BY + 2 * R;
  static constexpr int NT = BX * BY;
  static constexpr int NR = 2 * R + 1;   // psi planes in the ring
  static constexpr int NP = R + 1;       // parked population planes
  static constexpr size_t ring_bytes = sizeof(T) * NR * PX * PY;
  static constexpr size_t pops_bytes = sizeof(T) * NP * Q * NT;
  static constexpr size_t smem_bytes = ring_bytes + pops_bytes;
};

// Pull the 19 populations of every node of one padded plane (tile + R halo),
// form psi into the ring slot, park the interior populations if asked.
template <int P, int ST, int BX, int BY>
__device__ __forceinline__ void load_plane(const LatticeDesc& d, int x0, int y0, int w, int h,
                                           int zg, typename Storage<P>::T* ring_slot,
                                           typename Storage<P>::T* pops_slot, bool keep) {
  using Sh = StepShape<P, ST, BX, BY>;
  using T = typename Sh::T;
  using S = typename Storage<P>::S;
  constexpr int R = Sh::R, PX = Sh::PX, PY = Sh::PY, NT = Sh::NT;
  const S* __restrict__ src = static_cast<const S*>(d.src);
  const int nx = d.nx, ny = d.ny, nz = d.nz;
  const long long plane = d.plane;
  const T inv_scale = dparam<T>(1.0 / d.scale, d.inv_scalef);
  const T n0 = dparam<T>(d.n0, d.n0f);
  const int z = wrap(zg, nz);
  const int zm = wrap(z - 1, nz), zp = wrap(z + 1, nz);
  const int tid = threadIdx.x;
  for (int j = tid; j < PX * PY; j += NT) {
    const int jx = j % PX, jy = j / PX;
    if (jx >= w + 2 * R || jy >= h + 2 * R) continue;
    const int gx = wrap(x0 + jx - R, nx), gy = wrap(y0 + jy - R, ny);
    const int xs[3] = {wrap(gx + 1, nx), gx, wrap(gx - 1, nx)};   // source x for c_x = -1, 0, +1
    const int ys[3] = {wrap(gy + 1, ny), gy, wrap(gy - 1, ny)};
    const int zs[3] = {zp, z, zm};
    const bool interior = keep && jx >= R && jx < R + w && jy >= R && jy < R + h;
    const int li = (jy - R) * BX + (jx - R);
    T v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const long long idx = (long long)i * plane +
                            ((long long)zs[cz(i) + 1] * ny + ys[cy(i) + 1]) * nx + xs[cx(i) + 1];
      v[i] = Storage<P>::load(src + idx, inv_scale);
      if (interior) pops_slot[i * NT + li] = v[i];
    }
    ring_slot[jy * PX + jx] = psi_of<T>(n0 + sum19(v), d.eos);
  }
}

// Shan-Chen force (sc_force_at) from psi planes in shared memory.  planes[dz + R]
// points at the node's own position in the psi plane at offset dz; rows are PX
// apart.
// OWN: own[dz + R] holds psi of the node's own column at offset dz (the caller
// formed those values and kept them in registers); differences along the node's
// own column take them from there instead of from shared memory.
template <typename T, int ST, int PX, bool OWN = false>
__device__ __forceinline__ void sc_force_pairs(const T* const* planes, Coupling<T> G, T& Fx, T& Fy, T& Fz,
                                               const T* own = nullptr) {
  constexpr int R = stencil_radius<ST>();
  auto at = [&](int dx, int dy, int dz) {
    if (OWN && dx == 0 && dy == 0) return own[R + dz];
    return planes[R + dz][dy * PX + dx];
  };
  sc_force_at<T, ST>(at, at(0, 0, 0), G, Fx, Fy, Fz);
}

// Force at interior node (tx, ty) of the current plane from the psi ring;
// slots[k] is the ring slot of plane z + k - R.
template <int P, int ST, int BX, int BY>
__device__ __forceinline__ void sc_force(const typename Storage<P>::T* ring, const int* slots, int tx,
                                         int ty, Coupling<typename Storage<P>::T> G,
                                         typename Storage<P>::T& Fx, typename Storage<P>::T& Fy,
                                         typename Storage<P>::T& Fz) {
  using Sh = StepShape<P, ST, BX, BY>;
  using T = typename Sh::T;
  constexpr int R = Sh::R, PX = Sh::PX, PY = Sh::PY;
  const T* planes[2 * R + 1];
#pragma unroll
  for (int k = 0; k <= 2 * R; ++k) planes[k] = ring + slots[k] * (PX * PY) + (ty + R) * PX + (tx + R);
  sc_force_pairs<T, ST, PX>(planes, G, Fx, Fy, Fz);
}

template <typename T>
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

// A float as a double by its bits: the conversion instruction runs at the FP64 rate,
// which is what the observable pass is bound by, the integer pipe is idle there.
// (Denormals, infinities and NaN take the instruction.)
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu, sign = u & 0x80000000u;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)f;
  return __hiloint2double((int)(m == 0u ? sign : sign | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }
// tests on the bits, off the FP64 pipe
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool positive_finite_bits(double v) {
  const int hi = __double2hiint(v);
  return (unsigned)hi < 0x7ff00000u && (hi | __double2loint(v)) != 0;
}

// whether vrcp takes v: below, 1/v or its correction would overflow, above it would be
// flushed, and of an infinity or zero vrcp makes NaN where the division makes 0 or an infinity
__device__ __forceinline__ bool rcp_range_bits(double v) {   // 2^-1000 <= |v| < 2^1000
  return (unsigned)((__double2hiint(v) & 0x7fffffff) - 0x01700000) < 0x7e700000u - 0x01700000u;
}

// minimum-image displacement of coordinate X from the centre node n/2; the plane at
// exactly half the box (even sizes) is both images and counts as 0
__device__ __forceinline__ int centre_displacement(int X, int n) {
  int dd = X - n / 2;
  if (2 * dd >= n) dd -= n; else if (2 * dd < -n) dd += n;
  return 2 * dd == -n ? 0 : dd;
}

enum Mode : int { kModeStep = 0, kModeObs = 1 };

// One CTA: tile (blockIdx.x over tiles), z chunk (blockIdx.y).
template <int P, int ST, int BX, int BY, int MODE>
__global__ void __launch_bounds__(BX * BY)
lattice_kernel(LatticeDesc d, int zchunk, ObsArgs oa) {
  using Sh = StepShape<P, ST, BX, BY>;
  using T = typename Sh::T;
  using S = typename Storage<P>::S;
  constexpr int R = Sh::R, NR = Sh::NR, NP = Sh::NP, NT = Sh::NT, PX = Sh::PX, PY = Sh::PY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);
  T* pops = reinterpret_cast<T*>(smem_raw + Sh::ring_bytes);

  const int tiles_x = (d.nx + BX - 1) / BX;
  const int x0 = (blockIdx.x % tiles_x) * BX;
  const int y0 = (blockIdx.x / tiles_x) * BY;
  const int w = min(BX, d.nx - x0), h = min(BY, d.ny - y0);
  const int z0 = blockIdx.y * zchunk;
  const int zc = min(zchunk, d.nz - z0);
  const int tid = threadIdx.x;
  const int tx = tid % BX, ty = tid / BX;
  const bool active = tx < w && ty < h;

  // prologue: planes z0-R .. z0+R-1 (q = 0 .. 2R-1); populations kept for z0 .. z0+R-1
#pragma unroll 1
  for (int q = 0; q < 2 * R; ++q) {
    const int kk = q - R;   // plane index relative to z0
    load_plane<P, ST, BX, BY>(d, x0, y0, w, h, z0 + kk, ring + (q % NR) * PX * PY,
                              pops + ((kk + NP) % NP) * Q * NT, kk >= 0 && kk < zc);
  }

  const Coupling<T> G(d.eos);
  const T omega = dparam<T>(d.omega, d.omegaf), n0 = dparam<T>(d.n0, d.n0f);
  const T scale = dparam<T>(d.scale, d.scalef);
  const long long plane = d.plane;
  double acc_mass = 0, acc_w = 0, acc_wz = 0, acc_du = 0, acc_max = 0;   // acc_max: |u|^2
  int acc_bad = 0;
  double nout = 0;
  if (MODE == kModeObs) nout = *oa.n_out;

#pragma unroll 1
  for (int k = 0; k < zc; ++k) {
    // lead plane z0 + k + R (q = k + 2R)
    {
      const int q = k + 2 * R;
      const int kk = k + R;
      load_plane<P, ST, BX, BY>(d, x0, y0, w, h, z0 + kk, ring + (q % NR) * PX * PY,
                                pops + (kk % NP) * Q * NT, kk < zc);
    }
    __syncthreads();
    if (active) {
      int slots[2 * R + 1];
#pragma unroll
      for (int s = 0; s <= 2 * R; ++s) slots[s] = (k + s) % NR;
      const T* pk = pops + (k % NP) * Q * NT;
      T g[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) g[i] = pk[i * NT + tid];
      T Fx, Fy, Fz;
      sc_force<P, ST, BX, BY>(ring, slots, tx, ty, G, Fx, Fy, Fz);
      const int z = z0 + k;
      const long long node = ((long long)z * d.ny + (y0 + ty)) * d.nx + (x0 + tx);
      if (MODE == kModeStep) {
        T dn, jx, jy, jz;
        moments(g, dn, jx, jy, jz);
        const T n = n0 + dn;
        collide<T>(g, dn, n, jx, jy, jz, Fx, Fy, Fz, omega);
        S* __restrict__ dst = static_cast<S*>(d.dst);
#pragma unroll
        for (int i = 0; i < Q; ++i) Storage<P>::store(dst + (long long)i * plane + node, g[i], scale);
      } else {
        // Observables: moments and velocity accumulated in FP64 whatever the storage.  The
        // pass is bound by its FP64 instructions (about 70 a node): one reciprocal for
        // the three velocities, |u|^2 instead of |u| (the root of the maximum is the
        // maximum of the roots), displacements along x and y applied once per thread.
        // A call of lbm_observables at 128^3 FP32, with the two kernels of lbm_obs.cu:
        // 863 -> 563 us.
        double gd[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) gd[i] = widen(g[i]);
        double dnd, jxd, jyd, jzd;
        moments(gd, dnd, jxd, jyd, jzd);
        const double nd = d.n0 + dnd, inv_n = rcp_range_bits(nd) ? vrcp(nd) : 1.0 / nd;
        const double uxd = __fma_rn(0.5, widen(Fx), jxd) * inv_n;
        const double uyd = __fma_rn(0.5, widen(Fy), jyd) * inv_n;
        const double uzd = __fma_rn(0.5, widen(Fz), jzd) * inv_n;
        acc_mass += nd;
        if (!positive_finite_bits(nd) || !finite_bits(uxd) || !finite_bits(uyd) || !finite_bits(uzd)) ++acc_bad;
        const double wgt = nd - nout;
        acc_w += wgt;
        acc_wz += wgt * centre_displacement(z, d.nz);
        acc_max = fmax(acc_max, uxd * uxd + uyd * uyd + uzd * uzd);
        if (P == kF64) {
          double* uo = static_cast<double*>(oa.u_old);
          if (oa.have_u_old)
            acc_du += fabs(uxd - uo[node]) + fabs(uyd - uo[plane + node]) + fabs(uzd - uo[2 * plane + node]);
          if (oa.write_u_old) {
            uo[node] = uxd;
            uo[plane + node] = uyd;
            uo[2 * plane + node] = uzd;
          }
        } else {
          float* uo = static_cast<float*>(oa.u_old);
          if (oa.have_u_old)
            acc_du += fabs(uxd - widen(uo[node])) + fabs(uyd - widen(uo[plane + node])) +
                      fabs(uzd - widen(uo[2 * plane + node]));
          if (oa.write_u_old) {
            uo[node] = (float)uxd;
            uo[plane + node] = (float)uyd;
            uo[2 * plane + node] = (float)uzd;
          }
        }
        if (oa.rho_out) oa.rho_out[node] = nd;
        if (oa.u_out) {
          oa.u_out[node] = uxd;
          oa.u_out[plane + node] = uyd;
          oa.u_out[2 * plane + node] = uzd;
        }
      }
    }
    __syncthreads();
  }

  if (MODE == kModeObs) {
    __shared__ double red[8][NT / 32];
    double v[8] = {acc_mass, acc_w, acc_w * centre_displacement(x0 + tx, d.nx),
                   acc_w * centre_displacement(y0 + ty, d.ny), acc_wz, acc_du, (double)acc_bad, acc_max};
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int q = 0; q < 7; ++q) v[q] = warp_sum<double>(v[q]);
    v[7] = warp_max(v[7]);
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) red[q][warp] = v[q];
    }
    __syncthreads();
    if (tid == 0) {
      double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int wi = 0; wi < NT / 32; ++wi) {
#pragma unroll
        for (int q = 0; q < 7; ++q) s[q] += red[q][wi];
        s[7] = fmax(s[7], red[7][wi]);
      }
      FieldPartial& out = oa.partials[blockIdx.y * gridDim.x + blockIdx.x];
      out.mass = s[0];
      out.wsum = s[1];
      out.wd[0] = s[2];
      out.wd[1] = s[3];
      out.wd[2] = s[4];
      out.du = s[5];
      out.bad = s[6];
      out.max_u = sqrt(s[7]);
    }
  }
}

}  // namespace lbm
