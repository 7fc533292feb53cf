// Observables of one lattice: point samples of the lattice pressure tensor
// and the closing FP64 reduction + closed forms.
//
// Point pass (one thread per sampled node): n and P^xx, P^yy of Eq. (9)
//   P^{mu nu}(x) = n c_s^2 delta + (G c_s^2 / 2) psi(x) sum_a W_a psi(x + xi_a) xi_a^mu xi_a^nu
// at the centre node c (P_in), the farthest corner (P_out) and along the +x
// half axis c + r e_x, r = 0..nx/2 (P_T(r) = P^yy, Sec. III below Eq. (22);
// P_N(r) = P^xx, used by the flat interface's sigma_0, Eq. (25)).
//
// Finalize (one CTA, fixed reduction order, so the result is deterministic):
//   mass M, centre of mass of n - n_out, delta u (Sec. IV), max |u|,
//   R_e from M = 4 pi R_e^3 n_in/3 + (V - 4 pi R_e^3/3) n_out (Sec. IV),
//   C = int r^2 (P_out - P_T) dr, D = int r (P_out - P_T) dr (trapezoid on the
//   nodes), R_s = (6 C / dP)^(1/3) -- the minimum of
//   sigma[R] = dP R / 3 + C / R^2, Eq. (21) with the step P_J integrated
//   exactly -- and sigma_s = dP R_s / 2 (Eq. (12)).
#include <math.h>

#include "lbm.h"
#include "lbm_launch.h"

namespace lbm {

namespace {

template <int P>
__device__ double density_at(const LatticeDesc& d, int x, int y, int z) {
  using S = typename Storage<P>::S;
  using T = typename Storage<P>::T;
  const S* src = static_cast<const S*>(d.src);
  const T inv_scale = (T)(1.0 / d.scale);
  double sum = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xx = wrap(x - cx(i), d.nx), yy = wrap(y - cy(i), d.ny), zz = wrap(z - cz(i), d.nz);
    sum += widen(Storage<P>::load(src + (long long)i * d.plane + ((long long)zz * d.ny + yy) * d.nx + xx, inv_scale));
  }
  return d.n0 + sum;
}

// One warp per sampled node, a lane per stencil vector: a node's 19 densities of 19
// FP64 additions each would otherwise be one thread's chain (64 clocks an addition).
// Measured with lbm_observables at 128^3: 502 us a call, 563 with the lanes one by one.
template <int P, int ST>
__global__ void point_obs_kernel(LatticeDesc d, PointOut* pts, double* n_line, double* PT_line,
                                 double* PN_line, int line_len) {
  constexpr int R = stencil_radius<ST>();
  const int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (t >= 2 + line_len) return;
  const int c[3] = {d.nx / 2, d.ny / 2, d.nz / 2};
  int p[3];
  if (t == 0) {
    p[0] = c[0]; p[1] = c[1]; p[2] = c[2];
  } else if (t == 1) {
    p[0] = (c[0] + d.nx / 2) % d.nx;
    p[1] = (c[1] + d.ny / 2) % d.ny;
    p[2] = (c[2] + d.nz / 2) % d.nz;
  } else {
    p[0] = (c[0] + (t - 2)) % d.nx; p[1] = c[1]; p[2] = c[2];
  }
  // The stencil's vectors in raster order go to lanes 0 .. 30 in turn, the node itself
  // to lane 31.  Each lane finds its vector first, so that a round's densities are
  // formed by all lanes at once.
  double n = 0.0, psic = 0.0, sxx = 0.0, syy = 0.0;
  int total = 0;
  for (int round = 0; round == 0 || round * 31 < total; ++round) {
    int v[3] = {0, 0, 0}, count = 0;
    double W = 0.0;
    bool has = lane == 31 && round == 0;
#pragma unroll
    for (int dz = -R; dz <= R; ++dz)
#pragma unroll
      for (int dy = -R; dy <= R; ++dy)
#pragma unroll
        for (int dx = -R; dx <= R; ++dx) {
          const int m2 = dx * dx + dy * dy + dz * dz;
          if (m2 == 0 || shell_weight<ST>(m2) == 0.0) continue;
          if (lane < 31 && count == round * 31 + lane) {
            v[0] = dx; v[1] = dy; v[2] = dz;
            W = shell_weight<ST>(m2);
            has = true;
          }
          ++count;
        }
    total = count;
    if (has) {
      const double nb = density_at<P>(d, wrap(p[0] + v[0], d.nx), wrap(p[1] + v[1], d.ny), wrap(p[2] + v[2], d.nz));
      const double ps = psi_of<double>(nb, d.eos);
      if (lane == 31) {
        n = nb;
        psic = ps;
      } else {
        sxx += W * ps * (double)(v[0] * v[0]);
        syy += W * ps * (double)(v[1] * v[1]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sxx += __shfl_xor_sync(0xffffffffu, sxx, o);
    syy += __shfl_xor_sync(0xffffffffu, syy, o);
  }
  if (lane != 31) return;
  const double k = 0.5 * d.eos.G * (1.0 / 3.0) * psic;
  const double Pxx = n * (1.0 / 3.0) + k * sxx;
  const double Pyy = n * (1.0 / 3.0) + k * syy;
  if (t == 0) { pts->n_in = n; pts->P_in = Pxx; }
  else if (t == 1) { pts->n_out = n; pts->P_out = Pxx; }
  else { n_line[t - 2] = n; PT_line[t - 2] = Pyy; PN_line[t - 2] = Pxx; }
}

__global__ void finalize_kernel(FinalizeArgs a) {
  constexpr int NT = 256;
  __shared__ double red[8][NT];
  const int t = threadIdx.x;
  double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // mass, wsum, wd0, wd1, wd2, du, bad, max_u
  for (long long k = t; k < a.n_partials; k += NT) {
    const FieldPartial& p = a.partials[k];
    s[0] += p.mass; s[1] += p.wsum; s[2] += p.wd[0]; s[3] += p.wd[1]; s[4] += p.wd[2];
    s[5] += p.du; s[6] += p.bad; s[7] = fmax(s[7], p.max_u);
  }
  for (int q = 0; q < 8; ++q) red[q][t] = s[q];
  __syncthreads();
  for (int off = NT / 2; off > 0; off >>= 1) {
    if (t < off) {
      for (int q = 0; q < 7; ++q) red[q][t] += red[q][t + off];
      red[7][t] = fmax(red[7][t], red[7][t + off]);
    }
    __syncthreads();
  }
  // trapezoid rule on r = 0..line_len-1, and the closed forms in warps of their own:
  // one thread's FP64 chain is what this kernel's time is
  const PointOut pt = *a.pts;
  __shared__ double line[2][NT], form[8];
  {
    double C = 0.0, D = 0.0;
    for (int r = t; r < a.line_len; r += NT) {
      const double g = pt.P_out - a.PT_line[r];
      const double wt = (r == 0 || r == a.line_len - 1) ? 0.5 : 1.0;
      C += wt * (double)r * (double)r * g;
      D += wt * (double)r * g;
    }
    line[0][t] = C;
    line[1][t] = D;
  }
  __syncthreads();
  for (int off = NT / 2; off > 0; off >>= 1) {
    if (t < off) {
      line[0][t] += line[0][t + off];
      line[1][t] += line[1][t + off];
    }
    __syncthreads();
  }
  const double V = (double)a.volume, dP = pt.P_in - pt.P_out;
  const double q = (dP != 0.0) ? line[0][0] / dP : -1.0;
  // centre of mass of n - n_out: mean minimum-image displacement
  if (t == 0 || t == 32 || t == 64) form[t / 32] = red[2 + t / 32][0] / red[1][0];
  if (t == 96) form[3] = cbrt(3.0 * (red[0][0] - V * pt.n_out) / (4.0 * M_PI * (pt.n_in - pt.n_out)));
  if (t == 128) form[4] = q > 0.0 ? cbrt(6.0 * q) : NAN;
  __syncthreads();
  if (t != 0) return;
  lbm_obs o;
  o.n_in = pt.n_in;
  o.n_out = pt.n_out;
  o.P_in = pt.P_in;
  o.P_out = pt.P_out;
  o.dP = dP;
  o.mass = red[0][0];
  const double rel[3] = {form[0], form[1], form[2]};
  for (int k = 0; k < 3; ++k) o.com[k] = (double)a.center[k] + rel[k];
  o.R_e = form[3];
  o.C = line[0][0];
  o.D = line[1][0];
  unsigned st = 0;
  if (q > 0.0) {
    o.R_s = form[4];
    o.sigma_s = 0.5 * o.dP * o.R_s;
  } else {
    o.R_s = NAN;
    o.sigma_s = NAN;
    st |= 1u;
  }
  if (a.contrast0 > 0.0 && fabs(o.n_in - o.n_out) < 1e-2 * a.contrast0) st |= 2u;
  for (int k = 0; k < 3; ++k)
    if (!(fabs(rel[k]) <= 1e-3)) st |= 4u;
  if (red[6][0] > 0.0 || !isfinite(o.mass)) st |= 8u;
  if (a.err && *a.err) st |= 16u;
  o.max_u = red[7][0];
  o.du = a.have_u_old ? red[5][0] / V : 0.0;
  const double prev = *a.dP_prev;
  o.dP_rel_change = isnan(prev) ? NAN : fabs(o.dP - prev) / fabs(prev);
  *a.dP_prev = o.dP;
  o.steps = a.steps;
  o.status_bits = st;
  o.criterion = 0;
  *static_cast<lbm_obs*>(a.obs_out) = o;
}

}  // namespace

cudaError_t launch_point_obs(int prec, int stencil, const LatticeDesc& d, PointOut* pts,
                             double* n_line, double* PT_line, double* PN_line, cudaStream_t s) {
  const int line_len = d.nx / 2 + 1;
  const int n = 2 + line_len;
  const dim3 grid((n + 1) / 2);   // two warps a block
#define LBM_POINT(PR, STC) \
  point_obs_kernel<PR, STC><<<grid, 64, 0, s>>>(d, pts, n_line, PT_line, PN_line, line_len)
  if (stencil != 4 && stencil != 6 && stencil != 8) return cudaErrorInvalidValue;
  switch (prec) {
    case kF64: if (stencil == 4) LBM_POINT(kF64, 4); else if (stencil == 6) LBM_POINT(kF64, 6); else LBM_POINT(kF64, 8); break;
    case kF32: if (stencil == 4) LBM_POINT(kF32, 4); else if (stencil == 6) LBM_POINT(kF32, 6); else LBM_POINT(kF32, 8); break;
    case kF16: if (stencil == 4) LBM_POINT(kF16, 4); else if (stencil == 6) LBM_POINT(kF16, 6); else LBM_POINT(kF16, 8); break;
    default: return cudaErrorInvalidValue;
  }
#undef LBM_POINT
  return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeArgs& a, cudaStream_t s) {
  finalize_kernel<<<1, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace lbm
