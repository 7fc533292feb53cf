// Arithmetic of one node, written once for scalar (double, float) and packed
// (float2: two nodes) operands.
//
// Every multiply-add is an explicit fused operation and every other operation an
// explicitly rounded one, so the compiler has no contraction to choose and each
// kernel kind -- scalar or packed -- forms bitwise the same values.
#pragma once

#include "lbm_common.cuh"

namespace lbm {

__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
// a - b = b (-1) + a: exactly the rounding of the subtraction
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }

template <typename V> struct Lane { using T = V; static __device__ __forceinline__ V all(T x) { return x; } };
template <> struct Lane<float2> {
  using T = float;
  static __device__ __forceinline__ float2 all(float x) { return make_float2(x, x); }
};

// 1/n to within an ulp of the division: the hardware's approximate reciprocal y
// (relative error e = 1 - n y of 2^-23 in FP32, about 2^-20 in FP64) and one
// Newton-Raphson correction y (1 + e) in FP32 (the rest is e^2), the third-order one
// y (1 + e + e^2) in FP64 (the rest is e^3).  An IEEE division costs three times the
// instructions.  For normal n with a normal reciprocal; of 0 and of infinities it
// makes NaN, as the collision of such a node does anyhow (n u.u is 0 times infinity).
__device__ __forceinline__ float vrcp(float n) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(n));
  return __fmaf_rn(y, __fmaf_rn(-n, y, 1.0f), y);
}
__device__ __forceinline__ double vrcp(double n) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(n));
  const double e = __fma_rn(-n, y, 1.0);
  return __fma_rn(y, __fma_rn(e, e, e), y);
}
__device__ __forceinline__ float2 vrcp(float2 n) { return make_float2(vrcp(n.x), vrcp(n.y)); }

// ---------------------------------------------------------------- sums over the populations
// Mirror-exact summation.  The box, the droplet and its initial profile are
// symmetric under the three reflections x -> -x, y -> -y, z -> -z about the centre
// node, and so is the exact dynamics; floating-point sums keep that symmetry only
// if each reflection maps every sum onto the same operations.  A reflection
// permutes the populations (x: 1<->2, 7<->10, 8<->9, 11<->14, 12<->13; y: 3<->4,
// 7<->9, 8<->10, 15<->18, 16<->17; z: 5<->6, 11<->13, 12<->14, 15<->17, 16<->18), so
// the sums below add opposite pairs first and then exactly the pair sums a
// reflection swaps; a + b = b + a and a - b = -(b - a) hold exactly, so a mirrored
// state gives bitwise mirrored densities, momenta and forces, the drop's centre of
// mass stays on the centre node, and rounding (FP16 storage above all) cannot push
// the drop off it.
//
// sum of the nine opposite-pair sums g_i + g_ibar, grouped by the reflections
template <typename V>
__device__ __forceinline__ V pair_sum9(V p12, V p34, V p56, V p78, V p910, V p1112, V p1314, V p1516, V p1718) {
  return vadd(vadd(vadd(p12, p34), p56), vadd(vadd(vadd(p78, p910), vadd(p1112, p1314)), vadd(p1516, p1718)));
}

// density: rest population plus the mirror-exact sum of the pair sums (the order
// is fixed, so every kernel forms bitwise the same density)
template <typename V>
__device__ __forceinline__ V sum19(const V* v) {
  return vadd(v[0], pair_sum9<V>(vadd(v[1], v[2]), vadd(v[3], v[4]), vadd(v[5], v[6]), vadd(v[7], v[8]),
                                 vadd(v[9], v[10]), vadd(v[11], v[12]), vadd(v[13], v[14]), vadd(v[15], v[16]),
                                 vadd(v[17], v[18])));
}

// density and momentum of one node: momentum from the differences of the nine
// opposite pairs (1,2), (3,4), ..., (17,18) of the population order
template <typename V>
__device__ __forceinline__ void moments(const V* g, V& dn, V& jx, V& jy, V& jz) {
  dn = sum19(g);
  const V d12 = vsub(g[1], g[2]), d34 = vsub(g[3], g[4]), d56 = vsub(g[5], g[6]);
  const V d78 = vsub(g[7], g[8]), d910 = vsub(g[9], g[10]), d1112 = vsub(g[11], g[12]);
  const V d1314 = vsub(g[13], g[14]), d1516 = vsub(g[15], g[16]), d1718 = vsub(g[17], g[18]);
  // x: 1 (+), 7 (+), 9 (+), 11 (+), 13 (+); y: 3, 7, 10, 15, 17 (+); z: 5, 11, 14, 15, 18 (+);
  // the differences a reflection swaps are added (or subtracted) first: mirror-exact
  jx = vadd(vadd(d12, vadd(d78, d910)), vadd(d1112, d1314));
  jy = vadd(vadd(d34, vsub(d78, d910)), vadd(d1516, d1718));
  jz = vadd(vadd(d56, vsub(d1112, d1314)), vsub(d1516, d1718));
}

// ---------------------------------------------------------------- stencils
// Shell weights W(|xi|^2) of the forcing stencils (Sec. II; the wider stencils
// are the isotropic ones the paper cites) as integers over one denominator:
// E4 W = 1/6, 1/12; E6 2/15, 1/15, 1/60, 1/120; E8 4/45, 1/21, 2/105, 5/504,
// 1/315, 1/630, 1/5040.  0 where a vector is not used.
template <int ST>
__host__ __device__ constexpr int shell_int(int s) {
  if (ST == 4) return s == 1 ? 2 : (s == 2 ? 1 : 0);
  if (ST == 6) return s == 1 ? 16 : s == 2 ? 8 : s == 3 ? 2 : s == 4 ? 1 : 0;
  return s == 1 ? 448 : s == 2 ? 240 : s == 3 ? 96 : s == 4 ? 50 : s == 5 ? 16 : s == 6 ? 8 : s == 8 ? 1 : 0;
}
template <int ST>
__host__ __device__ constexpr double shell_denominator() { return ST == 4 ? 12.0 : (ST == 6 ? 120.0 : 5040.0); }
template <int ST>
__host__ __device__ constexpr double shell_weight(int s) { return shell_int<ST>(s) / shell_denominator<ST>(); }
template <int ST> constexpr int stencil_radius() { return ST == 4 ? 1 : 2; }

// Shan-Chen force (Eq. (8)); at(dx, dy, dz) is psi at that offset from the node.
// The stencil is summed through the differences D(xi) = psi(x + xi) -
// psi(x - xi), so that two psi values cancel before they are scaled: a uniform
// region gives exactly F = 0 and the rounding error scales with F, not with the
// psi values.  (Summing the 18 terms one by one in raster order lets FP32 rounding
// build a spurious force that grows the density error of a 1000-step droplet run
// tenfold.)
// Mirror-exact order: component a of the force is, per shell, a sum over the
// orbits of the stencil vectors with xi_a > 0 under the two reflections that
// leave axis a alone -- {(xi_a, +-b, +-c)} -- each orbit summed as
// ((D(a,b,c) + D(a,-b,c)) + (D(a,b,-c) + D(a,-b,-c))); the shells are then
// weighted by their integers and added in a fixed order.  A reflection of the
// field maps every orbit sum onto itself (reordered by exactly commuting
// additions) or onto its negative, so mirrored psi gives a bitwise mirrored force.
template <typename V, int ST, typename At>
__device__ __forceinline__ V sc_force_axis(At at, int axis) {
  using L = Lane<V>;
  constexpr int R = stencil_radius<ST>();
  V F = L::all(0);
  bool any_shell = false;
#pragma unroll
  for (int sh = 3 * R * R; sh >= 1; --sh) {   // the outermost shell has weight 1
    const int W = shell_int<ST>(sh);
    if (W == 0) continue;
    V S = L::all(0);
    bool any = false;
#pragma unroll
    for (int a = 1; a <= R; ++a) {
#pragma unroll
      for (int b = 0; b <= R; ++b) {
#pragma unroll
        for (int c = 0; c <= R; ++c) {
          if (a * a + b * b + c * c != sh) continue;
          // the vector (a, b, c) in the frame of `axis`: a along it, b and c along the
          // other two axes in increasing order
          auto D = [&](int bb, int cc) {
            return axis == 0 ? vsub(at(a, bb, cc), at(-a, -bb, -cc))
                 : axis == 1 ? vsub(at(bb, a, cc), at(-bb, -a, -cc))
                             : vsub(at(bb, cc, a), at(-bb, -cc, -a));
          };
          V O;
          if (b > 0 && c > 0) O = vadd(vadd(D(b, c), D(-b, c)), vadd(D(b, -c), D(-b, -c)));
          else if (b > 0) O = vadd(D(b, 0), D(-b, 0));
          else if (c > 0) O = vadd(D(0, c), D(0, -c));
          else O = D(0, 0);
          if (a != 1) O = vadd(O, O);   // a = 2
          S = any ? vadd(S, O) : O;
          any = true;
        }
      }
    }
    if (!any) continue;
    F = any_shell ? vfma(L::all(W), S, F) : (W == 1 ? S : vmul(L::all(W), S));
    any_shell = true;
  }
  return F;
}

template <typename V, int ST, typename At>
__device__ __forceinline__ void sc_force_at(At at, V psi0, Coupling<typename Lane<V>::T> cpl, V& Fx, V& Fy, V& Fz) {
  using T = typename Lane<V>::T;
  V k;
  if constexpr (sizeof(T) == 4) {
    // FP32: in two floats, one rounding.  One float is a G off by up to 1e-7 at every node
    // and step, which the interface amplifies (48x40x44 bubble, G -4.6, 160 steps:
    // populations off by 2.3e-5, now 2.9e-6).
    constexpr int i = ST == 4 ? 0 : (ST == 6 ? 1 : 2);
    k = vfma(Lane<V>::all(cpl.e.Khi[i]), psi0, vmul(Lane<V>::all(cpl.e.Klo[i]), psi0));
  } else {
    k = vmul(Lane<V>::all(-cpl.e.G * (T)(1.0 / (3.0 * shell_denominator<ST>()))), psi0);
  }
  Fx = vmul(k, sc_force_axis<V, ST>(at, 0));
  Fy = vmul(k, sc_force_axis<V, ST>(at, 1));
  Fz = vmul(k, sc_force_axis<V, ST>(at, 2));
}

// ---------------------------------------------------------------- collision
// BGK + Guo collision of one node in shifted form, g_i = f_i - w_i n0:
//   g*_i = (1 - omega) g_i + omega g_i^eq + F_i
//   g_i^eq = w_i [dn + n (3 e.u + 9/2 (e.u)^2 - 3/2 u.u)]          Eq. (6)
//   F_i    = (1 - omega/2) w_i [3 e.F + 9 (e.u)(e.F) - 3 u.F]       Eq. (5)
// With n u = j + F/2 (Eq. (7)) the equilibrium and the force terms combine:
//   q = omega j + (2 - omega/2) F,   p = omega j + F,
//   base = omega dn - 3/2 u.q,
//   omega g_i^eq + F_i = w_i [base + 9/2 (e.u)(e.q) + 3 e.p],
// which takes half the operations of forming g_i^eq and F_i one by one (the FP64
// step is bound by its FP64 instructions and the FP16 step by instruction issue).
// Scaled to the diagonal weight 1/36: B = base/36, U = u/8, P = p/36; an axis
// population is twice [B + U_a q_a +- 3 P_a].  (P = p/12 would scale every momentum by
// the error of 1/12 in FP32, 3.0e-8, four times that of 1/36.)  Opposite velocities share the even
// part; the odd part flips sign.
//
// Mass closure: sum g*_i = dn holds exactly for exact weights, but the rounded
// ones do not sum to exactly 1 (FP32: 1 + 1.5e-8), which would add a systematic
// error proportional to n - n0 to every node every step; the rest population is
// set to dn - sum_{i>0} g*_i instead (the same value in exact arithmetic; the
// pair sums without their odd parts, which cancel), so mass changes only by
// uncorrelated rounding.
// UNIT: omega = 1 (tau = 1, the relaxation time the method uses); then old(i) is
// never read.  SCALED: the outputs come multiplied by wscale, a power of two
// (FP16 storage's 2^k), which commutes with every rounding.
// old(i): population i before the collision; store(i, g): takes g*_i.
template <typename V, bool UNIT, bool SCALED, typename Old, typename Store>
__device__ __forceinline__ void collide_nodes(V dn, V n, V jx, V jy, V jz, V Fx, V Fy, V Fz,
                                              typename Lane<V>::T omega, typename Lane<V>::T wscale, Old old,
                                              Store store) {
  using T = typename Lane<V>::T;
  using L = Lane<V>;
  const V inv_n = vrcp(n);
  const V half = L::all((T)0.5);
  const V ux = vmul(vfma(half, Fx, jx), inv_n);
  const V uy = vmul(vfma(half, Fy, jy), inv_n);
  const V uz = vmul(vfma(half, Fz, jz), inv_n);
  const T om1 = (T)1 - omega;
  const V cq = L::all(UNIT ? (T)1.5 : (T)2 - (T)0.5 * omega);
  V qx, qy, qz, px, py, pz, base;
  if (UNIT) {
    qx = vfma(cq, Fx, jx); qy = vfma(cq, Fy, jy); qz = vfma(cq, Fz, jz);
    px = vadd(jx, Fx); py = vadd(jy, Fy); pz = vadd(jz, Fz);
    base = dn;
  } else {
    const V om = L::all(omega);
    const V kx = vmul(om, jx), ky = vmul(om, jy), kz = vmul(om, jz);
    qx = vfma(cq, Fx, kx); qy = vfma(cq, Fy, ky); qz = vfma(cq, Fz, kz);
    px = vadd(kx, Fx); py = vadd(ky, Fy); pz = vadd(kz, Fz);
    base = vmul(om, dn);
  }
  const V uq = vfma(uz, qz, vfma(uy, qy, vmul(ux, qx)));
  base = vfma(L::all((T)-1.5), uq, base);
  const T s = SCALED ? wscale : (T)1;
  const V c8 = L::all((T)0.125 * s), c36 = L::all((T)(1.0 / 36.0) * s);
  const V B = vmul(base, c36);
  const V Ux = vmul(ux, c8), Uy = vmul(uy, c8), Uz = vmul(uz, c8);
  px = vmul(px, c36); py = vmul(py, c36); pz = vmul(pz, c36);
  const V two = L::all((T)2), three = L::all((T)3), six = L::all((T)6), vom1 = L::all(om1);
  // One opposite pair: g*_i, g*_{i+1} and its even part ev (an axis pair: twice the
  // diagonal one, formed with one fused operation each).  Without omega = 1 the old
  // populations' share is added, and the pair's sum (2 ev, or 4 ev for an axis) takes
  // theirs; with om1 = 0 that adds nothing, so both forms agree bitwise.
  auto pair = [&](int i, V ga, V gb, V ev, T ev_mul) {
    if (UNIT) {
      store(i, ga);
      store(i + 1, gb);
      return ev;
    } else {
      const V a = old(i), b = old(i + 1);
      store(i, vfma(vom1, a, ga));
      store(i + 1, vfma(vom1, b, gb));
      return vfma(vom1, vadd(a, b), vmul(L::all(ev_mul), ev));
    }
  };
  auto axis = [&](int i, V U, V q, V P) {
    const V ev = vfma(U, q, B), P2 = vmul(six, P);
    return pair(i, vfma(two, ev, P2), vsub(vadd(ev, ev), P2), ev, (T)4);
  };
  auto diag = [&](int i, V U, V q, V P) {
    const V ev = vfma(U, q, B);
    return pair(i, vfma(three, P, ev), vfma(L::all((T)-3), P, ev), ev, (T)2);
  };
  const V a12 = axis(1, Ux, qx, px), a34 = axis(3, Uy, qy, py), a56 = axis(5, Uz, qz, pz);
  const V d78 = diag(7, vadd(Ux, Uy), vadd(qx, qy), vadd(px, py));
  const V d910 = diag(9, vsub(Ux, Uy), vsub(qx, qy), vsub(px, py));
  const V d1112 = diag(11, vadd(Ux, Uz), vadd(qx, qz), vadd(px, pz));
  const V d1314 = diag(13, vsub(Ux, Uz), vsub(qx, qz), vsub(px, pz));
  const V d1516 = diag(15, vadd(Uy, Uz), vadd(qy, qz), vadd(py, pz));
  const V d1718 = diag(17, vsub(Uy, Uz), vsub(qy, qz), vsub(py, pz));
  const V A = vadd(vadd(a12, a34), a56);
  const V D = vadd(vadd(vadd(d78, d910), vadd(d1112, d1314)), vadd(d1516, d1718));
  const V rest = SCALED ? vmul(dn, L::all(s)) : dn;
  store(0, UNIT ? vfma(L::all((T)-2), vfma(two, A, D), rest) : vsub(rest, vadd(A, D)));
}

// the same for a node's populations in an array
template <typename T, bool UNIT = false, bool SCALED = false>
__device__ __forceinline__ void collide(T* g, T dn, T n, T jx, T jy, T jz, T Fx, T Fy, T Fz, T omega,
                                        T wscale = (T)1) {
  collide_nodes<T, UNIT, SCALED>(dn, n, jx, jy, jz, Fx, Fy, Fz, omega, wscale, [&](int i) { return g[i]; },
                                 [&](int i, T v) { g[i] = v; });
}

}  // namespace lbm
