// Unit-tau Shan-Chen step on whole rows, fed by bulk copies (cp.async.bulk).
//
// The moment kernel's scheme (lbm_kernels_moment.cuh) -- at tau = 1 a collision
// needs a node's populations only through n and j, so a plane's stage is free as
// soon as its densities are formed -- with another tile, other copies and several
// nodes per thread:
//
//  * A CTA owns `by` whole rows (all of x) and marches through z.  The padded rows
//    y0 - R .. y0 + by + R of one population and plane are then ONE contiguous block
//    of memory, copied by one cp.async.bulk (two where the block wraps around the
//    box in y).  A bulk copy costs the SM about 70 clocks whatever its size up to
//    1 KB and reaches the full HBM rate from 2 KB on (measured: 160 B 0.73, 544 B
//    2.4, 1 KB 4.3, 2 KB and more 7.1-7.3 TB/s over 152 SMs), so blocks of rows are
//    what it wants; tiles of 32 x 8 nodes would need 190 small copies a plane.  There
//    is no x halo, and the x wrap is an index offset on chip.
//  * Nodes are numbered flat within the plane's block (j = row * nx + x): lanes take
//    consecutive nodes whatever nx is, every shared-memory access is conflict-free,
//    the interior is one contiguous block of global memory, and odd boxes (the
//    paper's own) run like even ones.  Rows that are no whole number of 16 bytes:
//    a block's copy is widened to 16-byte boundaries and its elements sit in the
//    slot at their own alignment (see `shift`).
//  * A thread takes two nodes at a time, their arithmetic packed (FFMA2 and FADD2 of
//    sm_100 and later: two FP32 operations per instruction); the operations and
//    their order are those of the scalar kernels, so the fields are bitwise equal.
//  * Roles.  One producer warp issues the copies, density warps form n, j and psi of
//    the padded plane, collision warps collide the plane R behind; psi and the
//    moments pass through shared memory, one barrier of both per plane.  An SM's
//    stores go out at about 28 B/clk (measured), so a plane's collision waits for its
//    own stores; in warps of their own it does so while the next densities form (one
//    set of warps doing both in turn: 256^3 475 us a step, against 395).
//  * The populations are staged once (no second stage) in four groups with a full /
//    empty mbarrier pair each: a group's slots are refilled with the next plane as
//    soon as every density warp has read them, so nearly a whole stage is in flight.
//
// What bounds it: HBM from 128^3 nodes on in FP32 with aligned rows (256^3: 375 us a
// step, 1.00 of the measured copy rate; 192^3 171 us, 0.92; the moment kernel 481 and
// 214); an SM's own time per plane (loads and stores of shared memory, latency) for
// FP16 (192^3 96.5 us, 0.82; 154.9) and unaligned rows (157^3 100 us, 0.87; 142);
// the step's latency below 100^3 (96^3 22.1 us; 30.3).
// What did not help: four x-neighbours a thread with 16-byte accesses (128^3 67 us
// against 54: bank conflicts of their outer neighbours, half the warps), two CTAs of
// half the size per SM, a second stage, stores through bulk copies (18 B/clk).
//
// Bounded waits: a wait that gives up after kTmaPolls polls sets a flag in shared
// memory, at which every later wait of the CTA gives up at once; the loops run to
// their end (so no barrier is left waiting), the producer issues nothing more and
// waits (bounded) for the copies it has in flight, and *d.err is set.
#pragma once

#include "lbm_kernels_tma.cuh"
#include "lbm_launch.h"

namespace lbm {

constexpr int kRowGroups = 4;
constexpr int kRowDead = 248;   // byte of the give-up flag (behind the mbarriers)
// populations of group g: [row_group_first(g), row_group_first(g + 1))
__host__ __device__ constexpr int row_group_first(int g) { return g == 0 ? 0 : (g == 1 ? 7 : (g == 2 ? 11 : (g == 3 ? 15 : Q))); }

// Shared memory of one row CTA (row_caps gives SLOT, MCAP and KD per storage).
template <int P_>
struct RowShape {
  static constexpr int P = P_, ST = 4;
  using T = typename Storage<P>::T;
  using S = typename Storage<P>::S;
  static constexpr int R = stencil_radius<ST>();
  static constexpr RowCaps caps = row_caps(P);
  static constexpr int SLOT = caps.slot;                   // elements of one population's slot
  static constexpr int MCAP = caps.mcap;                   // interior nodes of an item at most
  static constexpr int KD = caps.kd;                       // packed operands a density thread takes
  static constexpr bool PAIRS = P == kF16;                 // operands are x-neighbours where rows are aligned
  static constexpr int VE = 16 / (int)sizeof(S);
  static constexpr int NR = 2 * R + 2;                     // psi planes in the ring
  static constexpr int NM = R + 2;                         // planes of moments
  static constexpr int PW = 2;                             // nodes of a packed operand
  static constexpr unsigned head_bytes = 256;              // mbarriers, the give-up flag
  static constexpr unsigned stage_bytes = (unsigned)sizeof(S) * Q * SLOT;
  static constexpr unsigned ring_off = head_bytes + stage_bytes;
  static constexpr unsigned ring_bytes = (unsigned)sizeof(T) * SLOT;   // a psi plane
  static constexpr unsigned mom_off = ring_off + NR * ring_bytes;
  static constexpr unsigned comp_bytes = (unsigned)sizeof(T) * MCAP;
  static constexpr unsigned mom_bytes = 4 * comp_bytes;
  // (and what a collision thread reads of a second node past the item's last one)
  static constexpr size_t smem_bytes = mom_off + NM * mom_bytes + 32 * sizeof(T);
  static_assert(SLOT % VE == 0 && SLOT % 4 == 0 && MCAP % 4 == 0, "slots, ring and moments start on 16 bytes");
  static_assert(smem_bytes <= kMaxSmemPerCta, "one CTA per SM");
};

__device__ __forceinline__ float row_node(float2 v, int w) { return w == 0 ? v.x : v.y; }

__device__ __forceinline__ void row_bulk_copy(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   tma_smem(dst)),
               "l"(src), "r"(bytes), "r"(tma_smem(bar))
               : "memory");
}
__device__ __forceinline__ void row_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tma_smem(bar)) : "memory");
}
__device__ __forceinline__ void row_barrier(int threads) {   // the consumer warps
  asm volatile("bar.sync 1, %0;\n" ::"r"(threads) : "memory");
}
// wait for the phase of parity `par` ;
// gives up after kTmaPolls polls or once another wait of the CTA has
__device__ __forceinline__ bool row_try(unsigned long long* bar, unsigned par) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(tma_smem(bar)), "r"(par)
      : "memory");
  return ok != 0;
}
static __device__ __noinline__ void row_wait_long(unsigned long long* bar, unsigned par, volatile int* dead) {
  for (int k = 0; k < kTmaPolls; ++k) {
    if (row_try(bar, par)) return;
    if ((k & 15) == 15 && *dead) return;
  }
  *dead = 1;
}
__device__ __forceinline__ void row_wait(unsigned long long* bar, unsigned par, volatile int* dead) {
  if (!row_try(bar, par)) row_wait_long(bar, par, dead);
}

template <typename X>
__device__ __forceinline__ X row_ld(const unsigned char* smem, unsigned off) {
  return *reinterpret_cast<const X*>(smem + off);
}
// two stored values that lie side by side, aligned, as a packed operand
template <int P>
__device__ __forceinline__ float2 row_ld_pair(const unsigned char* smem, unsigned off) {
  if constexpr (P == kF16) return __half22float2(row_ld<__half2>(smem, off));
  else return row_ld<float2>(smem, off);
}

// The nodes a thread takes at a time: one packed operand of two.
// A padded plane's nodes are numbered flat, j = row nx + x, in the population slots,
// the psi planes and (interior nodes) the moments alike.
//  * PAIR (aligned rows): two x-neighbours at an even x;
//  * else nodes j and j + 32: a warp reads 32 consecutive words whatever nx is.
template <class Sh, bool ALIGNED>
struct RowNodes {
  static constexpr int P = Sh::P;
  using T = typename Sh::T;
  using S = typename Sh::S;
  static constexpr int PW = Sh::PW, R = Sh::R;
  static constexpr bool PAIR = ALIGNED && Sh::PAIRS;
  static constexpr int NEXT = PAIR ? 1 : 32;    // second node's distance from the first
  static constexpr int NL = PAIR ? 1 : PW;
  int j;               // first node
  int l[NL], r[NL];    // x-neighbours: left and right of each node (PAIR: left of the first, right of the second)

  // flat index of the first node of a thread's t-th unit, t consecutive over a warp
  static __device__ __forceinline__ int first(int t) {
    return PAIR ? 2 * t : (t & ~31) * 2 + (t & 31);
  }
  __device__ __forceinline__ void set(int j0, int nx) {
    j = j0;
#pragma unroll
    for (int w = 0; w < NL; ++w) {
      const int jw = j0 + w * NEXT, x = jw % nx;
      l[w] = jw + (x == 0 ? nx - 1 : -1);
      r[w] = PAIR ? jw + (x + 2 == nx ? -x : 2) : jw + (x == nx - 1 ? 1 - nx : 1);
    }
  }
  // node w's x-neighbour at dx = -1, 0, 1
  __device__ __forceinline__ int at(int w, int dx) const {
    if constexpr (PAIR) return dx == 0 ? j + w : (dx < 0 ? (w == 0 ? l[0] : j) : (w == 0 ? j + 1 : r[0]));
    else return dx == 0 ? j + w * NEXT : (dx < 0 ? l[w] : r[w]);
  }
};

// psi of a packed density, one branch on its kind
__device__ __forceinline__ float2 row_psi(float2 n, const EosParams& e) {
  EosParams k = e;
  auto both = [&](int kind) {
    k.kind = kind;
    return make_float2(psi_of<float>(n.x, k), psi_of<float>(n.y, k));
  };
  if (e.kind == kPsiOneMinusExp) return both(kPsiOneMinusExp);
  if (e.kind == kPsiExpInv) return both(kPsiExpInv);
  return both(kPsiCS);
}

// One item: rows [y0, y0 + h), planes [z0, z0 + zc) of lattice d, walked upwards
// (flip: downwards).  `uses` counts the planes staged so far by this CTA; stages,
// psi planes and moment planes are taken in turn by it, across items.
template <class Sh, bool ALIGNED>
__device__ __forceinline__ void row_process_item(const LatticeDesc& d, const RowCfg& c, int item, bool flip,
                                                 unsigned char* smem, unsigned& uses) {
  using N = RowNodes<Sh, ALIGNED>;
  using T = typename Sh::T;
  using S = typename Sh::S;
  using V = float2;
  constexpr int P = Sh::P, R = Sh::R, PW = Sh::PW, VE = Sh::VE, SLOT = Sh::SLOT;
  unsigned long long* full = reinterpret_cast<unsigned long long*>(smem);
  unsigned long long* empty = full + kRowGroups;
  volatile int* dead = reinterpret_cast<volatile int*>(smem + kRowDead);

  const int nx = d.nx, ny = d.ny, nz = d.nz;
  const int ncols = (ny + c.by - 1) / c.by;
  const int y0 = (item % ncols) * c.by, z0 = (item / ncols) * c.zc;
  const int h = min(c.by, ny - y0), zc = min(c.zc, nz - z0);
  const int nplanes = zc + 2 * R, rows = h + 2 * R;
  const int tid = threadIdx.x;
  auto plane_z = [&](int q) { return wrap(flip ? z0 + zc - 1 + R - q : z0 - R + q, nz); };
  // the block of a population with this c_y starts with source row first_row(c_y)
  auto first_row = [&](int cyi) { return wrap(y0 - R - cyi, ny); };
  // unaligned rows: past the wrap in y a block's elements lie `delta` further on
  // than they would follow the others; delta makes the second copy's alignment come
  // out right and keeps the two widened copies apart
  const int delta = ALIGNED ? 0 : VE + (int)((-(long long)ny * nx) & (VE - 1));

  if (tid >= c.nd + c.nc) {   // producer warp: four lanes (wrap segments) per population of a group
    const int lane = tid & 31, seg = lane & 3;
    const S* src = static_cast<const S*>(d.src);
    S* const slots = reinterpret_cast<S*>(smem + Sh::head_bytes);
    const int pl = ny * nx;
    // this lane's copy of each group, as far as it does not depend on the plane: the
    // source element at z = 0, that of the block's first segment (unaligned rows), the
    // slot position and the number of elements.  Everything but z is out of the plane
    // loop: a producer that computes its addresses there is what the CTA waits for.
    long long e_at[kRowGroups], e_first[ALIGNED ? 1 : kRowGroups];
    int at[kRowGroups], len[kRowGroups], dz[kRowGroups];
    unsigned total[kRowGroups];
#pragma unroll
    for (int g = 0; g < kRowGroups; ++g) {
      const int i = row_group_first(g) + (lane >> 2);
      const bool mine = i < row_group_first(g + 1);
      const int cyi = mine ? cy_rt(i) : 0, y_first = first_row(cyi);
      int y = y_first, r0 = 0, n = min(rows, ny - y);
      for (int s = 0; s < seg; ++s) { r0 += n; y = 0; n = min(rows - r0, ny); }
      dz[g] = mine ? cz_rt(i) : 0;
      e_at[g] = (long long)i * d.plane + (long long)y * nx;
      len[g] = mine ? n * nx : 0;
      at[g] = i * SLOT + r0 * nx + (ALIGNED || seg == 0 ? 0 : delta);
      if constexpr (ALIGNED) total[g] = __reduce_add_sync(0xffffffffu, (unsigned)(len[g] * (int)sizeof(S)));
      else e_first[g] = (long long)i * d.plane + (long long)y_first * nx;
    }
#pragma unroll 1
    for (int q = 0; q < nplanes; ++q) {
      if (__any_sync(0xffffffffu, *dead != 0)) {   // nothing more is issued; `uses` keeps what was
        uses += q;
        return;
      }
      const int z = plane_z(q);
      const int zo[3] = {wrap(z + 1, nz) * pl, z * pl, wrap(z - 1, nz) * pl};   // for c_z = -1, 0, +1
      const unsigned use = uses + q;
#pragma unroll
      for (int g = 0; g < kRowGroups; ++g) {
        long long e = e_at[g] + (dz[g] < 0 ? zo[0] : (dz[g] > 0 ? zo[2] : zo[1]));
        int pos = at[g];
        unsigned bytes = (unsigned)(len[g] * (int)sizeof(S)), sum;
        if constexpr (ALIGNED) {
          sum = total[g];
        } else {   // widened to whole 16-byte pieces
          const int a = (int)(e & (VE - 1));
          pos += (int)((e - e_at[g] + e_first[g]) & (VE - 1)) - a;
          e -= a;
          bytes = len[g] > 0 ? (unsigned)((a + len[g] + VE - 1) / VE * 16) : 0u;
          sum = __reduce_add_sync(0xffffffffu, bytes);
        }
        unsigned long long* const bar = full + g;
        if (use > 0) row_wait(empty + g, (use - 1) & 1, dead);
        if (lane == 0) tma_mbar_expect(bar, sum);
        __syncwarp();
        if (bytes) row_bulk_copy(slots + pos, src + e, bytes, bar);
      }
    }
    uses += nplanes;
    return;
  }

  const int ncons = c.nd + c.nc;
  const T n0 = dparam<T>(d.n0, d.n0f);

  if (tid < c.nd) {   // density warps: n, psi and j of every node of the padded plane
    const T inv_scale = dparam<T>(1.0 / d.scale, d.inv_scalef);
    const bool lane0 = (tid & 31) == 0;
    const int nodes = rows * nx;
    constexpr int KD = Sh::KD;
    N nd[KD];
    unsigned dy[ALIGNED ? 1 : KD][PW][3];   // bytes past the wrap in y, for c_y = -1, 0, +1
    bool some[KD];                          // the warp has a node in this unit
    unsigned long long at0 = 0;             // unaligned rows: alignment of each block's first element at z = 0, 3 bits each
    if constexpr (!ALIGNED) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        at0 |= (unsigned long long)(((unsigned long long)i * (unsigned long long)d.plane +
                                     (unsigned long long)first_row(cy(i)) * nx) & (VE - 1)) << (3 * i);
    }
#pragma unroll
    for (int k = 0; k < KD; ++k) {
      const int f = N::first(tid + c.nd * k);
      some[k] = N::first((tid & ~31) + c.nd * k) < nodes;
      nd[k].set(f, nx);       // nodes past the plane's end read (unused) what lies there, in range
      if constexpr (!ALIGNED) {
#pragma unroll
        for (int w = 0; w < PW; ++w)
#pragma unroll
          for (int cyi = -1; cyi <= 1; ++cyi)
            dy[k][w][cyi + 1] = first_row(cyi) + (f + w * N::NEXT) / nx < ny ? 0u : (unsigned)(delta * (int)sizeof(S));
      }
    }
#pragma unroll 1
    for (int q = 0; q < nplanes; ++q) {
      const int z = plane_z(q);
      const unsigned use = uses + q;
      // unaligned rows: population i's block starts this many bytes into its slot
      unsigned zt[3] = {0, 0, 0};   // what plane z - c_z adds, for c_z = -1, 0, +1
      if constexpr (!ALIGNED) {
#pragma unroll
        for (int czi = -1; czi <= 1; ++czi)
          zt[czi + 1] = ((unsigned)wrap(z - czi, nz) * (unsigned)(ny * nx)) & (VE - 1);
      }
      auto shift = [&](int i) -> unsigned {
        if (ALIGNED) return 0u;
        return (((unsigned)(at0 >> (3 * i)) + zt[cz(i) + 1]) & (VE - 1)) * (unsigned)sizeof(S);
      };
      // population i pulled to the nodes of unit k
      auto load = [&](int i, int k) {
        const unsigned slot = Sh::head_bytes + (unsigned)(i * SLOT * (int)sizeof(S)) + shift(i);
        if constexpr (N::PAIR) {
          if (cx(i) == 0) return row_ld_pair<P>(smem, slot + (unsigned)(nd[k].j * (int)sizeof(S)));
        }
        T v[2] = {(T)0, (T)0};
#pragma unroll
        for (int w = 0; w < PW; ++w)
          v[w] = staged_value<P>(row_ld<S>(smem, slot + (unsigned)(nd[k].at(w, -cx(i)) * (int)sizeof(S)) +
                                                     (ALIGNED ? 0u : dy[ALIGNED ? 0 : k][w][cy(i) + 1])));
        return make_float2(v[0], v[1]);
      };
      auto wait = [&](int g) { row_wait(full + g, use & 1, dead); };
      auto done = [&](int g) {
        __syncwarp();
        if (lane0) row_arrive(empty + g);
      };
      // the sums of moments() (lbm_math.cuh), group by group as the copies arrive
      V v0[KD], A[KD], D[KD], jx[KD], jy[KD], jz[KD];
      wait(0);
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        if (!some[k]) continue;
        v0[k] = load(0, k);
        const V a1 = load(1, k), a2 = load(2, k), a3 = load(3, k), a4 = load(4, k), a5 = load(5, k), a6 = load(6, k);
        A[k] = vadd(vadd(vadd(a1, a2), vadd(a3, a4)), vadd(a5, a6));
        jx[k] = vsub(a1, a2);
        jy[k] = vsub(a3, a4);
        jz[k] = vsub(a5, a6);
      }
      done(0);
      wait(1);
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        if (!some[k]) continue;
        const V a = load(7, k), b = load(8, k), e = load(9, k), f = load(10, k);
        D[k] = vadd(vadd(a, b), vadd(e, f));
        const V d78 = vsub(a, b), d910 = vsub(e, f);
        jx[k] = vadd(jx[k], vadd(d78, d910));
        jy[k] = vadd(jy[k], vsub(d78, d910));
      }
      done(1);
      wait(2);
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        if (!some[k]) continue;
        const V a = load(11, k), b = load(12, k), e = load(13, k), f = load(14, k);
        D[k] = vadd(D[k], vadd(vadd(a, b), vadd(e, f)));
        const V d1112 = vsub(a, b), d1314 = vsub(e, f);
        jx[k] = vadd(jx[k], vadd(d1112, d1314));
        jz[k] = vadd(jz[k], vsub(d1112, d1314));
      }
      done(2);
      wait(3);
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        if (!some[k]) continue;
        const V a = load(15, k), b = load(16, k), e = load(17, k), f = load(18, k);
        D[k] = vadd(D[k], vadd(vadd(a, b), vadd(e, f)));
        const V d1516 = vsub(a, b), d1718 = vsub(e, f);
        jy[k] = vadd(jy[k], vadd(d1516, d1718));
        jz[k] = vadd(jz[k], vsub(d1516, d1718));
      }
      done(3);
      const unsigned ring = Sh::ring_off + (use % Sh::NR) * Sh::ring_bytes;
      const unsigned mq = Sh::mom_off + (use % Sh::NM) * Sh::mom_bytes;
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        if (!some[k]) continue;
        V dn = vadd(v0[k], vadd(A[k], D[k]));
        if constexpr (P == kF16) {   // the staged values are scaled by 2^k
          const V is = Lane<V>::all(inv_scale);
          dn = vmul(dn, is);
          jx[k] = vmul(jx[k], is);
          jy[k] = vmul(jy[k], is);
          jz[k] = vmul(jz[k], is);
        }
        const V psi = row_psi(vadd(Lane<V>::all(n0), dn), d.eos);
        const int f = nd[k].j, m = f - R * nx;     // m: interior index (halo rows keep psi only)
        if constexpr (N::PAIR) {   // a pair is whole: in the plane or not, interior or not
          if (f < nodes) *reinterpret_cast<V*>(smem + ring + (unsigned)(f * 4)) = psi;
          if (m >= 0 && m < h * nx) {
            unsigned char* const to = smem + mq + (unsigned)(m * 4);
            *reinterpret_cast<V*>(to) = dn;
            *reinterpret_cast<V*>(to + Sh::comp_bytes) = jx[k];
            *reinterpret_cast<V*>(to + 2 * Sh::comp_bytes) = jy[k];
            *reinterpret_cast<V*>(to + 3 * Sh::comp_bytes) = jz[k];
          }
        } else {
#pragma unroll
          for (int w = 0; w < PW; ++w) {
            if (f + w * N::NEXT >= nodes) continue;
            *reinterpret_cast<T*>(smem + ring + (unsigned)((f + w * N::NEXT) * (int)sizeof(T))) = row_node(psi, w);
            const int mw = m + w * N::NEXT;
            if (mw < 0 || mw >= h * nx) continue;
            unsigned char* const to = smem + mq + (unsigned)(mw * (int)sizeof(T));
            *reinterpret_cast<T*>(to) = row_node(dn, w);
            *reinterpret_cast<T*>(to + Sh::comp_bytes) = row_node(jx[k], w);
            *reinterpret_cast<T*>(to + 2 * Sh::comp_bytes) = row_node(jy[k], w);
            *reinterpret_cast<T*>(to + 3 * Sh::comp_bytes) = row_node(jz[k], w);
          }
        }
      }
      row_barrier(ncons);
    }
    uses += nplanes;
    return;
  }

  // collision warps
  const Coupling<T> G(d.eos);
  const T scale = dparam<T>(d.scale, d.scalef);
  const int tc = tid - c.nd;
  const int inner = h * nx;
  const long long pbytes = d.plane * (long long)sizeof(S);
  // which of the thread's nodes (unit u, node w: bit u PW + w) have wrapping x-neighbours
  unsigned lm = 0, rm = 0;
  {
    int u = 0;
    for (int f = N::first(tc); f < inner; f = N::first(tc + ++u * c.nc)) {
#pragma unroll
      for (int w = 0; w < PW; ++w) {
        const int x = (f + w * N::NEXT) % nx;
        const unsigned bit = 1u << (u * PW + w);
        if (x == 0) lm |= bit;
        if (x == nx - 1) rm |= bit;
      }
    }
  }
  const unsigned lw = (unsigned)((nx - 1) * (int)sizeof(T)), rw = (unsigned)((1 - nx) * (int)sizeof(T));
  // After the barrier that ends plane q's densities, plane q - R is collided while
  // the density warps form plane q + 1, in a psi plane and moments not read here.
#pragma unroll 1
  for (int q = 0; q < nplanes; ++q) {
    row_barrier(ncons);
    if (q < 2 * R) continue;
    const unsigned use = uses + q;
    const int z = flip ? z0 + zc - 1 + 2 * R - q : z0 - 2 * R + q;   // plane q - R, inside the box
    unsigned pl[2 * R + 1][2 * R + 1];   // psi row (dy, dz) of the block's first interior row
#pragma unroll
    for (int dz = -R; dz <= R; ++dz)
#pragma unroll
      for (int dy = -R; dy <= R; ++dy)
        pl[dz + R][dy + R] = Sh::ring_off + ((use - R + (flip ? -dz : dz)) % Sh::NR) * Sh::ring_bytes +
                             (unsigned)((R + dy) * nx * (int)sizeof(T));
    const unsigned mq = Sh::mom_off + ((use - R) % Sh::NM) * Sh::mom_bytes;
    char* const out0 = static_cast<char*>(d.dst) + (((long long)z * ny + y0) * nx) * (long long)sizeof(S);
#pragma unroll 1
    for (int u = 0;; ++u) {
      const int f = N::first(tc + u * c.nc);
      if (f >= inner) break;
      const unsigned jc = (unsigned)(f * (int)sizeof(T));
      // x-neighbours of node w at dx = -1, +1, bytes
      unsigned xl[PW], xr[PW];
#pragma unroll
      for (int w = 0; w < PW; ++w) {
        const unsigned jw = jc + (unsigned)(w * N::NEXT * (int)sizeof(T)), bit = 1u << (u * PW + w);
        xl[w] = jw + ((lm & bit) ? lw : (unsigned)-(int)sizeof(T));
        xr[w] = jw + ((rm & bit) ? rw : (unsigned)sizeof(T));
      }
      auto at = [&](int dx, int dy, int dz) {
        const unsigned row = pl[dz + R][dy + R];
        if constexpr (N::PAIR) {
          if (dx == 0) return row_ld<V>(smem, row + jc);
          if (dx < 0) return make_float2(row_ld<T>(smem, row + xl[0]), row_ld<T>(smem, row + jc));
          return make_float2(row_ld<T>(smem, row + jc + (unsigned)sizeof(T)), row_ld<T>(smem, row + xr[PW - 1]));
        } else {
          T v[2] = {(T)0, (T)0};
#pragma unroll
          for (int w = 0; w < PW; ++w)
            v[w] = row_ld<T>(smem, row + (dx == 0 ? jc + (unsigned)(w * N::NEXT * (int)sizeof(T)) : dx > 0 ? xr[w] : xl[w]));
          return make_float2(v[0], v[1]);
        }
      };
      auto moment = [&](int comp) {
        const unsigned off = mq + comp * Sh::comp_bytes + (unsigned)(f * (int)sizeof(T));
        if constexpr (N::PAIR) return row_ld<V>(smem, off);
        else return make_float2(row_ld<T>(smem, off), row_ld<T>(smem, off + N::NEXT * (unsigned)sizeof(T)));
      };
      V Fx, Fy, Fz;
      sc_force_at<V, Sh::ST>(at, at(0, 0, 0), G, Fx, Fy, Fz);
      const V dn = moment(0);
      char* const rest = out0 + (long long)f * (long long)sizeof(S);
      char* o = rest;
      const bool ok1 = f + N::NEXT < inner;
      collide_nodes<V, true, P == kF16>(
          dn, vadd(Lane<V>::all(n0), dn), moment(1), moment(2), moment(3), Fx, Fy, Fz, (T)1, scale,
          [](int) { return Lane<V>::all(0); },
          [&](int i, V g) {
            o += pbytes;   // populations come in the order 1 .. 18, 0
            char* const to = i == 0 ? rest : o;
            if constexpr (N::PAIR) {
              if constexpr (P == kF16) *reinterpret_cast<__half2*>(to) = __float22half2_rn(g);
              else *reinterpret_cast<V*>(to) = g;
            } else {
              auto put = [&](char* at, T v) {
                if constexpr (P == kF16) *reinterpret_cast<__half*>(at) = __float2half_rn(v);
                else *reinterpret_cast<T*>(at) = v;
              };
              put(to, row_node(g, 0));
              if (ok1) put(to + N::NEXT * sizeof(S), row_node(g, 1));
            }
          });
    }
  }
  uses += nplanes;
}

// mbarriers: `full` takes the producer's arrival and its copies' bytes, `empty` one
// arrival of each density warp
__device__ __forceinline__ void row_init(unsigned char* smem, const RowCfg& c) {
  unsigned long long* full = reinterpret_cast<unsigned long long*>(smem);
  if (threadIdx.x == 0) {
    for (int g = 0; g < kRowGroups; ++g) {
      tma_mbar_init(full + g, 1);
      tma_mbar_init(full + kRowGroups + g, (unsigned)(c.nd / 32));
    }
    *reinterpret_cast<volatile int*>(smem + kRowDead) = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
}
// end of a CTA's items: a wait that gave up is reported, and the producer (whose
// `uses` counts the planes it issued) waits, bounded, for its copies in flight
__device__ __forceinline__ void row_finish(unsigned char* smem, const RowCfg& c, unsigned uses, int* err) {
  if (*reinterpret_cast<volatile int*>(smem + kRowDead) == 0) return;
  unsigned long long* full = reinterpret_cast<unsigned long long*>(smem);
  if (err) *reinterpret_cast<volatile int*>(err) = 1;
  if ((int)threadIdx.x >= c.nd + c.nc && uses > 0)
    for (int g = 0; g < kRowGroups; ++g) tma_wait(full + g, (uses - 1) & 1);
}

template <class Sh, bool ALIGNED>
__global__ void __launch_bounds__(kRowThreads, 1) lattice_row_kernel(LatticeDesc d, RowCfg c, int flip) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  row_init(smem_raw, c);
  step_grid_enter();
  __syncthreads();
  const int items = ((d.ny + c.by - 1) / c.by) * ((d.nz + c.zc - 1) / c.zc);
  unsigned uses = 0;
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x)
    row_process_item<Sh, ALIGNED>(d, c, item, flip != 0, smem_raw, uses);
  row_finish(smem_raw, c, uses, d.err);
}

// A batch of tau = 1 lattices (see lattice_async_batch_kernel for the table; here
// every entry has its rows per item in `rows`).  Each role keeps its own copy of the
// item's lattice in shared memory: in registers it would spill, and roles may be
// at different items.
template <class Sh, bool ALIGNED>
__global__ void __launch_bounds__(kRowThreads, 1)
lattice_row_batch_kernel(const BatchEntry* __restrict__ table, const BatchHeader* __restrict__ hdr, int step) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ LatticeDesc lattice[3];
  RowCfg c{0, 0, kRowBatchDensityWarps * 32, (int)blockDim.x - (kRowBatchDensityWarps + 1) * 32};
  row_init(smem_raw, c);
  step_grid_enter();
  __syncthreads();
  const int n = hdr->n;
  const long long total = hdr->total_items;
  const int tid = threadIdx.x, role = tid < c.nd ? 0 : (tid < c.nd + c.nc ? 1 : 2);
  const int first = role == 0 ? 0 : (role == 1 ? c.nd : c.nd + c.nc);
  const int members = role == 0 ? c.nd : (role == 1 ? c.nc : 32);
  LatticeDesc& d = lattice[role];
  unsigned uses = 0;
#pragma unroll 1
  for (long long item = blockIdx.x; item < total; item += gridDim.x) {
    int lo = 0, hi = n - 1;          // last entry with item_begin <= item
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (table[mid].item_begin <= item) lo = mid; else hi = mid - 1;
    }
    const BatchEntry& e = table[lo];
    asm volatile("bar.sync %0, %1;\n" ::"r"(2 + role), "r"(members) : "memory");   // the role is done with the last one
    if (tid == first) {
      d = e.d;
      if ((e.parity ^ step) & 1) {
        d.src = e.d.dst;
        d.dst = const_cast<void*>(e.d.src);
      }
    }
    asm volatile("bar.sync %0, %1;\n" ::"r"(2 + role), "r"(members) : "memory");
    c.by = e.rows;
    c.zc = e.zchunk;
    row_process_item<Sh, ALIGNED>(d, c, (int)(item - e.item_begin), false, smem_raw, uses);
    if (*reinterpret_cast<volatile int*>(smem_raw + kRowDead)) {   // this and every later item of the CTA
      if (d.err) *reinterpret_cast<volatile int*>(d.err) = 1;
    }
  }
  row_finish(smem_raw, c, uses, nullptr);
}

}  // namespace lbm
