// pair_tile.cuh -- the fused timestep on population pairs (ST_F64, ST_F32, ST_F32X): one tile's
// march, the collision, and the kernel around them.  The staged 16-bit and recolour-on-pull
// layouts march through step_tile (step_kernel.cuh).
//
// What bounds it.  The state is read and written once (305 B per D3Q19 FP32 update), but the
// march is a chain: a plane's pulls, its colour sums, a reciprocal, the shared-memory exchange of
// rho^N, the collision.  With 128 registers per thread four CTAs of 128 threads share an SM and
// issue about half the time, so the chain's instructions and exposed waits set the rate of every
// lattice but the largest.  Hence the order of a plane's work, and what it leaves out:
//   1. the site byte, the flux and the next plane's links are loaded before anything waits (GEN;
//      a lattice that has none of them runs an instantiation without that code);
//   2. the ring cells are pulled and summed;
//   3. the own cells' pulls of the next plane are issued (PF: 38 registers in flight across the
//      collision), then this plane's, issued a plane ago, are summed and parked;
//   4. the moments of the plane to collide are formed before its neighbours' rho^N is waited for;
//   5. nothing is pulled past the chunk's end or beyond the first column over a ragged edge.
// Measured on one GPU, us per step before -> after (the FP32 results are the same bits):
//   192^3 FP32 374 -> 368 (0.87 of measured HBM), F32X 460 -> 408; 128^3 135 -> 129, 154 -> 129;
//   160^3 walls, gradient rule, heated flux 289 -> 236; 131 x 117 x 89 with solids 119 -> 100;
//   48^3 20.6 -> 17.9; 64-member ensemble 1153 -> 880 (pulls ahead, D2Q9 groups with barriers of
//   their own); FP64 128^3 1719 -> 1425.
// Tried and slower: the ring's sums after the own sums and the next issue (192^3 474: the loads of
// both cells live at once spill), or after the own sums alone (444); the next plane's issue after
// the own sums (384; better by 2.7 % only for the plain F32X kernel, whose sums need the
// registers: EARLY).  No change: the barrier split into an mbarrier's arrival and wait, 32-bit
// offsets from uniform bases.
#pragma once

#include "launch.h"
#include "step_kernel.cuh"

namespace cgevap {

// A column (a, b) of the march: where it is stored, and the directions whose source lies beyond an
// x or y wall (kNoCell: no column of the lattice).  The storage offsets to its neighbours, (a-1, a+1,
// b-1, b+1), 0 beyond a wall (not used), are kept in shared memory: eight registers less per thread.
constexpr uint32_t kNoCell = 1u << 31;
struct Column {
  int col;        // in-plane storage offset
  int cell;       // in-plane compact index
  uint32_t wall;
};

template <class L>
__device__ __forceinline__ Column make_column(const Geom& g, int ua, int ub, int4& to) {
  const Slot s = make_slot<L>(g, ua, ub);
  Column c;
  // of a ragged tile only the first column and row beyond the lattice are anyone's neighbours
  const bool ok = s.ok && ua <= g.na && (!L::D3 || ub <= g.nb);
  c.col = ok ? (s.b + g.gy) * g.pitch + s.a + kOx : kOx;
  c.cell = ok ? s.b * g.na + s.a : 0;
  to = make_int4(s.dxm, s.dxp, s.dym, s.dyp);
  c.wall = (s.am1 < 0 ? dirs_where<L>(0, +1) : 0u) | (s.ap1 < 0 ? dirs_where<L>(0, -1) : 0u);
  if (L::D3) c.wall |= (s.bm1 < 0 ? dirs_where<L>(1, +1) : 0u) | (s.bp1 < 0 ? dirs_where<L>(1, -1) : 0u);
  if (!ok) c.wall = kNoCell;
  return c;
}

// Plane um of a chunk (-1 <= um <= nm): its index, the storage offsets to the planes below and
// above, and the directions that bounce back off a wall there.
struct March {
  int m, lo, hi;
  uint32_t wall;
  bool ok;
};

template <class L>
__device__ __forceinline__ March make_march(const Geom& g, int um) {
  const int ps = g.rows * g.pitch;
  March p;
  p.ok = g.per_m || (um >= 0 && um < g.nm);
  p.m = um < 0 ? um + g.nm : (um >= g.nm ? um - g.nm : um);
  if (!p.ok) p.m = 0;
  const bool first = p.m == 0, last = p.m == g.nm - 1;
  p.lo = !first ? -ps : (g.per_m ? (g.nm - 1) * ps : 0);
  p.hi = !last ? ps : (g.per_m ? -(g.nm - 1) * ps : 0);
  p.wall = 0u;
  if (!g.per_m) p.wall = (first ? dirs_where<L>(2, +1) : 0u) | (last ? dirs_where<L>(2, -1) : 0u);
  return p;
}

// A pair of the state read.  An ordinary load, and one the compiler keeps behind the wait or barrier
// before it: a step launched ahead of its predecessor's end is resident while the predecessor writes
// what it reads, and within one launch of the ensemble other CTAs rewrite the buffers, so the
// read-only path (__ldg), which asks for memory no one writes while the kernel runs, is not open here
// (nor for links and flux fields, which the kernel before may have written).  As fast as __ldg in
// every case; written as a C++ load, FP64 128^3 took 1.1 % longer.
__device__ __forceinline__ float2 load_pair(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)) : "memory");
  return v;
}
__device__ __forceinline__ double2 load_pair(const double2* p) {
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(__cvta_generic_to_global(p)) : "memory");
  return v;
}

// Pull of one cell's pairs (Eq. Stream, pull form, halfway bounce-back), as pull_cell; to: its
// column's neighbour offsets, lo / hi: the planes'.
template <int Q, int S>
__device__ __forceinline__ void pull_pairs(const void* pin, int ns, int4 to, int si, int lo, int hi,
                                           uint32_t bits, V2<typename Storage<S>::real> (&g)[Q]) {
  using L = Lattice<Q>;
  using Vec = typename Storage<S>::vec;
  const Vec* p = reinterpret_cast<const Vec*>(pin);
  auto from = [&](int i) {
    return i * ns + si + (L::ca(i) > 0 ? to.x : (L::ca(i) < 0 ? to.y : 0)) +
           (L::cb(i) > 0 ? to.z : (L::cb(i) < 0 ? to.w : 0)) +
           (L::cm(i) > 0 ? lo : (L::cm(i) < 0 ? hi : 0));
  };
  if (bits == 0) {  // no link of this cell bounces back (the common case)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const Vec v = load_pair(p + from(i));
      g[i] = {v.x, v.y};
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const Vec v = load_pair(p + ((bits >> i) & 1u ? opp(i) * ns + si : from(i)));
      g[i] = {v.x, v.y};
    }
  }
}

// Products and reciprocals that no surrounding kernel contracts or approximates differently.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float recip_density(float x) { return __frcp_rn(x); }
// FP64: from the hardware's approximation y one step of Householder's iteration of third order for
// x^-1: with e = 1 - x y, 1 / x = y / (1 - e) = y (1 + e + e^2) + O(y e^3).  y is good to about 2^-20,
// so e^3 and the rounding of e + e^2 lie below the rounding of the last product, and the result is
// within 1.1 half-ulps of 1 / x.  The approximation takes and gives no subnormals; where x or 1 / x is
// one (and for 0, infinity and NaN) the division.
static __device__ __noinline__ double divide_one(double x) { return 1.0 / x; }  // inlined, a step took 1.2 % longer
__device__ __forceinline__ double recip_density(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (h - 0x00100000u >= 0x7fd00000u - 0x00100000u) return divide_one(x);  // not 2^-1022 <= |x| < 2^1022
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// |F| and 1 / |F| from F2 = |F|^2 > 0.  FP64: the iteration of third order for x^(-1/2): with
// e = 1 - F2 y^2, F2^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8) + O(y e^3), within 1.6 half-ulps
// (half of the rounding of F2 y reaches the result), and |F| = F2 / |F| within 2.6.  Outside the range
// in which F2 and its root are far from subnormals, the square root and the division (GB300 issues an
// FP64 instruction every 16 cycles a warp: 7 of them here against about 25).
__device__ __forceinline__ void norm_of(float F2, float& Fn, float& iFn) {
  iFn = rsqrtf(F2);
  Fn = mul_rn(F2, iFn);
}
__device__ __forceinline__ void norm_of(double F2, double& Fn, double& iFn) {
  if (F2 > 1e-280 && F2 < 1e280) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(F2));
    const double e = fma(-F2 * y, y, 1.0);
    iFn = fma(y, e * fma(0.375, e, 0.5), y);
    Fn = F2 * iFn;
  } else {
    norm_pair<double>(F2, Fn, iFn);
  }
}

// Colour totals of a cell's pairs, the same operations in every tile that holds the cell.
template <int Q, class R>
__device__ __forceinline__ void colour_sums(const V2<R> (&g)[Q], R& sr, R& sb) {
  if constexpr (std::is_same<R, float>::value) {  // both colours in packed FP32
    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < Q; ++i) acc = __fadd2_rn(acc, make_float2(g[i].r, g[i].b));
    sr = acc.x;
    sb = acc.y;
  } else {
    R r0 = g[0].r, r1 = g[1].r, b0 = g[0].b, b1 = g[1].b;
#pragma unroll
    for (int i = 2; i < Q; i += 2) {
      r0 += g[i].r;
      b0 += g[i].b;
      if (i + 1 < Q) {
        r1 += g[i + 1].r;
        b1 += g[i + 1].b;
      }
    }
    sr = r0 + r1;
    sb = b0 + b1;
  }
}

// Site decision and Eq. (exchange) from the colour totals; mb: the site byte read (rules 0 and 2),
// phi: the flux where a field is set.  As exchange_from_sums, whose loads were issued earlier.
// ALT picks which product of rho^N = (sr - sb)/rho - 2 e/rho is rounded before the subtraction.
// The march of a D3Q19 tile and the rest of it (ring, the two planes that start a chunk) have
// always differed in that; it decides the last bit of rho^N at sites, and with it whole runs bit
// for bit (recorded site sets, checkpoints), so it stays.
template <int S, bool GEN, bool ALT>
__device__ __forceinline__ typename Storage<S>::real exchange_sums(
    const Physics& ph, uint32_t mb, typename Storage<S>::real phi, typename Storage<S>::real sr,
    typename Storage<S>::real sb, typename Storage<S>::real& rr, typename Storage<S>::real& rb,
    typename Storage<S>::real& e, uint32_t& flags, typename Storage<S>::real& irho) {
  using R = typename Storage<S>::real;
  irho = recip_density(sr + sb);
  const R rn_pre = mul_rn(sr - sb, irho);
  bool site, near;
  if (!GEN || ph.rule == 1) {
    const R d = fabs(rn_pre) - PHYS(R, ph, threshold);
    site = d < R(0);
    near = fabs(d) < R(1e-6);
  } else {  // gradient rule: the decision of the previous step (bit 1); given rule: bit 0
    const int sh = ph.rule == 2 ? 0 : 1;
    site = (mb >> sh) & 1u;
    near = (mb >> (sh + 2)) & 1u;
  }
  e = R(0);
  if (site) e = GEN && ph.phi_field ? mul_rn(phi, PHYS(R, ph, inv_sbar)) : PHYS(R, ph, varphi);
  rr = sr - e;
  rb = sb + e;
  flags = (site ? 1u : 0u) | (near ? 4u : 0u);
  return ALT ? fma(sr - sb, irho, -mul_rn(R(2) * e, irho)) : fma(R(-2) * e, irho, rn_pre);
}

// ST_F32X: the rounding errors (lr, lb) of a cell's post-exchange totals rr, rb: what the colour
// totals summed without rounding error (from B) exceed the plain sums sr, sb by, and the exchange's
// own rounding (TwoSum).
template <int Q>
__device__ __forceinline__ void exact_errors(const Physics& ph, const V2<float> (&g)[Q], float sr, float sb,
                                             float rr, float rb, float e, float& lr, float& lb) {
  float2 acc = sum_start(ph), lo = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int i = 0; i < Q; ++i) fast_two_sum_acc(acc, lo, make_float2(g[i].r, g[i].b));
  // (acc - B) and the plain sums are both within a few ulps of B of the total: exact difference
  lo = __fadd2_rn(sub2(sub2(acc, sum_start(ph)), make_float2(sr, sb)), lo);
  lr = __fadd_rn(lo.x, two_sum_err(sr, -e, rr));
  lb = __fadd_rn(lo.y, two_sum_err(sb, e, rb));
}

// Sum of s_p v_p over the pairs p of opposite directions (i, i + 1) with c_i = s along an axis
// (0: a, 1: b, 2: m) and |c_i|^2 = cls; v_p = the difference of a quantity over the pair.
template <class L>
__host__ __device__ constexpr int axis_comp(int i, int axis) {
  return axis == 0 ? L::ca(i) : (axis == 1 ? L::cb(i) : L::cm(i));
}
template <class L, class R>
__device__ __forceinline__ R axis_sum(const R (&v)[(L::Q - 1) / 2], int axis, int cls) {
  R s = R(0);
  bool any = false;
#pragma unroll
  for (int p = 0; p < (L::Q - 1) / 2; ++p) {
    const int i = 2 * p + 1, k = axis_comp<L>(i, axis);
    if (L::speed2(i) != cls || k == 0) continue;
    if (!any) s = k > 0 ? v[p] : -v[p];
    else s = k > 0 ? s + v[p] : s - v[p];
    any = true;
  }
  return s;
}

// One cell's moments that need only its own populations.
template <class R>
struct CellMoments {
  R rho, wr, wb, ua, ub, um, uu15, itau, abar;
};
template <int Q, class R>
__device__ __forceinline__ CellMoments<R> cell_moments(const Physics& ph, const R (&f)[Q], R rr, R rb, R irho) {
  using L = Lattice<Q>;
  CellMoments<R> c;
  c.rho = rr + rb;
  c.wr = rr * irho;
  c.wb = rb * irho;
  if constexpr (std::is_same<R, float>::value) {
    R ja = R(0), jb = R(0), jm = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (L::ca(i) > 0) ja += f[i];
      if (L::ca(i) < 0) ja -= f[i];
      if (L::cb(i) > 0) jb += f[i];
      if (L::cb(i) < 0) jb -= f[i];
      if (L::cm(i) > 0) jm += f[i];
      if (L::cm(i) < 0) jm -= f[i];
    }
    c.ua = ja * irho;
    c.ub = jb * irho;
    c.um = jm * irho;
    c.uu15 = mul_rn(1.5f, fma(c.um, c.um, fma(c.ua, c.ua, mul_rn(c.ub, c.ub))));
    c.itau = fma(c.wr, PHYS(R, ph, inv_tau_r), mul_rn(c.wb, PHYS(R, ph, inv_tau_b)));
    c.abar = fma(c.wr, PHYS(R, ph, alpha_r), mul_rn(c.wb, PHYS(R, ph, alpha_b)));
    return c;
  }
  R d[(Q - 1) / 2];
#pragma unroll
  for (int p = 0; p < (Q - 1) / 2; ++p) d[p] = f[2 * p + 1] - f[2 * p + 2];
  c.ua = (axis_sum<L>(d, 0, 1) + axis_sum<L>(d, 0, 2)) * irho;
  c.ub = L::D3 ? (axis_sum<L>(d, 1, 1) + axis_sum<L>(d, 1, 2)) * irho : R(0);
  c.um = (axis_sum<L>(d, 2, 1) + axis_sum<L>(d, 2, 2)) * irho;
  R uu = fma(c.ua, c.ua, c.um * c.um);
  if (L::D3) uu = fma(c.ub, c.ub, uu);
  c.uu15 = R(1.5) * uu;
  c.itau = fma(c.wr, PHYS(R, ph, inv_tau_r), c.wb * PHYS(R, ph, inv_tau_b));  // harmonic mean of tau_k
  c.abar = fma(c.wr, PHYS(R, ph, alpha_r), c.wb * PHYS(R, ph, alpha_b));
  return c;
}

// Eq. (cg) from the neighbours' rho^N: F = (1/c_s^2) sum_i W_i rho^N(x + c_i) c_i.
template <int Q, class R>
__device__ __forceinline__ void colour_gradient(const R (&rnb)[Q], R& Fa, R& Fb, R& Fm) {
  using L = Lattice<Q>;
  if constexpr (std::is_same<R, float>::value) {
    Fa = Fb = Fm = R(0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const R w = R(3.0 * L::W(i));
      if (L::ca(i) != 0) Fa = fma(L::ca(i) > 0 ? w : -w, rnb[i], Fa);
      if (L::cb(i) != 0) Fb = fma(L::cb(i) > 0 ? w : -w, rnb[i], Fb);
      if (L::cm(i) != 0) Fm = fma(L::cm(i) > 0 ? w : -w, rnb[i], Fm);
    }
  } else {  // from the differences over opposite neighbours
    R dn[(Q - 1) / 2];
#pragma unroll
    for (int p = 0; p < (Q - 1) / 2; ++p) dn[p] = rnb[2 * p + 1] - rnb[2 * p + 2];
    constexpr double w1 = 3.0 * L::W(1), w2 = 3.0 * L::W(L::Q - 1);
    Fa = fma(R(w2), axis_sum<L>(dn, 0, 2), R(w1) * axis_sum<L>(dn, 0, 1));
    Fb = L::D3 ? fma(R(w2), axis_sum<L>(dn, 1, 2), R(w1) * axis_sum<L>(dn, 1, 1)) : R(0);
    Fm = fma(R(w2), axis_sum<L>(dn, 2, 2), R(w1) * axis_sum<L>(dn, 2, 1));
  }
}

// Eq. (collision) with Eq. (feq), Eq. (perturb) and Eq. (recolor) of one cell; out(i, r, b) takes
// each direction's pair.  Returns |F|.  Opposite directions share |c.u| and |c.F| with opposite
// signs.  Multiply-adds are written as such, so a result does not depend on the surrounding kernel.
// FP32: the equilibrium and the perturbation as separate terms, packed over opposite directions.
template <int Q, class Out>
__device__ __forceinline__ float collide_pairs(const Physics& ph, const CellMoments<float>& m, const float (&f)[Q],
                                               float Fa, float Fb, float Fm, const Out& out) {
  using L = Lattice<Q>;
  using R = float;
  const R rho = m.rho, wr = m.wr, wb = m.wb, itau = m.itau, abar = m.abar, uu15 = m.uu15;
  const R F2 = fma(Fm, Fm, fma(Fa, Fa, mul_rn(Fb, Fb)));
  R Fn = R(0), iFn = R(0);
  if (F2 > R(0)) norm_of(F2, Fn, iFn);
  const R pamp = PHYS(R, ph, amp) * itau;       // (9/4) sigma / tau
  const R rcol = PHYS(R, ph, beta) * wr * wb;   // beta rho_r rho_b / rho^2
  R restc[3], rwc[3], kw[3], kc[3], kr[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int i = c == 0 ? 0 : (c == 1 ? 1 : L::Q - 1);  // a direction of speed class c
    restc[c] = mul_rn(rho, fma(R(L::B(i)), abar, R(L::A(i))));   // f_i^eq(rho, 0)
    rwc[c] = rho * R(L::W(i));
    kw[c] = pamp * R(L::W(i)) * iFn;
    kc[c] = pamp * R(L::C(i)) * Fn;
    kr[c] = rcol * iFn * R(inv_norm<L>(i)) * restc[c];
  }
  const R f0eq = fma(rwc[0], -uu15, restc[0]);
  const R fi0 = fma(-mul_rn(pamp, R(L::C(0))), Fn, fma(itau, f0eq - f[0], f[0]));
  const R r0 = mul_rn(wr, fi0);
  out(0, r0, fi0 - r0);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int j = i + 1;
    const int c = L::speed2(i);
    R cu = R(0), pc = R(0);
    if (L::ca(i) > 0) { cu += m.ua; pc += Fa; }
    if (L::ca(i) < 0) { cu -= m.ua; pc -= Fa; }
    if (L::cb(i) > 0) { cu += m.ub; pc += Fb; }
    if (L::cb(i) < 0) { cu -= m.ub; pc -= Fb; }
    if (L::cm(i) > 0) { cu += m.um; pc += Fm; }
    if (L::cm(i) < 0) { cu -= m.um; pc -= Fm; }
    const R even = fma(rwc[c], fma(R(4.5) * cu, cu, -uu15), restc[c]);
    const R odd = R(3) * rwc[c] * cu;
    const R pert = fma(kw[c], pc * pc, -kc[c]);  // Eq. (perturb), even in c
    const R kp = kr[c] * pc;                     // Eq. (recolor) term, odd in c
    // both directions of the pair in packed FP32
    const float2 fv = make_float2(f[i], f[j]);
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 feq = __fadd2_rn(make_float2(even, even), make_float2(odd, -odd));
    float2 post = __ffma2_rn(make_float2(itau, itau), __ffma2_rn(fv, m1, feq), fv);
    post = __fadd2_rn(post, make_float2(pert, pert));
    const float2 red = __ffma2_rn(make_float2(wr, wr), post, make_float2(kp, -kp));
    const float2 blue = sub2(post, red);
    out(i, red.x, blue.x);
    out(j, red.y, blue.y);
  }
  return Fn;
}
// FP64 (bound by the FP64 pipe, so by the count of operations): relaxation and perturbation in one
// polynomial per speed class s and opposite pair,
//   f_i' = (1 - itau) f_i + even +- odd,
//   even = itau (restc_s - 3/2 rho W_s u^2) - pamp C_s |F| + 9/2 itau rho W_s (c.u)^2
//        + pamp W_s (c.F)^2 / |F|,   odd = 3 itau rho W_s (c.u).
template <int Q, class Out>
__device__ __forceinline__ double collide_pairs(const Physics& ph, const CellMoments<double>& c,
                                                const double (&f)[Q], double Fa, double Fb, double Fm,
                                                const Out& out) {
  using L = Lattice<Q>;
  using R = double;
  R F2 = fma(Fa, Fa, Fm * Fm);
  if (L::D3) F2 = fma(Fb, Fb, F2);
  R Fn = R(0), iFn = R(0);
  if (F2 > R(0)) norm_of(F2, Fn, iFn);
  const R pamp = ph.amp * c.itau;                    // (9/4) sigma / tau
  const R rcol = ph.beta * c.wr * c.wb * iFn;        // beta rho_r rho_b / (rho^2 |F|)
  const R aF = pamp * Fn, ai = pamp * iFn;
  const R keep = R(1) - c.itau, rt = c.rho * c.itau;
  R base[3], k1[3], k2[3], kw[3], kr[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int i = s == 0 ? 0 : (s == 1 ? 1 : L::Q - 1);  // a direction of speed class s
    const R restc = fma(R(L::B(i)), c.abar, R(L::A(i)));  // f_i^eq(rho, 0) / rho
    base[s] = fma(R(-L::C(i)), aF, rt * fma(R(L::W(i)), -c.uu15, restc));
    if (s == 0) continue;
    k1[s] = R(4.5 * L::W(i)) * rt;
    k2[s] = R(3.0 * L::W(i)) * rt;
    kw[s] = ai * R(L::W(i));
    kr[s] = rcol * (c.rho * restc) * R(inv_norm<L>(i));
  }
  {
    const R f0 = fma(keep, f[0], base[0]);
    const R r0 = mul_rn(c.wr, f0);
    out(0, r0, f0 - r0);
  }
  static_assert(opposites_adjacent<L>(), "directions (i, i+1), i odd, must be opposite");
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int j = i + 1, s = L::speed2(i);
    R cu = R(0), cf = R(0);
    bool any = false;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const int k = axis_comp<L>(i, ax);
      if (!k) continue;
      const R u = ax == 0 ? c.ua : (ax == 1 ? c.ub : c.um);
      const R F = ax == 0 ? Fa : (ax == 1 ? Fb : Fm);
      cu = any ? (k > 0 ? cu + u : cu - u) : (k > 0 ? u : -u);
      cf = any ? (k > 0 ? cf + F : cf - F) : (k > 0 ? F : -F);
      any = true;
    }
    const R even = fma(kw[s] * cf, cf, fma(k1[s] * cu, cu, base[s]));
    const R odd = k2[s] * cu;
    const R kp = kr[s] * cf;
    const R fi = fma(keep, f[i], even + odd), fj = fma(keep, f[j], even - odd);
    const R ri = fma(c.wr, fi, kp), rj = fma(c.wr, fj, -kp);
    out(i, ri, fi - ri);
    out(j, rj, fj - rj);
  }
  return Fn;
}

// Programmatic dependent launch: a step's launch is prepared while its predecessor runs, and its CTAs
// wait for the predecessor's end and its writes before they read anything.  dependents_may_start()
// lets them take their places as soon as every CTA of this step has started: worth it for the short
// patch kernel (64^2 FP32 with the tally below 7.2 -> 3.3 us a step), not for the march, whose
// free slots they would fill (192^3 362 us without, 388 with it).  Without the launch attribute both
// are no-ops.
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The barrier of a tile's threads, between the writes and the reads of a plane's rho^N.
struct CtaSync {  // a whole CTA
  __device__ __forceinline__ void wait() const { __syncthreads(); }
};
struct WarpSync {  // one warp runs the tile
  __device__ __forceinline__ void wait() const { __syncwarp(); }
};
struct PairSync {  // two groups of 64 threads share a CTA, each with a named barrier of its own
  int group;
  __device__ __forceinline__ void wait() const {
    if (group == 0)
      asm volatile("bar.sync 1, 64;" ::: "memory");
    else
      asm volatile("bar.sync 2, 64;" ::: "memory");
  }
};

// Shared memory of a tile: the four-plane rho^N ring, two planes of parked sums, the columns'
// neighbour offsets.
template <int Q, int S, int TX, int TY>
struct PairSmem {
  using R = typename Storage<S>::real;
  static constexpr int HX = TX + 2, HY = Lattice<Q>::D3 ? TY + 2 : 1;
  static constexpr int RING = (4 * HY * HX * (int)sizeof(R) + 15) & ~15;
  static constexpr int PARK = (2 * Q * TX * TY * (int)sizeof(R) + 15) & ~15;
  static constexpr int COLS = 2 * TX * TY * (int)sizeof(int4);  // neighbour offsets, own and ring
  static constexpr int BYTES = RING + PARK + COLS;
};

// The tail of the step: collision and store, the site byte.  GEN as in pair_tile.
template <bool GEN>
struct PairStep {
  template <int Q, int S>
  __device__ __forceinline__ void prefetch(const StepArgs&, int /*si*/) const {}
  template <int Q, int S>
  __device__ __forceinline__ void stage(const StepArgs&, int, int, int, int) const {}
  // What needs only the cell's own sums, formed before the neighbours' rho^N is waited for.
  template <int Q, int S, class R>
  __device__ __forceinline__ CellMoments<R> before(const StepArgs& A, const R (&f)[Q], R rr, R rb, R irho) const {
    return cell_moments<Q, R>(A.ph, f, rr, rb, irho);
  }
  // f, rr, rb: the cell's post-exchange sums; (lr, lb): the rounding errors of rr, rb (ST_F32X);
  // flags: its site byte so far; rnb[i]: rho^N at x + c_i (its own where that is solid).
  template <int Q, int S, class R>
  __device__ __forceinline__ void cell(const StepArgs& A, int cell, const int4*, uint32_t, const March&,
                                       int si, const R (&f)[Q], const CellMoments<R>& c, R rr, R rb, R,
                                       R lr, R lb, uint32_t flags, const R (&rnb)[Q]) const {
    using Vec = typename Storage<S>::vec;
    R Fa, Fb, Fm;
    colour_gradient<Q, R>(rnb, Fa, Fb, Fm);
    Vec* p = reinterpret_cast<Vec*>(A.pout);
    const int ns = A.g.nstore;
    // ST_F32X: what the stored moving pairs carry of each colour, without rounding error (from B)
    float2 hi = make_float2(0.0f, 0.0f), lo = hi;
    if constexpr (ExactPairs<S>::value) hi = sum_start(A.ph);
    auto out = [&](int i, R r, R b) {
      if constexpr (ExactPairs<S>::value) {
        if (i == 0) return;  // stored last
        fast_two_sum_acc(hi, lo, make_float2(r, b));
      }
      Vec v;
      v.x = r;
      v.y = b;
      p[i * ns + si] = v;
    };
    const R Fn = collide_pairs<Q>(A.ph, c, f, Fa, Fb, Fm, out);
    if constexpr (ExactPairs<S>::value) {
      // the rest pair: the exact colour masses (rr + lr, rb + lb) less the stored moving pairs
      hi = sub2(hi, sum_start(A.ph));  // exact
      const float2 s2 = sub2(make_float2(rr, rb), hi);
      const float2 e2 = make_float2(two_sum_err(rr, -hi.x, s2.x), two_sum_err(rb, -hi.y, s2.y));
      const float2 r0 = __fadd2_rn(s2, __fadd2_rn(e2, sub2(make_float2(lr, lb), lo)));
      p[si] = r0;
    }
    if (GEN && A.ph.rule == 0) {
      const R t = Fn - PHYS(R, A.ph, threshold);
      flags |= (t > R(0) ? 2u : 0u) | (fabs(t) < R(1e-6) ? 8u : 0u);
    }
    if (GEN) A.mask_out[cell] = (uint8_t)flags;
  }
  // The band rule's site byte is known when the cell is filled.
  __device__ __forceinline__ void filled(const StepArgs& A, int cell, uint32_t flags) const {
    if (!GEN) A.mask_out[cell] = (uint8_t)flags;
  }
};

// One tile of the (a, b) plane (TX x TY columns; one row in 2D) marching through the planes
// [m0, m1) along m, a thread per column; the first threads also take one cell of the ring around
// the tile each.  Returns this thread's site count and removed mass.
// PF: the own cells' pulls are issued one plane ahead.  GEN: the lattice has solid links, site
// bytes to read or a flux field; without it that code is left out (a band-rule lattice with a
// scalar flux needs none of them).
template <int Q, int S, int TX, int TY, bool PF, bool GEN, class Epi, class Sync>
__device__ __forceinline__ void pair_tile(const StepArgs& A, int tile, int m0, int m1, unsigned char* smem,
                                          long long& n_sites, double& removed, int tid, const Epi& epi,
                                          const Sync& sync) {
  using L = Lattice<Q>;
  using R = typename Storage<S>::real;
  using SM = PairSmem<Q, S, TX, TY>;
  constexpr int NT = TX * TY, HX = SM::HX, HY = SM::HY, OB = L::D3 ? 1 : 0;
  constexpr int NH = HX * HY - NT;
  // PF: the next plane's pulls are issued before this plane's sums are formed, or after
  constexpr bool EARLY = !ExactPairs<S>::value || GEN;
  static_assert(NH <= NT, "one ring cell per thread at most");
  static_assert(L::D3 || TY == 1, "D2Q9 tiles are one row");
  R* const ring = reinterpret_cast<R*>(smem);              // [4][HY][HX]
  R* const park = reinterpret_cast<R*>(smem + SM::RING);   // [2][Q][NT]
  const Geom& G = A.g;
  const int a0 = (tile % A.ntx) * TX, b0 = (tile / A.ntx) * TY;
  const int lx = tid % TX, ly = tid / TX;
  const bool active = a0 + lx < G.na && b0 + ly < G.nb;
  int4* const own_to = reinterpret_cast<int4*>(smem + SM::RING + SM::PARK) + tid;
  int4* const halo_to = own_to + NT;
  const Column me = make_column<L>(G, a0 + lx, b0 + ly, *own_to);
  const int own_at = (ly + OB) * HX + lx + 1;  // this thread's place in a plane of the ring
  const bool has_halo = tid < NH;
  int hx = 0, hy = 0;
  if (has_halo) {
    if (!L::D3) {
      hx = tid == 0 ? 0 : HX - 1;
    } else if (tid < 2 * HX) {
      hx = tid < HX ? tid : tid - HX;
      hy = tid < HX ? 0 : HY - 1;
    } else {
      const int k = tid - 2 * HX;
      hx = (k & 1) ? HX - 1 : 0;
      hy = 1 + (k >> 1);
    }
  }
  const Column hc = make_column<L>(G, a0 + hx - 1, b0 + hy - OB, *halo_to);
  const int halo_at = hy * HX + hx;
  const int pstore = G.rows * G.pitch, pcell = G.na * G.nb;

  // links of a cell of column c in plane p (kNoCell: no fluid cell there)
  auto bits_of = [&](const Column& c, const March& p, uint32_t link) -> uint32_t {
    const uint32_t w = c.wall | p.wall | (GEN ? link : 0u);
    return p.ok && !(w & kNoCell) ? w : kNoCell;
  };
  auto link_at = [&](const Column& c, int um) -> uint32_t {
    if (!GEN || !G.links || (c.wall & kNoCell)) return 0u;
    const March p = make_march<L>(G, um);
    return p.ok ? G.links[p.m * pcell + c.cell] : 0u;
  };

  V2<R> pf[Q];  // the own cell's pulled populations (PF: of the next plane to fill)
  uint32_t pf_bits = kNoCell;
  auto issue = [&](int um, uint32_t link) {
    const March p = make_march<L>(G, um);
    pf_bits = bits_of(me, p, link);
    if (!(pf_bits & kNoCell))
      pull_pairs<Q, S>(A.pin, G.nstore, *own_to, p.m * pstore + me.col, p.lo, p.hi, pf_bits, pf);
  };
  // the site byte (rules 0 and 2) and the flux of a cell
  auto extras = [&](const Column& c, const March& p, uint32_t& mb, R& phi) {
    mb = 0u;
    phi = R(0);
    if (!GEN || !p.ok || (c.wall & kNoCell)) return;
    const int cell = p.m * pcell + c.cell;
    if (A.ph.rule != 1) mb = A.mask_in[cell];
    if (A.ph.phi_field) phi = reinterpret_cast<const R*>(A.ph.phi_field)[cell];
  };

  struct Cell {
    R rr, rb, irho, lr, lb;
    uint32_t flags, bits;
  };
  uint32_t halo_link = 0u;  // of the ring cell in the next plane to fill
  Cell cur, nxt;
  nxt.rr = nxt.rb = nxt.irho = nxt.lr = nxt.lb = R(0);
  nxt.flags = 0u;
  nxt.bits = kNoCell;
  int nloc = 0;
  double rem = 0.0;
  // Fill plane um: rho^N of the tile and its ring into slot (um - m0 + 1) & 3, the own cell's
  // sums into park plane (um - m0) & 1.  count: the plane is the chunk's own (its sites count).
  auto fill = [&](int um, bool count, bool more, auto march) {
    R* const plane = ring + ((um - m0 + 1) & 3) * (HY * HX);
    R* const pk = park + ((um - m0) & 1) * (Q * NT) + tid;
    const March p = make_march<L>(G, um);
    uint32_t mb, link = 0u;
    R phi;
    extras(me, p, mb, phi);
    if (GEN && (!PF || more)) link = link_at(me, PF ? um + 1 : um);
    if (has_halo) {
      R rn = R(0);
      const uint32_t bits = bits_of(hc, p, halo_link);
      if (!(bits & kNoCell)) {
        V2<R> h[Q];
        uint32_t hmb, fl;
        R hphi, sr, sb, rr, rb, e, irho;
        extras(hc, p, hmb, hphi);
        pull_pairs<Q, S>(A.pin, G.nstore, *halo_to, p.m * pstore + hc.col, p.lo, p.hi, bits, h);
        colour_sums<Q, R>(h, sr, sb);
        rn = exchange_sums<S, GEN, false>(A.ph, hmb, hphi, sr, sb, rr, rb, e, fl, irho);
      }
      plane[halo_at] = rn;
      if (GEN && more) halo_link = link_at(hc, um + 1);
    }
    if (!PF) issue(um, link);
    V2<R> g[Q];
    nxt.bits = pf_bits;
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = pf[i];
    if (EARLY && PF && more) issue(um + 1, link);
    R rn = R(0);
    if (!(nxt.bits & kNoCell)) {
      R sr, sb, e;
      colour_sums<Q, R>(g, sr, sb);
      rn = exchange_sums<S, GEN, decltype(march)::value>(A.ph, mb, phi, sr, sb, nxt.rr, nxt.rb, e, nxt.flags, nxt.irho);
      if constexpr (ExactPairs<S>::value) {
        exact_errors<Q>(A.ph, g, sr, sb, nxt.rr, nxt.rb, e, nxt.lr, nxt.lb);
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) pk[i * NT] = i == 0 ? (g[0].r - e) + (g[0].b + e) : g[i].r + g[i].b;
      if (count && active) {
        epi.filled(A, um * pcell + me.cell, nxt.flags);
        if (nxt.flags & 1u) {
          ++nloc;
          rem += (double)e;
        }
      }
    }
    plane[own_at] = rn;
    if (!EARLY && PF && more) issue(um + 1, link);
  };

  epi.template stage<Q, S>(A, a0, b0, m0 - 1, tid);
  epi.template stage<Q, S>(A, a0, b0, m0, tid);
  if (GEN && has_halo) halo_link = link_at(hc, m0 - 1);
  if (PF) issue(m0 - 1, link_at(me, m0 - 1));
  fill(m0 - 1, false, true, std::false_type());
  fill(m0, true, true, std::false_type());
  cur = nxt;
  for (int m = m0; m < m1; ++m) {
    epi.template stage<Q, S>(A, a0, b0, m + 1, tid);
    const bool run = active && !(cur.bits & kNoCell);
    const March pm = make_march<L>(G, m);
    const int si = m * pstore + me.col;
    if (run) epi.template prefetch<Q, S>(A, si);
    fill(m + 1, m + 1 < m1, m + 1 < m1, std::integral_constant<bool, L::D3>());
    const R* pk = park + ((m - m0) & 1) * (Q * NT) + tid;
    R f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = pk[i * NT];
    const auto own = epi.template before<Q, S>(A, f, cur.rr, cur.rb, cur.irho);
    sync.wait();
    if (run) {
      const R* const pl[3] = {ring + ((m - m0) & 3) * (HY * HX) + own_at,
                              ring + ((m - m0 + 1) & 3) * (HY * HX) + own_at,
                              ring + ((m - m0 + 2) & 3) * (HY * HX) + own_at};
      R rnb[Q];
      if (cur.bits == 0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) rnb[i] = pl[1 + L::cm(i)][L::cb(i) * HX + L::ca(i)];
      } else {  // a solid neighbour, or one beyond a wall, counts as the cell itself
        const R here = pl[1][0];
#pragma unroll
        for (int i = 0; i < Q; ++i)  // x + c_i is the source of the opposite direction
          rnb[i] = (cur.bits >> opp(i)) & 1u ? here : pl[1 + L::cm(i)][L::cb(i) * HX + L::ca(i)];
      }
      epi.template cell<Q, S>(A, m * pcell + me.cell, own_to, cur.bits, pm, si, f, own, cur.rr, cur.rb, cur.irho,
                              cur.lr, cur.lb, cur.flags, rnb);
    }
    cur = nxt;
  }
  n_sites += nloc;
  // a scalar flux moves varphi at every site: n varphi in FP64, exact to one rounding
  removed += A.ph.phi_field ? rem : (double)nloc * A.ph.varphi;
}

// march(tile, m0, m1) over a CTA's planes: a chunk of one tile or (EVEN, pc = 0) an even share of
// all tiles' planes counted tile after tile.  An even share crosses a tile's end at most
// (share - 1) / nm + 1 times, each crossing costs two planes' sums, and no CTA is idle: FP64, which is
// bound by its pipe, 128^3 1424 -> 1345 us a step, 192^3 4665 -> 4435, 131 x 117 x 89 1084 -> 994.
// Not for FP32: tiles that march at different planes no longer find one another's rows in L2
// (192^3 362 -> 639 us).
template <bool EVEN, class M>
__device__ __forceinline__ void for_planes(const StepArgs& A, const M& march) {
  const int nm = A.g.nm;
  if (!EVEN || A.pc > 0) {
    const int m0 = blockIdx.y * A.pc;
    march(blockIdx.x, m0, min(m0 + A.pc, nm));
    return;
  }
  const long long all = (long long)A.ntx * A.nty * nm;
  int p = (int)(all * blockIdx.x / gridDim.x);
  const int end = (int)(all * (blockIdx.x + 1) / gridDim.x);
  while (p < end) {
    const int tile = p / nm, m0 = p - tile * nm, m1 = min(nm, m0 + end - p);
    march(tile, m0, m1);
    p += m1 - m0;
    if (p < end) __syncthreads();  // the next tile's planes take the shared memory over
  }
}

template <int Q, int S, int TX, int TY, int MINB, bool PF, bool GEN>
__global__ void __launch_bounds__(TX* TY, MINB) cg_pair_kernel(const __grid_constant__ StepArgs A) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  long long n = 0;
  double d = 0.0;
  wait_for_previous();
  for_planes<S == ST_F64>(A, [&](int tile, int m0, int m1) {
    pair_tile<Q, S, TX, TY, PF, GEN>(A, tile, m0, m1, dyn_smem, n, d, threadIdx.x, PairStep<GEN>(), CtaSync());
  });
  block_sum<TX * TY>(n, d);
  ledger_fold(A.red, n, d);
}

// ---- D2Q9 without a march ------------------------------------------------------------------------
// A plane lattice is small: marched in rows, 64^2 ran three serial fills a step on 64 CTAs (one row
// each) and 256^2 pulled three rows for each row written.  Here a CTA takes a TX x TY patch and
// every cell of the patch and of the ring around it has a thread of its own: one round of pulls,
// one barrier, the collision.  The inner cells come first, so that the warps which collide are full.
template <int TX, int TY>
struct PatchShape {
  static constexpr int NI = TX * TY, HX = TX + 2, HY = TY + 2, NR = HX * HY - NI;
  static constexpr int THREADS = NI + ((NR + 31) & ~31);
  static_assert(NI % 32 == 0, "whole warps of inner cells");
};

template <int S, int TX, int TY, bool GEN>
__global__ void __launch_bounds__(PatchShape<TX, TY>::THREADS) cg_patch_kernel(const __grid_constant__ StepArgs A) {
  constexpr int Q = 9;
  using L = Lattice<Q>;
  using R = typename Storage<S>::real;
  using P = PatchShape<TX, TY>;
  __shared__ R ring[P::HY][P::HX];
  const Geom& G = A.g;
  const int tid = threadIdx.x;
  const bool inner = tid < P::NI;
  int hx, hy;  // place in the patch with its ring
  if (inner) {
    hx = tid % TX + 1;
    hy = tid / TX + 1;
  } else {
    const int k = tid - P::NI;
    if (k < 2 * P::HX) {
      hx = k < P::HX ? k : k - P::HX;
      hy = k < P::HX ? 0 : P::HY - 1;
    } else {
      hx = (k & 1) ? P::HX - 1 : 0;
      hy = 1 + ((k - 2 * P::HX) >> 1);
    }
  }
  const int ua = blockIdx.x * TX + hx - 1, um = blockIdx.y * TY + hy - 1;
  const bool mine = inner && ua < G.na && um < G.nm;
  dependents_may_start();
  R e = R(0);
  R rr = R(0), rb = R(0), irho = R(0), lr = R(0), lb = R(0), rn = R(0);
  R f[Q];
  uint32_t flags = 0u, bits = kNoCell;
  int si = 0, cell = 0;
  PairStep<GEN> epi;
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = R(0);
  int4 to;
  March p;
  wait_for_previous();
  // ring threads past the ring, and cells beyond the first over a ragged edge, have nothing to do
  if (tid < P::NI + P::NR && um <= G.nm) {
    const Column c = make_column<L>(G, ua, 0, to);
    p = make_march<L>(G, um);
    if (p.ok && !(c.wall & kNoCell)) {
      cell = p.m * G.na + c.cell;
      bits = c.wall | p.wall;
      if (GEN && G.links) {
        const uint32_t link = G.links[cell];
        bits = link & kNoCell ? kNoCell : bits | link;
      }
    }
    if (bits != kNoCell) {
      uint32_t mb = 0u;
      R phi = R(0);
      if (GEN && A.ph.rule != 1) mb = A.mask_in[cell];
      if (GEN && A.ph.phi_field) phi = reinterpret_cast<const R*>(A.ph.phi_field)[cell];
      si = p.m * G.rows * G.pitch + c.col;
      V2<R> g[Q];
      pull_pairs<Q, S>(A.pin, G.nstore, to, si, p.lo, p.hi, bits, g);
      R sr, sb;
      colour_sums<Q, R>(g, sr, sb);
      rn = exchange_sums<S, GEN, false>(A.ph, mb, phi, sr, sb, rr, rb, e, flags, irho);
      if (mine) {
        if constexpr (ExactPairs<S>::value) exact_errors<Q>(A.ph, g, sr, sb, rr, rb, e, lr, lb);
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = i == 0 ? (g[0].r - e) + (g[0].b + e) : g[i].r + g[i].b;
        epi.filled(A, cell, flags);
      }
    }
    ring[hy][hx] = rn;
  }
  const CellMoments<R> own = cell_moments<Q, R>(A.ph, f, rr, rb, irho);
  const bool site = mine && (flags & 1u);
  const int sites = __syncthreads_count(site);
  if (GEN && A.ph.phi_field) {
    long long n = site ? 1 : 0;
    double removed = site ? (double)e : 0.0;
    block_sum<P::THREADS>(n, removed);
    ledger_fold(A.red, n, removed);
  } else if (tid == 0) {
    // a scalar flux moves varphi at every site: one 64-bit sum of arrivals (above bit 40) and sites,
    // order-free, in the place of partials, a fence and a fold by the last CTA
    const unsigned long long one = 1ull << 40, word = one | (unsigned)sites;
    const unsigned long long all = atomicAdd(A.red.tally, word) + word;
    if (all >> 40 == (unsigned long long)gridDim.x * gridDim.y) {
      const long long c = (long long)(all & (one - 1));
      const double s = (double)c * A.ph.varphi;
      DevLedger* led = A.red.ledger;
      led->evaporated += s;
      led->last_removed = s;
      led->site_steps += c;
      led->last_sites = c;
      led->steps += 1;
      *A.red.tally = 0ull;
    }
  }
  if (mine && bits != kNoCell) {
    R rnb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R v = ring[hy + L::cm(i)][hx + L::ca(i)];
      rnb[i] = (bits >> opp(i)) & 1u ? rn : v;  // a solid neighbour counts as the cell itself
    }
    epi.template cell<Q, S>(A, cell, &to, bits, p, si, f, own, rr, rb, irho, lr, lb, flags, rnb);
  }
}

template <int S, int TX, int TY>
static KernelRef patch_ref() {
  KernelRef k{(const void*)cg_patch_kernel<S, TX, TY, true>, PatchShape<TX, TY>::THREADS};
  k.tx = TX;
  k.ty = TY;
  k.plain = (const void*)cg_patch_kernel<S, TX, TY, false>;
  k.pdl = 1;
  return k;
}
// Patches of 16 x 8 cells were the fastest or level with the fastest of 8 x 4, 8 x 8, 32 x 4, 16 x 8 and
// 32 x 8 from 64^2 to 1024^2 (us per step at 64^2 / 256^2 / 1024^2, FP32: 3.3 / 4.6 / 28.1; marched 8.7 /
// 11.3 / 38.2; F32X 3.4 / 4.9 / 33.0, marched 9.4 / 11.6 / 39.5).  FP64 is held by the FP64 pipe of the
// SMs it runs on: 8 x 4 until every SM has four of them (64^2: 8.7 against 10.0, marched 19.6), then
// 16 x 8 (256^2 29.0, marched 43.1; 1024^2 363, marched 371).
template <int S>
static KernelRef patch_pick(long long cells) {
  if (S == ST_F64 && cells <= 152LL * 4 * 32) return patch_ref<S, 8, 4>();
  return patch_ref<S, 16, 8>();
}

// The launch record of a pair kernel: the general instantiation and the plain one.
template <int Q, int S, int TX, int TY, int MINB, bool PF>
static KernelRef pair_ref() {
  constexpr int smem = PairSmem<Q, S, TX, TY>::BYTES;
  const void* fn = (const void*)cg_pair_kernel<Q, S, TX, TY, MINB, PF, true>;
  const void* plain = (const void*)cg_pair_kernel<Q, S, TX, TY, MINB, PF, false>;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(plain, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
      return {nullptr, 0};
    attr = true;
  }
  KernelRef k{fn, TX * TY};
  k.smem = smem;
  k.tx = TX;
  k.ty = TY;
  k.plain = plain;
  k.pdl = 1;
  k.shares = S == ST_F64 ? 1 : 0;
  return k;
}

}  // namespace cgevap
