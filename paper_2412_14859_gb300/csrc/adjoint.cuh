// adjoint.cuh -- reverse-mode derivative of one fused step with respect to its input state and
// the flux field, with the site set x_I of the step held fixed.
//
// The step maps the stored state f^n to f^{n+1}: for every fluid cell x
//   g(x)    = pulled populations (Eq. Stream, halfway bounce-back), then Eq. (exchange):
//             g_0^r -= m(x) phi(x)/S-bar, g_0^b += m(x) phi(x)/S-bar;
//   F(x)    = 3 sum_i W_i c_i rho^N(n_i(x)),  n_i(x) = x + c_i, or x where x + c_i is solid or
//             beyond a wall (Eq. cg), rho^N = (rho_r - rho_b)/rho of the post-exchange g;
//   f^{n+1}(x) = C(g(x), F(x)): Eq. (feq), (collision), (perturb), (recolor).
// Given lambda^{n+1} = dL/df^{n+1} and w = dL/dV(n+1) for the observable
// V(n+1) = sum_x (1 + rho^N(x))/2 (the stored densities of f^{n+1} are those of g: the
// collision, the perturbation and the recoloring conserve rho_r and rho_b per cell), the sweep is
//   (1) local:   lg(x) = (dC/dg)^T lambda^{n+1}(x),  lF(x) = (dC/dF)^T lambda^{n+1}(x),
//                plus d rho^N/d(rho_r, rho_b) = (2 rho_b, -2 rho_r)/rho^2          [kernel A]
//   (2) stencil: mu(y) = w/2 + sum_{(x,i): n_i(x) = y} 3 W_i c_i . lF(x);
//                lg_total(y) = lg(y) + mu(y) d rho^N/d(rho_r, rho_b) on every direction;
//                dL/dphi(y) += m(y) (lg_total_0^b(y) - lg_total_0^r(y)) / S-bar     [kernel B1]
//   (3) pull^T:  lambda^n_j(y) = lg_total_j(y + c_j), or lg_total_{opp j}(y) where y + c_j is
//                solid or beyond a wall (the transpose of the pull with bounce-back): kernel A
//                pushes the lg part to where the pull read from, the next kernel A adds the ab
//                part of the writer as it reads lambda^{n+1}
// Kernel A recomputes the forward quantities of its tile exactly as the step does (it runs the
// step's own tile code with this file's epilogue in place of the collision and store).
#pragma once

#include "launch.h"
#include "pair_tile.cuh"

namespace cgevap {

// Minority fraction product w_r w_b below which the adjoint holds the recoloring direction fixed.
constexpr double kBulkTrace = 1e-6;

// Pull source of direction i from storage index si (see pull_pairs).
template <class L>
__device__ __forceinline__ int pull_source(int4 to, int lo, int hi, int si, int i) {
  return si + (L::ca(i) > 0 ? to.x : (L::ca(i) < 0 ? to.y : 0)) +
         (L::cb(i) > 0 ? to.z : (L::cb(i) < 0 ? to.w : 0)) + (L::cm(i) > 0 ? lo : (L::cm(i) < 0 ? hi : 0));
}

// (1) for one cell: from its moments c0, F and the colour-blind sums f of its post-exchange
// populations, the terms of collide_pairs run backwards.  lam_at(i): lambda^{n+1} of direction i
// (read where it is used); out: lg_out(i, v) takes lg_i = dL/dg_i through this cell's own
// collision, lF = dL/dF.
//
// With d_i = lambda^r_i - lambda^b_i and q_i = w_r d_i + lambda^b_i (dL/d of the colour-blind
// output), the derivative with respect to every per-cell quantity is a polynomial in c_i.u and
// c_i.e (e = F/|F|) summed over directions, so per speed class s it needs only
//   scalars  D0 = sum d, Q0 = sum q, DU = sum d (c.u)^2, DN = sum d (c.e)^2,
//   vectors  DV = sum d c, QV = sum q c, UV = sum q (c.u) c, PV = sum q (c.e) c,
// plus sum d f and sum q f; opposite directions enter as sums and differences.  Kernel A is bound
// by its instruction count, and this takes about 16 operations a direction where running each
// direction's own chain backwards took about 45: FP32, 1.57 M cells under ncu, 99.4 M warp
// instructions and 228 us before, 84.9 M and 177 us with it and with the pulls a plane ahead
// (72.1 -> 69.3 ms a fit iteration of 32 steps on the full cap for the latter); FP64 fit on the
// reduced cap 15.6 -> 12.6 ms.  At 128 registers (four CTAs per SM) it spills: 87 ms.
//
// Where w_r w_b < kBulkTrace (bulk: one colour is a trace) the recoloring direction e is held
// fixed: that term is homogeneous of degree 1 in the trace, so its derivative with respect to F
// stays O(beta w_r / |F|) however small the trace, and the linearised trace dynamics grows
// without bound while the traces themselves stay negligible.
template <int Q, class R, class LamAt, class LgOut>
__device__ __forceinline__ void collide_adjoint(const Physics& ph, const CellMoments<R>& c0, const R (&f)[Q],
                                                R irho, R Fa, R Fb, R Fm, const LamAt& lam_at,
                                                const LgOut& lg_out, R (&lF)[3]) {
  using L = Lattice<Q>;
  const R rho = c0.rho, wr = c0.wr, wb = c0.wb, itau = c0.itau, uu15 = c0.uu15;
  const R u[3] = {c0.ua, c0.ub, c0.um};
  const R ir = PHYS(R, ph, inv_tau_r), ib = PHYS(R, ph, inv_tau_b);
  R F2 = fma(Fa, Fa, Fm * Fm);
  if (L::D3) F2 = fma(Fb, Fb, F2);
  R Fn = R(0), iFn = R(0);
  if (F2 > R(0)) norm_of(F2, Fn, iFn);
  const R e[3] = {Fa * iFn, Fb * iFn, Fm * iFn};
  // sums over the directions of speed classes 1 and 2 (index 0: the rest direction)
  R D0[3], Q0[3], DU[3], DN[3], DV[3][3], QV[3][3], UV[3][3], PV[3][3], q[Q];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    D0[s] = Q0[s] = DU[s] = DN[s] = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) DV[s][k] = QV[s][k] = UV[s][k] = PV[s][k] = R(0);
  }
  R Sdf, Sqf;
  {
    const V2<R> l = lam_at(0);
    D0[0] = l.r - l.b;
    q[0] = Q0[0] = fma(wr, D0[0], l.b);
    Sdf = D0[0] * f[0];
    Sqf = q[0] * f[0];
  }
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int j = i + 1, s = L::speed2(i);
    const V2<R> li = lam_at(i), lj = lam_at(j);
    const R di = li.r - li.b, dj = lj.r - lj.b;
    q[i] = fma(wr, di, li.b);
    q[j] = fma(wr, dj, lj.b);
    Sdf = fma(dj, f[j], fma(di, f[i], Sdf));
    Sqf = fma(q[j], f[j], fma(q[i], f[i], Sqf));
    const R qs = q[i] + q[j], qd = q[i] - q[j], ds = di + dj, dd = di - dj;
    R cu = R(0), ce = R(0);
    bool any = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int c = axis_comp<L>(i, k);
      if (!c) continue;
      cu = any ? (c > 0 ? cu + u[k] : cu - u[k]) : (c > 0 ? u[k] : -u[k]);
      ce = any ? (c > 0 ? ce + e[k] : ce - e[k]) : (c > 0 ? e[k] : -e[k]);
      any = true;
    }
    Q0[s] += qs;
    D0[s] += ds;
    DU[s] = fma(ds * cu, cu, DU[s]);
    DN[s] = fma(ds * ce, ce, DN[s]);
    const R qu = qs * cu, qe = qs * ce;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int c = axis_comp<L>(i, k);
      if (!c) continue;
      DV[s][k] = c > 0 ? DV[s][k] + dd : DV[s][k] - dd;
      QV[s][k] = c > 0 ? QV[s][k] + qd : QV[s][k] - qd;
      UV[s][k] = c > 0 ? UV[s][k] + qu : UV[s][k] - qu;
      PV[s][k] = c > 0 ? PV[s][k] + qe : PV[s][k] - qe;
    }
  }
  const R amp = PHYS(R, ph, amp), beta = PHYS(R, ph, beta);
  const R pamp = amp * itau, rcol = beta * wr * wb;
  const R rdir = wr * wb < R(kBulkTrace) ? R(0) : rcol;  // bulk: e fixed
  R A_rcol = R(0), A_rho = R(0), A_abar = R(0), A_uu15 = R(0), Sqeq = R(0), Sdeq = R(0);
  R Spert_q = R(0), Spert_d = R(0), Sn = R(0), Sg = R(0);
  R Au[3] = {R(0), R(0), R(0)}, P[3] = {R(0), R(0), R(0)}, G[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int i = s == 0 ? 0 : (s == 1 ? 1 : L::Q - 1);  // a direction of speed class s
    const R W = R(L::W(i)), C = R(L::C(i)), nrm = R(inv_norm<L>(i));
    const R rest1 = fma(R(L::B(i)), c0.abar, R(L::A(i)));  // f_i^eq(rho, 0) / rho
    const R restc = rho * rest1, rw = rho * W;
    R qpoly = -uu15 * Q0[s], dpoly = -uu15 * D0[s], A_rest = itau * Q0[s];
    if (s > 0) {
      R uUV = R(0), uQV = R(0), uDV = R(0), eDV = R(0), ePV = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (!L::D3 && k == 1) continue;
        uUV = fma(u[k], UV[s][k], uUV);
        uQV = fma(u[k], QV[s][k], uQV);
        uDV = fma(u[k], DV[s][k], uDV);
        eDV = fma(e[k], DV[s][k], eDV);
        ePV = fma(e[k], PV[s][k], ePV);
      }
      // Eq. (feq): sums of q and d times rho W (9/2 (c.u)^2 + 3 c.u - 3/2 u^2)
      qpoly = fma(R(4.5), uUV, fma(R(3), uQV, qpoly));
      dpoly = fma(R(4.5), DU[s], fma(R(3), uDV, dpoly));
      // Eq. (recolor): rcol nrm restc (c.e)
      A_rcol = fma(nrm * restc, eDV, A_rcol);
      A_rest = fma(rcol * nrm, eDV, A_rest);
      const R kg = rdir * nrm * restc;
      Sg = fma(kg, eDV, Sg);
      const R rwt = itau * rw;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (!L::D3 && k == 1) continue;
        G[k] = fma(kg, DV[s][k], G[k]);
        P[k] = fma(R(2) * W, PV[s][k], P[k]);
        Au[k] = fma(rwt, fma(R(9), UV[s][k], R(3) * QV[s][k]), Au[k]);
      }
      // Eq. (perturb): |F| (W (c.e)^2 - C)
      Sn = fma(W, ePV, Sn);
      Spert_q = fma(W, ePV, Spert_q);
      Spert_d = fma(W, DN[s], Spert_d);
    }
    Sn = fma(C, Q0[s], Sn);
    Spert_q = fma(-C, Q0[s], Spert_q);
    Spert_d = fma(-C, D0[s], Spert_d);
    Sqeq = fma(rw, qpoly, fma(restc, Q0[s], Sqeq));
    Sdeq = fma(rw, dpoly, fma(restc, D0[s], Sdeq));
    A_uu15 = fma(-itau * rw, Q0[s], A_uu15);
    // restc = rho (A + B abar), rw = rho W
    A_rho = fma(A_rest, rest1, fma(itau * qpoly, W, A_rho));
    A_abar = fma(A_rest, rho * R(L::B(i)), A_abar);
  }
  const R A_pamp = Fn * Spert_q;
  // f_i' = f_i + itau (feq_i - f_i) + pamp pert_i;  f^r_i = wr f_i' + recoloring
  const R A_itau = fma(amp, A_pamp, Sqeq - Sqf);
  R A_wr = fma(itau, Sdeq - Sdf, fma(pamp, Fn * Spert_d, Sdf));
  A_wr = fma(A_rcol, beta * wb, fma(A_itau, ir, fma(A_abar, PHYS(R, ph, alpha_r), A_wr)));
  const R A_wb = fma(A_rcol, beta * wr, fma(A_itau, ib, A_abar * PHYS(R, ph, alpha_b)));
  // u = j / rho, uu15 = 3/2 |u|^2
  R Aj[3], Auu = R(0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const R a = fma(R(3) * A_uu15, u[k], Au[k]);
    Auu = fma(a, u[k], Auu);
    Aj[k] = a * irho;
  }
  A_rho = fma(-Auu, irho, A_rho);
  // dL/dF = 2 pamp sum W q (c.e) c - pamp Sn e + (G - Sg e) / |F| (zero where F = 0)
  const R se = fma(pamp, Sn, Sg * iFn);
#pragma unroll
  for (int k = 0; k < 3; ++k) lF[k] = fma(pamp, P[k], fma(G[k], iFn, -se * e[k]));
  // wr = rr / rho, wb = rb / rho, rho = rr + rb
  const R A_rr = fma((A_wr - A_wb) * wb, irho, A_rho);
  const R A_rb = fma((A_wb - A_wr) * wr, irho, A_rho);
  const R keep = R(1) - itau;
  lg_out.each([&](int i) -> V2<R> {
    R a = keep * q[i];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int c = axis_comp<L>(i, k);
      if (c) a = c > 0 ? a + Aj[k] : a - Aj[k];
    }
    return {a + A_rr, a + A_rb};
  });
}

// The auxiliary fields of kernel A: per cell (dL/dF_a, dL/dF_b, dL/dF_m, d rho^N/d rho_r) side by
// side, so that B1 takes a neighbour's gradient in one 16-byte load (two for FP64), and after those
// nstore cells a plane of d rho^N/d rho_b (a fit iteration of 32 steps on the full cap 72.56 ms with
// five planes, 72.26 so; at six or four CTAs per SM instead of eight 72.65 and 73.74).
template <class R>
struct AuxCell;
template <>
struct AuxCell<float> {
  float a, b, m, dr;
  static __device__ __forceinline__ AuxCell load(const void* aux, int si) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(aux) + si);
    return {v.x, v.y, v.z, v.w};
  }
  static __device__ __forceinline__ void store(void* aux, int si, const float (&F)[3], float dr) {
    reinterpret_cast<float4*>(aux)[si] = make_float4(F[0], F[1], F[2], dr);
  }
};
template <>
struct AuxCell<double> {
  double a, b, m, dr;
  static __device__ __forceinline__ AuxCell load(const void* aux, int si) {
    const double2* p = reinterpret_cast<const double2*>(aux) + 2 * (size_t)si;
    const double2 v = __ldg(p), w = __ldg(p + 1);
    return {v.x, v.y, w.x, w.y};
  }
  static __device__ __forceinline__ void store(void* aux, int si, const double (&F)[3], double dr) {
    double2* p = reinterpret_cast<double2*>(aux) + 2 * (size_t)si;
    p[0] = make_double2(F[0], F[1]);
    p[1] = make_double2(F[2], dr);
  }
};

// lg_i goes where the pull read g_i from: slot i of x - c_i, or slot opp(i) of x for a bounced link
// (element index in 32 bits: a state holds Q nstore < 2^31 vec2).
template <int Q, class R, class Vec>
struct PullPush {
  Vec* out;
  int ns, si, lo, hi;
  int4 to;
  uint32_t bits;
  template <class V>
  __device__ __forceinline__ void each(const V& value) const {
    using L = Lattice<Q>;
    if (bits == 0) {
#pragma unroll
      for (int i = 0; i < Q; ++i) put(i * ns + pull_source<L>(to, lo, hi, si, i), value(i));
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        put((bits >> i) & 1u ? opp(i) * ns + si : i * ns + pull_source<L>(to, lo, hi, si, i), value(i));
    }
  }
  __device__ __forceinline__ void put(int at, V2<R> v2) const {
    Vec v;
    v.x = v2.r;
    v.y = v2.b;
    out[at] = v;
  }
};

// Kernel A's per-cell tail (in the place of PairStep in pair_tile).  It reads lambda^{n+1} and
// writes the transpose of the pull of step n directly:
//   lambda^n_j(y) = lg_j(y + c_j) + ab(y + c_j), or lg_{opp j}(y) + ab(y) where y + c_j is solid
// or beyond a wall, with ab = mu d rho^N / d(rho_r, rho_b) from kernel B1 of the same step.  Its
// lg part is pushed here, each cell x writing lg_i(x) where the pull read g_i(x) from -- slot i
// of x - c_i, or slot opp(i) of x itself for a bounced link -- so every slot of a fluid cell has
// exactly one writer.  The ab part is added by the reader: the next adjoint step's kernel A reads
// the pushed values of its own cell (lam_in) and the ab of the writer, x = y + c_j, from a box
// of the tile's neighbourhood staged in shared memory per plane.  lambda^{n+1} of a cell of plane
// m is copied into this thread's shared-memory column `lam` (Q vec slots, stride TX TH) by prefetch(),
// at the start of the iteration that collides plane m, so the copies overlap the pulls of plane
// m + 1; cell() waits for them.  The ab box has four plane slots (m - 1 .. m + 2 in flight): plane
// um is staged at the start of the iteration that collides um - 1, and its slot was last read by
// the collision of um - 4, two barriers earlier.
template <int TX, int TH>
struct AdjointEpilogue {
  AdjointOut o;
  unsigned char* lam;   // this thread's column: Q slots of sizeof(vec), stride TX TH slots
  unsigned char* abox;  // [4][BY][BX] vec: ab of the planes in flight, one-cell halo

  template <int Q>
  static constexpr int box_x() { return TX + 2; }
  template <int Q>
  static constexpr int box_y() { return Lattice<Q>::D3 ? TH + 2 : 1; }
  template <int Q, int S>
  static constexpr int box_bytes() {
    return 4 * box_x<Q>() * box_y<Q>() * (int)sizeof(typename Storage<S>::vec);
  }

  template <int Q, int S>
  __device__ __forceinline__ void prefetch(const StepArgs& A, int si) const {
    using Vec = typename Storage<S>::vec;
    const int ns = A.g.nstore;
    const Vec* lin = reinterpret_cast<const Vec*>(o.lam_in);
    Vec* col = reinterpret_cast<Vec*>(lam);
#pragma unroll
    for (int i = 0; i < Q; ++i) async_copy<sizeof(Vec)>(col + i * (TX * TH), lin + (size_t)i * ns + si);
    async_commit();
  }
  // ab of plane um (unwrapped) over the tile and its one-cell halo into slot um & 3
  template <int Q, int S>
  __device__ __forceinline__ void stage(const StepArgs& A, int a0, int b0, int um, int tid) const {
    using L = Lattice<Q>;
    using Vec = typename Storage<S>::vec;
    constexpr int BX = box_x<Q>(), BY = box_y<Q>(), NB = BX * BY, NT = TX * TH;
    const Geom& G = A.g;
    const Plane p = make_plane(G, um);
    if (!p.ok) return;  // beyond a wall: never read (those links bounce back)
    const Vec* ab = reinterpret_cast<const Vec*>(o.ab);
    Vec* box = reinterpret_cast<Vec*>(abox) + (um & 3) * NB;
    for (int e = tid; e < NB; e += NT) {
      int a = a0 - 1 + e % BX, b = L::D3 ? b0 - 1 + e / BX : 0;
      bool ok = true;
      if (a < 0 || a >= G.na) {
        if (G.per_a) a = wrap(a, G.na); else ok = false;
      }
      if (L::D3 && (b < 0 || b >= G.nb)) {
        if (G.per_b) b = wrap(b, G.nb); else ok = false;
      }
      if (ok) box[e] = __ldg(ab + sidx(G, a, b, p.m));
    }
  }
  template <int Q, int S, class R>
  __device__ __forceinline__ CellMoments<R> before(const StepArgs& A, const R (&f)[Q], R rr, R rb, R irho) const {
    return cell_moments<Q, R>(A.ph, f, rr, rb, irho);
  }
  __device__ __forceinline__ void filled(const StepArgs&, int, uint32_t) const {}
  template <int Q, int S, class R>
  __device__ __forceinline__ void cell(const StepArgs& A, int /*cell*/, const int4* own_to, uint32_t sbits,
                                       const March& pm, int si, const R (&f)[Q], const CellMoments<R>& c,
                                       R rr, R rb, R irho, R, R, uint32_t /*flags*/,
                                       const R (&rnb)[Q]) const {
    using L = Lattice<Q>;
    using Vec = typename Storage<S>::vec;
    constexpr int BX = box_x<Q>(), NB = BX * box_y<Q>();
    const int m = pm.m;
    const int4 to = *own_to;
    const int ns = A.g.nstore;
    Vec* lout = reinterpret_cast<Vec*>(o.lam_g);
    // this cell's place in the ab box: the thread's own column of the tile (one cell per thread
    // and plane), one in from the halo
    const int bx = (int)threadIdx.x % TX + 1;
    const int by = L::D3 ? (int)threadIdx.x / TX + 1 : 0;
    const Vec* box = reinterpret_cast<const Vec*>(abox);
    const Vec* const here[3] = {box + ((m - 1) & 3) * NB + by * BX + bx, box + (m & 3) * NB + by * BX + bx,
                                box + ((m + 1) & 3) * NB + by * BX + bx};
    async_wait_all();  // this thread's copies of plane m (only it reads its column)
    const Vec* col = reinterpret_cast<const Vec*>(lam);
    auto lam_at = [&](int i) -> V2<R> {
      const Vec v = col[i * (TX * TH)];
      // ab of the slot's writer: x = y + c_i, or y itself where y + c_i is solid (the source of
      // this cell's direction opp(i))
      const bool self = i == 0 || ((sbits >> opp(i)) & 1u);
      const Vec w = *(self ? here[1] : here[1 + L::cm(i)] + L::cb(i) * BX + L::ca(i));
      return {v.x + w.x, v.y + w.y};
    };
    const PullPush<Q, R, Vec> lg_out{lout, ns, si, pm.lo, pm.hi, to, sbits};
    R lF[3];
    R Fa, Fb, Fm;
    colour_gradient<Q, R>(rnb, Fa, Fb, Fm);
    collide_adjoint<Q, R>(A.ph, c, f, irho, Fa, Fb, Fm, lam_at, lg_out, lF);
    AuxCell<R>::store(o.aux, si, lF, R(2) * rb * irho * irho);  // ... and d rho^N / d rho_r
    reinterpret_cast<R*>(o.aux)[4 * ns + si] = -R(2) * rr * irho * irho;  // d rho^N / d rho_b
  }
};

template <int Q, int S, int TX, int TY>
__global__ void __launch_bounds__(TX* TY, (S == ST_F64 ? 256 : 384) / (TX * TY))
    cg_adjoint_local_kernel(const __grid_constant__ StepArgs A,
                            const __grid_constant__ AdjointOut O) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  long long n = 0;
  double d = 0.0;
  using Vec = typename Storage<S>::vec;
  using Epi = AdjointEpilogue<TX, TY>;
  // lambda columns after the tile's own shared memory (slot i of thread t at i TX TY + t), then
  // the ab box
  constexpr int lam_bytes = Q * TX * TY * (int)sizeof(Vec);
  unsigned char* const lam0 = dyn_smem + PairSmem<Q, S, TX, TY>::BYTES;
  const Epi E{O, lam0 + threadIdx.x * sizeof(Vec), lam0 + lam_bytes};
  const int m0 = blockIdx.y * A.pc;
  pair_tile<Q, S, TX, TY, true, true>(A, blockIdx.x, m0, min(m0 + A.pc, A.g.nm), dyn_smem, n, d, threadIdx.x, E,
                                      CtaSync());
}

// (2) one thread per cell.  dLdV: pointer to dL/dV(n+1) (nullptr: 0).  The kernel was bound by its
// integer instructions (47 % of them; two divisions a cell for the coordinates), so the coordinates
// come from the launch: blocks of kStencilX x 256 / kStencilX cells of a plane (a row in 2D), planes
// along grid z, both strided where the grid is smaller than the lattice.
template <int Q>
__host__ __device__ constexpr int stencil_x() { return Q == 19 ? 64 : 256; }

template <int Q, class R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 8 : 5)  // FP32: 32 registers, all warps resident
    cg_adjoint_stencil_kernel(Geom G, const R* __restrict__ aux, const void* __restrict__ lam_g,
                              void* __restrict__ ab, const uint8_t* __restrict__ mask,
                              double* __restrict__ dphi, double inv_sbar,
                              const double* __restrict__ dLdV) {
  using L = Lattice<Q>;
  using Vec = typename std::conditional<sizeof(R) == 8, double2, float2>::type;
  constexpr int BX = stencil_x<Q>(), BY = 256 / BX;
  const int a = blockIdx.x * BX + threadIdx.x % BX;
  if (a >= G.na) return;
  const R w0 = dLdV ? R(0.5 * __ldg(dLdV)) : R(0);
  for (int m = blockIdx.z; m < G.nm; m += gridDim.z)
    for (int b = blockIdx.y * BY + threadIdx.x / BX; b < G.nb; b += gridDim.y * BY) {
      const int cell = (m * G.nb + b) * G.na + a;
      const Slot sl = make_slot<L>(G, a, b);
      const Plane p = make_plane(G, m);
      uint32_t bits = 0;
      if (!solid_bits<L>(G, sl, p, cell, bits)) continue;
      const PlaneOffsets po = plane_offsets(G, m);
      const int4 to = make_int4(sl.dxm, sl.dxp, sl.dym, sl.dyp);
      const int si = sidx(G, a, b, m);
      const int ns = G.nstore;  // 5 ns < Q nstore < 2^31
      const AuxCell<R> own = AuxCell<R>::load(aux, si);
      R mu = w0;
      auto along = [](int i, const AuxCell<R>& F) {  // F . c_i
        R t = R(0);
        if (L::ca(i)) t += R(L::ca(i)) * F.a;
        if (L::cb(i)) t += R(L::cb(i)) * F.b;
        if (L::cm(i)) t += R(L::cm(i)) * F.m;
        return t;
      };
      auto from = [&](int i) {  // F of x = y - c_i used rho^N(y) with weight 3 W_i c_i
        const int src = pull_source<L>(to, po.dm_lo, po.dm_hi, si, i);
        const AuxCell<R> F = AuxCell<R>::load(aux, src);
        return along(i, F);
      };
      if (bits == 0) {
#pragma unroll
        for (int i = 1; i < Q; ++i) mu += R(3.0 * L::W(i)) * from(i);
      } else {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          R t = R(0);
          if (!((bits >> i) & 1u)) t = from(i);  // x = y - c_i is fluid
          if ((bits >> opp(i)) & 1u)  // y + c_i is solid: y's own F used rho^N(y) in its place
            t += along(i, own);
          mu += R(3.0 * L::W(i)) * t;
        }
      }
      Vec v;
      v.x = mu * own.dr;
      v.y = mu * aux[4 * ns + si];
      reinterpret_cast<Vec*>(ab)[si] = v;
      if (mask[cell] & 1u) {  // Eq. (exchange): d g_0^r / d phi = -1/S-bar, d g_0^b / d phi = +1/S-bar
        const Vec l0 = reinterpret_cast<const Vec*>(lam_g)[si];
        dphi[cell] += ((double)(l0.y + v.y) - (double)(l0.x + v.x)) * inv_sbar;
      }
    }
}

__device__ __forceinline__ void cell_coords(const Geom& g, int cell, int& a, int& b, int& m) {
  a = cell % g.na;
  const int t = cell / g.na;
  b = t % g.nb;
  m = t / g.nb;
}

// V = sum over fluid cells of (1 + rho^N)/2 of a stored state, FP64, deterministic: fixed grid,
// per-block partials, the last block to arrive adds them in block order into *out.
template <int Q, int S>
__global__ void __launch_bounds__(256)
    cg_volume_kernel(Geom G, Physics ph, const void* __restrict__ state, double* __restrict__ part,
                     unsigned int* __restrict__ done, double* __restrict__ out) {
  using R = typename Storage<S>::real;
  __shared__ double red[8];
  __shared__ int is_last;
  double v = 0.0;
  const int stride = gridDim.x * blockDim.x;
  for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < G.ncell; cell += stride) {
    if (G.links && (__ldg(G.links + cell) >> 31)) continue;
    int a, b, m;
    cell_coords(G, cell, a, b, m);
    const int si = sidx(G, a, b, m);
    R rr = R(0), rb = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const V2<R> f = PopIO<S, Q>::load(state, G.nstore, i, i, si, ph);
      rr += f.r;
      rb += f.b;
    }
    // the liquid fraction in the storage's arithmetic (an FP64 division per cell would hold the
    // FP32 kernel to GB300's FP64 rate), summed in FP64
    v += (double)(rr / (rr + rb));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int tid = threadIdx.x;
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    part[blockIdx.x] = s;
    __threadfence();
    is_last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (is_last && tid < 32) {
    __threadfence();
    double s = 0.0;
    for (unsigned j = tid; j < gridDim.x; j += 32) s += __ldcg(part + j);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (tid == 0) {
      *out = s;
      *done = 0u;
    }
  }
}

}  // namespace cgevap
