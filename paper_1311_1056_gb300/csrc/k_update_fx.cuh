// k_update_fx.cuh -- the CL step of the FP64 and DF64 forms (link type L) in
// 64-bit fixed point (fixed.cuh): link copies and inverses, plaquettes, clover field and
// per-plaquette drift, the same quantities and formulas as k_update.cuh.
//
// Fields between the kernels (int4 words, SoA as the links): Ux, the links in
// fixed point, in the buffer that the update writes at the step's end; Ui
// their inverses; P, D, F, C.  F is an eighth of the clover field, negated for
// planes 1 and 4 (the sign of the pair 02|13), times 2^k that keeps the lattice's
// largest D / 2 just below the bound (fx_field_shift); its factor -i theta kappa (s below)
// comes in where the force is formed, times 2^-e, the factor that keeps the
// contributions C within bounds (drift_exponent, launch.h).
//
// A fixed-point number's error is the same whatever its size, ~1e-17, so fields are
// kept as large as the bounds allow.  (With F held times s 2^-e and C four times
// smaller, errors against 80-bit arithmetic on links scattered by 0.27: drift at
// theta = 1 1.3e-15 of its size, charge density 1.6e-15; now 1.5e-16 and 4.4e-16; FP64
// arithmetic 2.7e-16 and 4.5e-16.)
//
// A thread whose inputs or results leave the fixed-point range calls the
// general path, FP64 on the same fields (the whole warp for one plaquette,
// general_warp.cuh, or the bodies of k_update.cuh), for its plaquette; that code is out of line and costs the others nothing.
//
// Scales that keep every number within the fixed-point bound: D is stored
// halved (|D| < 2.9), the sums of leaves are averages, the sum of the dual fields
// over a plaquette's corners is a quarter.
#pragma once
#include "fixed.cuh"
#include "general_warp.cuh"
#include "k_update.cuh"
#include "link_fx.cuh"
#include "noise_fx.cuh"

namespace clgc {

// Fields of the general path.
__device__ __forceinline__ tagged tag(const int4* f) { return tagged{const_cast<int4*>(f), 0}; }
// the clover field (kept times 2^k / 8) times s
__device__ __forceinline__ tagged_c tag_F(const int4* f, int k, double sre, double sim) {
  return tagged_c{tagged{const_cast<int4*>(f), 3 - k}, cx<double>{sre, sim}};
}
__device__ __forceinline__ tagged tag_D(const int4* f) { return tagged{const_cast<int4*>(f), 1}; }

// The operands of the products come through an fx_pipe of two slots (fixed.cuh):
// 32^4: plaquettes and clover field 2.60 -> 2.48 ms a step, observables 3.03 ->
// 2.92 ms (2.59 and 3.03 since their sums are the fine ones).
const int FX_BLOCK = FX_PIPE_THREADS;  // largest block of the kernels that use it
const int FX_PIPE = fx_pipe<2>::WORDS, FX_PARK_BYTES = (FX_PIPE + fx_park::WORDS) * (int)sizeof(int4);

// ------------------------------------------------------ links and inverses
template <typename L>
__device__ __forceinline__ void fx_links_body(Geo g, const typename vec2_of<L>::type* __restrict__ U,
                                              int4* __restrict__ Ux, int4* __restrict__ Ui, unsigned* top, int vb) {
  if (vb == 0 && threadIdx.x == 0) *top = 0u;  // for the plaquette pass
  const int mu = vb % 4;
  const int s = (vb / 4) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  mat<fx> x, xi;
  const bool in = fx_load_link<L>(x, U, mu, s, g.V);
  fx_chk ck;
  fx_adj<fx_acc_fine>(xi, x, ck);
  if (!in || ck.bad()) {  // readers of either turn to U itself
    x.e[0].re.l = fx_raw_mark();
    xi.e[0].re.l = fx_raw_mark();
  }
  store<fx>(Ux, mu, s, g.V, x);
  store<fx>(Ui, mu, s, g.V, xi);
}

// ------------------------------------------------------------- plaquettes
// (a - b) / 2
__device__ __forceinline__ fx fx_half_diff(fx a, fx b) {
  const int d = (a.h >> 1) - (b.h >> 1), odd = (a.h & 1) - (b.h & 1);  // a.h - b.h = 2 d + odd
  return fx{fmaf(0.5f, a.l - b.l, (float)odd * 0x1p29f), d};
}
template <typename L>
static __device__ __noinline__ void general_plaq(Geo g, const typename vec2_of<L>::type* U, tagged Pq, tagged Dq, int vb) {
  k_plaq_body<double>(g, link_field<L>{U}, Pq, Dq, vb);
}
template <typename L>
__device__ __forceinline__ void fx_plaq_body(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                             const int4* __restrict__ Ui, int4* Pq, int4* Dq, unsigned* top, int4* sm,
                                             int vb) {
  const int p = vb % 6, mu = plane_mu(p), nu = plane_nu(p);
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int x[4];
  site_coords(g, s, x);
  fx_chk ck;
  mat<fx> Pm, b;
  fx_pipe<2> P(sm);
  P.ask(Ux, mu, s, g.V);
  P.ask(Ux, nu, hop(g, s, x, mu, 1), g.V);
  P.take(Pm, ck);
  P.ask(Ui, mu, hop(g, s, x, nu, 1), g.V);
  P.take(b, ck);
  P.ask(Ui, nu, s, g.V);
  fx_mul_left<FX_WIDE, 0, fx_acc_fine>(Pm, b, ck);
  P.take(b, ck);
  fx_mul_left<FX_WIDE, 0, fx_acc_fine>(Pm, b, ck);
  P.take(b, ck);
  fx_mul_left<FX_WIDE, 0, fx_acc_fine>(Pm, b, ck);
  fx_adj<fx_acc_fine>(b, Pm, ck);
  store<fx>(Pq, p, s, g.V, Pm);
#pragma unroll
  for (int k = 0; k < 9; ++k) Pm.e[k] = cx<fx>{fx_half_diff(Pm.e[k].re, b.e[k].re), fx_half_diff(Pm.e[k].im, b.e[k].im)};
  store<fx>(Dq, p, s, g.V, Pm);
  {
    int hi = ck.bad() ? 1 << 30 : 0, lo = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      hi = max(hi, max(Pm.e[k].re.h, Pm.e[k].im.h));
      lo = min(lo, min(Pm.e[k].re.h, Pm.e[k].im.h));
    }
    const int n = g.V - (s - (int)(threadIdx.x & 31));  // the warp's sites
    const unsigned m = __reduce_max_sync(n >= 32 ? 0xffffffffu : (1u << n) - 1u, (unsigned)max(hi, -lo));
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned*)top) atomicMax(top, m);
  }
  general_path(ck.bad(), s, g.V, [&](unsigned m, int t) { warp_plaq<L>(m, g, U, tag(Pq), tag_D(Dq), p, t); },
               [&] { general_plaq<L>(g, U, tagged{Pq, 0, 0u}, tag_D(Dq), vb); });
}

// ------------------------------------------------------------ clover field
template <typename L>
static __device__ __noinline__ void general_clover(Geo g, const typename vec2_of<L>::type* U, tagged Dq, tagged F, double scale, int vb) {
  k_clover_rot_body<double>(g, link_field<L>{U}, Dq, F, scale, 0.0, vb);
}
// Half of the leaves: E(x) = [D(x) + U_mu(x-mu)^{-1} D(x-mu) U_mu(x-mu)] / 4,
// the leaves L1 and L2 of x.  L3 and L4 of x are the same of x - nu carried
// along U_nu(x-nu), so two passes of two products each do what one pass does in
// six (32^4: plaquettes and clover field 3.00 -> 2.60 ms a step, observables
// 3.43 -> 3.04 ms; the second pass is partly bound by its 0.9 GB of E).
__device__ __forceinline__ void fx_clover_half_body(Geo g, const int4* __restrict__ Ux, const int4* __restrict__ Ui,
                                                    const int4* __restrict__ Dq, int4* E, const unsigned* top, int4* sm, int vb) {
  const int p = vb % 6, mu = plane_mu(p);
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int x[4];
  site_coords(g, s, x);
  const int xmm = hop(g, s, x, mu, -1);
  fx_chk ck;
  mat<fx> acc, w, d;
  fx_pipe<2> P(sm);
  P.ask(Ui, mu, xmm, g.V);
  P.ask(Dq, p, xmm, g.V);
  const int shift = fx_field_shift(top);
  P.take(w, ck);
  P.ask(Ux, mu, xmm, g.V);
  P.take(d, ck);
  P.ask(Dq, p, s, g.V);
  if (shift) fx_shift_up(d, shift);
  fx_mul_left<FX_WIDE, 1, fx_acc_fine>(w, d, ck);
  P.take(d, ck);
  P.take(acc, ck);
  if (shift) fx_shift_up(acc, shift);
  fx_mul_acc<FX_WIDE, +1, 1, fx_acc_fine>(acc, w, d, ck);
  if (ck.bad()) acc.e[0].re.l = fx_raw_mark();  // its readers start over from D
  store<fx>(E, p, s, g.V, acc);
}
// F = +- [E(x) + U_nu(x-nu)^{-1} E(x-nu) U_nu(x-nu)] / 2.
template <typename L>
__device__ __forceinline__ void fx_clover_body(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                               const int4* __restrict__ Ui, const int4* __restrict__ Dq,
                                               const int4* __restrict__ E, int4* F, const unsigned* top, int4* sm, int vb) {
  const int p = vb % 6, nu = plane_nu(p);
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const bool neg = p == 1 || p == 4;
  int x[4];
  site_coords(g, s, x);
  const int xmn = hop(g, s, x, nu, -1);
  fx_chk ck;
  mat<fx> acc, w, d;
  fx_pipe<2> P(sm);
  P.ask(Ui, nu, xmn, g.V);
  P.ask(E, p, xmn, g.V);
  P.take(w, ck);
  P.ask(Ux, nu, xmn, g.V);
  P.take(d, ck);
  P.ask(E, p, s, g.V);
  fx_mul_left<FX_WIDE, 1, fx_acc_fine>(w, d, ck);
  P.take(d, ck);
  P.take(acc, ck);
  fx_mul_acc<FX_WIDE, +1, 1, fx_acc_fine>(acc, w, d, ck);
  if (neg) {
#pragma unroll
    for (int k = 0; k < 9; ++k) acc.e[k] = cx<fx>{-acc.e[k].re, -acc.e[k].im};
  }
  store<fx>(F, p, s, g.V, acc);
  const auto scale = [&] { return ldexp(neg ? -0.125 : 0.125, fx_field_shift(top)); };
  general_path(ck.bad(), s, g.V, [&](unsigned m, int t) { warp_clover<L>(m, g, U, tag_D(Dq), tag(F), scale(), p, t); },
               [&] { general_clover<L>(g, U, tag_D(Dq), tag(F), scale(), vb); });
}

// ------------------------------------------------------- plaquette drift
template <typename L>
static __device__ __noinline__ void general_force_wilson(Geo g, const typename vec2_of<L>::type* U, tagged Dq, tagged C, double b6, int vb) {
  k_plaq_force_wilson_body<double>(g, link_field<L>{U}, Dq, C, b6, vb);
}
template <typename L>
__device__ __forceinline__ void fx_force_wilson_body(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                                     const int4* __restrict__ Ui, const int4* __restrict__ Dq, int4* C,
                                                     double b6, int4* sm, int vb) {
  const int p = vb % 6, mu = plane_mu(p), nu = plane_nu(p);
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  fx_chk ck;
  unsigned mag = 0;
  const fx b = fx_of_double(2.0 * b6, mag);
  mat<fx> M, t, a;
  fx_pipe<2> P(sm);
  P.ask(Dq, p, s, g.V);
  P.ask(Ui, nu, s, g.V);
  P.take(a, ck);
  P.ask(Ux, nu, s, g.V);
  fx_scaled<FX_WIDE>(M, a, b, ck);
  store<fx>(C, 4 * p + 1, s, g.V, M);
  // slot 3: u^{-1} (beta/6 D) u
  P.take(t, ck);
  P.ask(Ui, mu, s, g.V);
  fx_mul_left<FX_WIDE>(t, M, ck);
  P.take(a, ck);
  P.ask(Ux, mu, s, g.V);
  fx_mul_left<FX_WIDE>(t, a, ck);
  store<fx>(C, 4 * p + 3, s, g.V, t);
  // slots 0 and 2: -(beta/6) D and the same carried by a
#pragma unroll
  for (int k = 0; k < 9; ++k) M.e[k] = cx<fx>{-M.e[k].re, -M.e[k].im};
  store<fx>(C, 4 * p + 0, s, g.V, M);
  P.take(t, ck);
  fx_mul_left<FX_WIDE>(t, M, ck);
  P.take(a, ck);
  fx_mul_left<FX_WIDE>(t, a, ck);
  store<fx>(C, 4 * p + 2, s, g.V, t);
  general_path(ck.bad() || !fx_mag_ok(mag), s, g.V,
               [&](unsigned m, int t) { warp_force_wilson<L>(m, g, U, tag_D(Dq), tag(C), b6, p, t); },
               [&] { general_force_wilson<L>(g, U, tag_D(Dq), tag(C), b6, vb); });
}

// The dual field of plaquette p's corner c3 carried to its base point,
// T_p(x) = u G3 u^{-1}, u = U_nu(x), into C plane 4p + 3 (which stage b writes
// last).  The corner c2 of the plaquette at x - mu is the same field carried
// along one more link, so this pass saves stage a the products a b, its inverse
// and (a b) G2 (a b)^{-1} for two: 20 products a plaquette in place of 21.7
// (theta force of a 32^4 step 6.55 -> 6.38 ms).
__device__ __forceinline__ void fx_force_t_body(Geo g, const int4* __restrict__ Ux, const int4* __restrict__ Ui,
                                                const int4* __restrict__ F, int4* C, int4* sm, int vb) {
  const int p = vb % 6, nu = plane_nu(p), pc = 5 - p;
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int x[4];
  site_coords(g, s, x);
  fx_chk ck;
  mat<fx> A, B;
  fx_pipe<2> P(sm);
  P.ask(Ux, nu, s, g.V);
  P.ask(F, pc, hop(g, s, x, nu, 1), g.V);
  P.take(A, ck);
  P.ask(Ui, nu, s, g.V);
  P.take(B, ck);
  fx_mul_left<FX_WIDE>(A, B, ck);
  P.take(B, ck);
  fx_mul_left<FX_WIDE>(A, B, ck);
  if (ck.bad()) A.e[0].re.l = fx_raw_mark();  // its readers start over from F
  store<fx>(C, 4 * p + 3, s, g.V, A);
}

// Stage a of the theta force: corners c0 .. c2.  A quarter of the dual fields'
// sum and the partials of slots 0 and 2 go to Gq and C (planes of this plaquette
// that only stage b of the same thread's plaquette writes).  Both stages keep
// at most three matrices in registers at a time, parking and re-reading the
// rest: with a fourth they would spill.  s: the scale -i theta kappa 2^-e, |s| <=
// 1/32; it multiplies D (and P), so the fields' errors are scaled down with it.
__device__ __forceinline__ void fx_force_a_body(Geo g, const int4* __restrict__ Ux, const int4* __restrict__ Ui,
                                                const int4* __restrict__ Dq, const int4* __restrict__ F, int4* Gq,
                                                int4* C, double b6, double sre, double sim, const unsigned* top, int4* sm, int vb) {
  const int p = vb % 6, mu = plane_mu(p), pc = 5 - p;
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int x[4];
  site_coords(g, s, x);
  const int c1 = hop(g, s, x, mu, 1);
  fx_chk ck;
  unsigned mag = 0;
  mat<fx> A, B, M;
  fx_pipe<2> P(sm);
  const fx_park K(sm + FX_PIPE);
  // corner c1: G1^ = a G1 a^{-1}
  P.ask(Ux, mu, s, g.V);
  P.ask(F, pc, c1, g.V);
  P.take(A, ck);
  P.ask(Ui, mu, s, g.V);
  P.take(B, ck);
  P.ask(Dq, p, s, g.V);
  fx_mul_left<FX_WIDE>(A, B, ck);
  P.take(B, ck);
  P.ask(F, pc, s, g.V);
  fx_mul_left<FX_WIDE>(A, B, ck);
  K.put(A);
  // slot 0 partial -(beta/6) D + [s D, G0], slot 2 partial the same + [s D, G1^]
  P.take(A, ck);
  P.ask(F, pc, s, g.V);
  fx_scaled<FX_WIDE>(M, A, fx_of_double(-2.0 * b6, mag), ck);
  fx_cscaled<FX_WIDE>(A, fx_cscale(sre, sim, 4 - fx_field_shift(top), mag), ck);  // 8 s D = 16 s (D / 2)
  P.take(B, ck);
  P.ask(Ux, mu, s, g.V);
  fx_commutator_acc<FX_WIDE>(M, A, B, ck);
  store<fx>(C, 4 * p + 0, s, g.V, M);
  K.get(B);
  fx_commutator_acc<FX_WIDE>(M, A, B, ck);
  store<fx>(C, 4 * p + 2, s, g.V, M);
  P.take(M, ck);
  P.ask(C, 4 * p + 3, c1, g.V);
  fx_quarter_sum(M, B);  // (G0 + G1^) / 4
  // corner c2: G2^ = a T(x+mu) a^{-1}
  P.take(A, ck);
  P.ask(Ui, mu, s, g.V);
  P.take(B, ck);
  fx_mul_left<FX_WIDE, 2>(A, B, ck);
  P.take(B, ck);
  fx_mul_acc<FX_WIDE, +1>(M, A, B, ck);
  if (ck.bad() || !fx_mag_ok(mag)) M.e[0].re.l = fx_raw_mark();  // stage b starts over
  store<fx>(Gq, GQ_PLANE * p, s, g.V, M);
}

template <typename L>
static __device__ __noinline__ void general_force(Geo g, const typename vec2_of<L>::type* U, tagged Pq, tagged Dq, tagged_c F, tagged C,
                                                  double b6, int vb) {
  k_plaq_force_ab_body<double>(g, link_field<L>{U}, Pq, Dq, F, C, b6, vb);
}
// Stage b: corner c3, K and the four slots.
template <typename L>
__device__ __forceinline__ void fx_force_b_body(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                                const int4* __restrict__ Ui, const int4* Pq, const int4* Dq,
                                                const int4* F, const int4* Gq, int4* C, double b6, double sre, double sim,
                                                const unsigned* top, int4* sm, int vb) {
  const int p = vb % 6, mu = plane_mu(p), nu = plane_nu(p);
  const int s = (vb / 6) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  fx_chk ck;
  unsigned mag = 0;
  const fx pb = fx_of_double(2.0 * b6, mag);
  const int shift = fx_field_shift(top);
  mat<fx> A, B, M;
  // corner c3: A = G3r = T; slot 3 partial = [s D, G3r] + (beta/6) D
  fx_pipe<2> P(sm);
  P.ask(Dq, p, s, g.V);
  P.ask(C, 4 * p + 3, s, g.V);
  P.take(B, ck);
  P.ask(Pq, p, s, g.V);
  fx_scaled<FX_WIDE>(M, B, pb, ck);
  fx_cscaled<FX_WIDE>(B, fx_cscale(sre, sim, 4 - shift, mag), ck);  // 8 s D
  P.take(A, ck);
  P.ask(Dq, p, s, g.V);
  fx_commutator_acc<FX_WIDE>(M, B, A, ck);
  store<fx>(C, 4 * p + 3, s, g.V, M);
  // M = G^ / 4 += P G3r P^{-1} / 4, with P^{-1} = P - 2 (D / 2)
  P.take(B, ck);
  P.ask(Pq, p, s, g.V);
  fx_mul_left<FX_WIDE, 2>(B, A, ck);
  P.take(A, ck);
  P.ask(Gq, GQ_PLANE * p, s, g.V);
  P.take(M, ck);
  P.ask(Pq, p, s, g.V);
#pragma unroll
  for (int k = 0; k < 9; ++k) A.e[k] = cx<fx>{M.e[k].re - fx_twice(A.e[k].re), M.e[k].im - fx_twice(A.e[k].im)};
  P.take(M, ck);
  P.ask(C, 4 * p + 0, s, g.V);
  fx_mul_acc<FX_WIDE, +1>(M, B, A, ck);
  // K = 32 s (P^{-1} G^ / 4 + G^ / 4 P), s taken with P^{-1} and P
  P.take(B, ck);
  P.ask(Dq, p, s, g.V);
  fx_cscaled<FX_WIDE>(A, fx_cscale(sre, sim, 5 - shift, mag), ck);
  fx_mul_left<FX_WIDE>(A, M, ck);
  fx_cscaled<FX_WIDE>(B, fx_cscale(sre, sim, 5 - shift, mag), ck);
  fx_mul_acc<FX_MID, +1>(A, M, B, ck);
  // slot 0: partial + K; slot 1: (beta/6) D - K
  P.take(M, ck);
  P.ask(Ui, nu, s, g.V);
  fx_add_to<+1>(M, A, ck);
  store<fx>(C, 4 * p + 0, s, g.V, M);
  P.take(M, ck);
  P.ask(Ux, nu, s, g.V);
  fx_scaled<FX_WIDE>(M, M, pb, ck);
  fx_add_to<-1>(M, A, ck);
  store<fx>(C, 4 * p + 1, s, g.V, M);
  // slot 3: u^{-1} (partial - K) u
  load_rw(M, C, 4 * p + 3, s, g.V);
  fx_add_to<-1>(M, A, ck);
  P.take(B, ck);
  P.ask(C, 4 * p + 2, s, g.V);
  fx_mul_left<FX_WIDE>(B, M, ck);
  P.take(M, ck);
  P.ask(Ui, mu, s, g.V);
  fx_mul_left<FX_WIDE>(B, M, ck);
  store<fx>(C, 4 * p + 3, s, g.V, B);
  // slot 2: a^{-1} (partial + K) a
  P.take(M, ck);
  P.ask(Ux, mu, s, g.V);
  fx_add_to<+1>(M, A, ck);
  P.take(A, ck);
  fx_mul_left<FX_WIDE>(A, M, ck);
  P.take(M, ck);
  fx_mul_left<FX_WIDE>(A, M, ck);
  store<fx>(C, 4 * p + 2, s, g.V, A);
  // anything out of range: the whole plaquette again (its slots are its own)
  general_path(ck.bad() || !fx_mag_ok(mag), s, g.V,
               [&](unsigned m, int t) { warp_force<L>(m, g, U, tag(Pq), tag_D(Dq), tag_F(F, shift, sre, sim), tag(C), b6, p, t); },
               [&] { general_force<L>(g, U, tag(Pq), tag_D(Dq), tag_F(F, shift, sre, sim), tag(C), b6, vb); });
}

// --------------------------------------------------------------- gather
// The drift matrix 2^e sum C of link (s, MU) as doubles.
static __device__ __noinline__ void general_gather(mat<double>& X, Geo g, int s, const int* x, int MU, tagged C, double ce) {
  mat<double> t;
  set_zero(X);
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == MU) continue;
    const int p = MU < nu ? plane_index(MU, nu) : plane_index(nu, MU);
    load(t, C, 4 * p + (MU < nu ? 0 : 1), s, g.V);
#pragma unroll
    for (int k = 0; k < 9; ++k) X.e[k] = cadd(X.e[k], t.e[k]);
    load(t, C, 4 * p + (MU < nu ? 3 : 2), hop(g, s, x, nu, -1), g.V);
#pragma unroll
    for (int k = 0; k < 9; ++k) X.e[k] = cadd(X.e[k], t.e[k]);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) X.e[k] = cx<double>{ce * X.e[k].re, ce * X.e[k].im};
}
// The sums as 60-bit integers.  Six contributions below 1.44 could just pass
// the 64-bit range at 8: the first four must stay below 5.
__device__ __forceinline__ bool fx_gather(long long* X, const Geo& g, int s, const int* x, int MU, const int4* __restrict__ C) {
  fx_chk ck;
  unsigned m = 0;
  mat<fx> t, l;
#pragma unroll
  for (int k = 0; k < 18; ++k) X[k] = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int nu = j + (j >= MU ? 1 : 0);
    const int p = MU < nu ? plane_index(MU, nu) : plane_index(nu, MU);
    fx_load(t, C, 4 * p + (MU < nu ? 0 : 1), s, g.V, ck);
    fx_load(l, C, 4 * p + (MU < nu ? 3 : 2), hop(g, s, x, nu, -1), g.V, ck);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      X[2 * k] += fx_bits(t.e[k].re) + fx_bits(l.e[k].re);
      X[2 * k + 1] += fx_bits(t.e[k].im) + fx_bits(l.e[k].im);
      if (j == 1)
        m = max(m, max((unsigned)(int)(X[2 * k] >> 32) + (5u << 28), (unsigned)(int)(X[2 * k + 1] >> 32) + (5u << 28)));
    }
  }
  return !ck.bad() && m < (10u << 28);
}
__device__ __forceinline__ void gather_f64(mat<double>& X, const Geo& g, int s, const int* x, int MU,
                                           const int4* C, int cexp) {
  long long v[18];
  if (fx_gather(v, g, s, x, MU, C)) {
#pragma unroll
    for (int k = 0; k < 9; ++k)
      X.e[k] = cx<double>{fx_bits_to_double(v[2 * k], cexp), fx_bits_to_double(v[2 * k + 1], cexp)};
  } else {
    mat<double> Xg;  // a local of its own: its address goes out of line
    general_gather(Xg, g, s, x, MU, tag(C), ldexp(1.0, cexp));
    X = Xg;
  }
}

// --------------------------------------------------------------- update
// (X - Tr X / 3) / 4 of the 60-bit integers X; false out of range.
__device__ __forceinline__ bool fx_traceless_quarter(mat<fx>& Q, const long long* X) {
  fx_chk ck;
  // of the quarters: three diagonals of up to 8 leave 64 bits
  const long long tr = ((X[0] >> 2) + (X[8] >> 2) + (X[16] >> 2)) / 3, ti = ((X[1] >> 2) + (X[9] >> 2) + (X[17] >> 2)) / 3;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const long long re = (X[2 * k] >> 2) - (k % 4 == 0 ? tr : 0), im = (X[2 * k + 1] >> 2) - (k % 4 == 0 ? ti : 0);
    ck.see<FX_WIDE>((int)(re >> 32));
    ck.see<FX_WIDE>((int)(im >> 32));
    Q.e[k] = cx<fx>{fx_of_bits(re), fx_of_bits(im)};
  }
  return !ck.bad();
}
// (The constant 8 eps 2^cexp is held to 2^-57 like every number: at small eps that is
// fewer bits of it than a double has, but times |Q| < 1.44 still below what A resolves.)
// A = 2 eps (X - Tr X / 3) + i sqrt(eps) sqrt(2) g_a lambda_a from the traceless
// quarter of X 2^-cexp and g / 8 (element j at gs[j TUNE_MAX_BLOCK]).  The noise constant 8 sqrt(2 eps) passes the fixed-point
// bound at eps = 0.016, the drift's 8 eps 2^cexp at eps = 0.0112 for beta = 24 .. 48
// (cexp = 4), half that for the next octave of beta: from the lower one on A is
// formed as a quarter.  (Out of range every link takes the FP64 path: 16^4 step 1.06
// ms against 0.72.)
__device__ __forceinline__ bool fx_exponent(mat<fx>& A /* in: the quarter */, const fx* gs, double eps, double sqrt_eps,
                                            int cexp) {
  fx_chk ck;
  unsigned mag = 0;
  const bool quarter = !(sqrt_eps < 0.12 && ldexp(8.0 * eps, cexp) < 1.4375);
  const double ks = sqrt_eps * (quarter ? 2.0 * 1.41421356237309504880 : 8.0 * 1.41421356237309504880);
  const double kd = ldexp(quarter ? 2.0 * eps : 8.0 * eps, cexp);  // times X / 4
  const fx kf = fx_of_double(ks, mag);
  const fx_left d = fx_lhs(fx_of_double(kd, mag)), n = fx_lhs(kf), m = fx_lhs_neg(kf),
                n3 = fx_lhs(fx_times(n, fx_rhs(fx_constant(NFX_RSQRT3_H, NFX_RSQRT3_L)))), m3 = {-n3.h, fx_neg(n3.p)};
  if (!fx_mag_ok(mag)) return false;
  fx_right R[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) R[j] = fx_rhs(gs[j * TUNE_MAX_BLOCK]);
#pragma unroll
  for (int k = 0; k < 9; ++k)
#pragma unroll
    for (int im = 0; im < 2; ++im) {
      fx_acc s = fx_zero();
      fx_mac(s, d, fx_rhs(im ? A.e[k].im : A.e[k].re));
      // i H: H01 = g0 - i g1, H02 = g3 - i g4, H12 = g5 - i g6, Hermitian;
      // H00 = g2 + g7 / sqrt 3, H11 = -g2 + g7 / sqrt 3, H22 = -2 g7 / sqrt 3
      const int i = k / 3, j = k % 3;
      if (i == j) {
        if (im) {
          if (i < 2) fx_mac(s, i == 0 ? n : m, R[2]);
          fx_mac(s, i < 2 ? n3 : m3, R[7]);
          if (i == 2) fx_mac(s, m3, R[7]);  // (2 g7 / 8 passes the range at g7 = 8; |g| goes up to 8.6)
        }
      } else {
        const int q = i + j == 1 ? 0 : i + j == 2 ? 3 : 5;
        if (im)
          fx_mac(s, n, R[q]);
        else
          fx_mac(s, i < j ? n : m, R[q + 1]);
      }
      const long long r = fx_sum(s) - (1 << 29);
      if (quarter)
        ck.see<FX_NARROW>((int)(r >> 32));
      else
        ck.see<FX_WIDE>((int)(r >> 32));
      const fx w = fx_of_bits(quarter ? r << 2 : r);
      if (im)
        A.e[k].im = w;
      else
        A.e[k].re = w;
    }
  return !ck.bad();
}

// The adaptive step's drift pass: the operand of the update (the traceless
// quarter of X 2^-cexp, or X itself as doubles) into out; returns |K|^2 =
// 2 |X - Tr X / 3|_F^2.
__device__ __forceinline__ double drift_fx(const Geo& g, const int4* C, int4* o, int cexp, int s, const int* x, int MU,
                                           bool write) {
  long long v[18];
  mat<fx> Q;
  if (fx_gather(v, g, s, x, MU, C) && fx_traceless_quarter(Q, v)) {
    fx_acc n = fx_zero();
    float nf = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      fx_mac(n, fx_lhs(Q.e[k].re), fx_rhs(Q.e[k].re));
      fx_mac(n, fx_lhs(Q.e[k].im), fx_rhs(Q.e[k].im));
      nf = fmaf((float)Q.e[k].re.h, (float)Q.e[k].re.h, fmaf((float)Q.e[k].im.h, (float)Q.e[k].im.h, nf));
    }
    if (write) store<fx>(o, MU, s, g.V, Q);
    write = false;  // the words an update from C would use: the same step bit for bit
    if (nf < 7.5f * 0x1p60f) return fx_bits_to_double(fx_sum(n) - (1 << 29), 2 * cexp + 5);
  }
  mat<double> Xd;
  gather_f64(Xd, g, s, x, MU, C, cexp);
  if (write) store(tagged{o, cexp + 2, 0u}, MU, s, g.V, Xd);  // doubles: words are the traceless quarter
  return general_k2(Xd);
}

// The general update's X from the contributions, as drift_fx would have stored it.
static __device__ __noinline__ void general_operand(mat<double>& X, const Geo g, int s, const int* x, int MU, const int4* C,
                                                    int cexp) {
  long long v[18];
  mat<fx> Q;
  if (fx_gather(v, g, s, x, MU, C) && fx_traceless_quarter(Q, v)) {
    const double sc = ldexp(1.0, cexp + 2);
#pragma unroll
    for (int k = 0; k < 9; ++k) X.e[k] = cx<double>{fx_to_double(Q.e[k].re) * sc, fx_to_double(Q.e[k].im) * sc};
  } else {
    gather_f64(X, g, s, x, MU, C, cexp);
  }
}

// An eighth of a link beyond the fixed-point range (exp(A) U is linear in it),
// and the end of its update.
template <typename L>
static __device__ __noinline__ bool fx_link_eighth(mat<fx>& u, const typename vec2_of<L>::type* U, int mu, int s, int V) {
  mat<double> d;
  load_link_d<L>(d, U, mu, s, V);
  unsigned mag = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k)
    u.e[k] = cx<fx>{fx_of_double(0.125 * d.e[k].re, mag), fx_of_double(0.125 * d.e[k].im, mag)};
  return fx_mag_ok(mag);
}
template <class V2>
static __device__ __noinline__ void update_far(V2* out, const mat<fx>& W, int mu, int s, int V) {
  mat<double> d;
#pragma unroll
  for (int k = 0; k < 9; ++k) d.e[k] = cx<double>{fx_to_double(W.e[k].re, 3), fx_to_double(W.e[k].im, 3)};
  const cx<double> z = det_inv_cuberoot(det(d));
#pragma unroll
  for (int k = 0; k < 9; ++k) d.e[k] = cmul(d.e[k], z);
  store_link(out, mu, s, V, d);
}

// The whole update in fixed point: exp(A) U with U the fixed-point word that
// the links pass left in `out`, times det^{-1/3} = 1 - e/3 for |e = det - 1| <
// 2^-31 (the drift of the determinant over a step is 1e-15; the next term is
// below 2^-62).  What does not fit goes through general_update_f64.
template <typename L>
__device__ __forceinline__ void update_fx(const Geo& g, const typename vec2_of<L>::type* U, const int4* C, const int4* X,
                                          typename vec2_of<L>::type* out, const UpdArgs& a, uint32_t step, int s, const int* x,
                                          int MU) {
  const double eps = a.adaptive ? a.sd->eps_n : a.eps;
  const double sqrt_eps = a.adaptive ? a.sd->sqrt_eps_n : a.sqrt_eps;
  const tagged Xt = {const_cast<int4*>(X), a.cexp + 2};
  // The noise first, one pair at a time into shared memory (a thread's own
  // words): its code once instead of four times, which the warps fetched (a
  // sixth of their time; update 0.145 -> 0.136 ms at 16^4, 1.80 -> 1.76 at 32^4).
  __shared__ fx noise[8 * TUNE_MAX_BLOCK];
  fx* gs = noise + threadIdx.x;
#pragma unroll 1
  for (int j = 0; j < 4; ++j) {
    fx g0, g1;
    normal_pair_fx(g0, g1, a.seed, step, (uint32_t)s, (uint32_t)MU, STREAM_CL, (uint32_t)j);
    gs[2 * j * TUNE_MAX_BLOCK] = g0;
    gs[(2 * j + 1) * TUNE_MAX_BLOCK] = g1;
  }
  mat<fx> A;
  bool ok;
  if (C) {
    long long v[18];
    ok = fx_gather(v, g, s, x, MU, C) && fx_traceless_quarter(A, v);
  } else {
    fx_chk ck;
    fx_load(A, Xt.p, MU, s, g.V, ck);
    ok = !ck.bad();
  }
  if (ok) {
    ok = fx_exponent(A, gs, eps, sqrt_eps, a.cexp);
    ok = ok && fx_expm_traceless(A, fx_norm(A), TAYLOR_TOL_FP64);
    if (ok) {
      fx_chk ck;
      mat<fx> u;
      fx_load_plain(u, reinterpret_cast<const int4*>(out), MU, s, g.V);
      const bool far = fx_is_raw(u.e[0].re.l);
      if (far && !fx_link_eighth<L>(u, U, MU, s, g.V)) ck.fail();
      fx_mul_left<FX_WIDE>(A, u, ck);
      if (far && !ck.bad()) {
        const mat<fx> W = A;  // a local of its own: its address goes out of line
        update_far(out, W, MU, s, g.V);
        return;
      }
      const cx<fx> e = fx_det_minus_one(A, ck);
      if (!ck.bad() && e.re.h == 0 && e.im.h == 0) {
        const float er = e.re.l * (-1.0f / 3.0f), ei = e.im.l * (-1.0f / 3.0f);  // units of 2^-60
        typename vec2_of<L>::type* p = out + (size_t)MU * 9 * g.V + s;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const float ur = (float)A.e[k].re.h * 0x1p-30f, ui = (float)A.e[k].im.h * 0x1p-30f;
          const fx re = {A.e[k].re.l + fmaf(er, ur, -ei * ui), A.e[k].re.h};
          const fx im = {A.e[k].im.l + fmaf(er, ui, ei * ur), A.e[k].im.h};
          p[(size_t)k * g.V] = fx_link_word(out, cx<fx>{re, im});
        }
        return;
      }
    }
  }
  mat<double> Xg, u, r;
  if (C)
    general_operand(Xg, g, s, x, MU, C, a.cexp);
  else
    load(Xg, Xt, MU, s, g.V);
  load_link_d<L>(u, U, MU, s, g.V);
  general_update_f64(r, Xg, u, a.seed, step, s, MU, eps, sqrt_eps);
  store_link(out, MU, s, g.V, r);
}

// The modes of k_update_gather_body (k_update.cuh).  C and (DRIFTMAX's out,
// UPDATE_X's C) the drift are fixed-point fields.
template <typename L, int MODE>
__device__ __forceinline__ void fx_update_body(Geo g, const typename vec2_of<L>::type* __restrict__ U,
                                               const int4* __restrict__ C, void* __restrict__ out, UpdArgs a, uint32_t step,
                                               int vb) {
  typedef typename vec2_of<L>::type V2;
  const int MU = vb % 4;
  const int s_raw = (vb / 4) * blockDim.x + threadIdx.x;
  if (MODE != MODE_DRIFTMAX && s_raw >= g.V) return;
  const int s = s_raw < g.V ? s_raw : g.V - 1;
  int x[4];
  site_coords(g, s, x);
  if (MODE == MODE_DRIFT) {
    mat<double> X;
    gather_f64(X, g, s, x, MU, C, a.cexp);
    store_link((V2*)out, MU, s, g.V, X);
  } else if (MODE == MODE_DRIFTMAX) {
    kmax_update(a.sd, drift_fx(g, C, (int4*)out, a.cexp, s, x, MU, s_raw < g.V));
  } else {
    update_fx<L>(g, U, MODE == MODE_UPDATE ? C : nullptr, MODE == MODE_UPDATE ? nullptr : C, (V2*)out, a, step, s, x, MU);
  }
}

}  // namespace clgc
