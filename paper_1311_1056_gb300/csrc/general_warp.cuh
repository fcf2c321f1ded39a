// general_warp.cuh -- the general path of one plaquette by a whole warp, in FP64:
// nine lanes hold one entry of each 3x3 matrix, products go through shuffles.
//
// Why: in chains with skirts a few links in ten thousand leave the fixed-point
// range.  One thread's plaquette in FP64 is a chain of thousands of instructions
// at 64 cycles (theta force ~190 us), which the whole launch then waits for; nine
// lanes together take a ninth of it.  Worth it while few of a warp's threads fail
// (WARP_GENERAL); beyond that each does its own.
#pragma once
#include "lattice.cuh"
#include "link_fx.cuh"

namespace clgc {

const int WARP_GENERAL = 8;

struct wmat {  // lane 3 i + j < 9: entry (i, j); the other lanes work on copies
  cx<double> v;
};
struct warp_ops {
  unsigned mask;  // the warp's threads inside the lattice (at least nine)
  int i, j, k;    // this lane's entry
  __device__ __forceinline__ explicit warp_ops(unsigned m) : mask(m) {
    k = (threadIdx.x & 31) % 9;
    i = k / 3;
    j = k - 3 * i;
  }
  __device__ __forceinline__ cx<double> get(const wmat& a, int q) const {
    return cx<double>{__shfl_sync(mask, a.v.re, q), __shfl_sync(mask, a.v.im, q)};
  }
  __device__ __forceinline__ wmat mul(const wmat& a, const wmat& b) const {
    cx<double> r = cmul(get(a, 3 * i), get(b, j));
    r = cfma(get(a, 3 * i + 1), get(b, 3 + j), r);
    return wmat{cfma(get(a, 3 * i + 2), get(b, 6 + j), r)};
  }
  __device__ __forceinline__ wmat adj(const wmat& a) const {
    const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
    const cx<double> p = get(a, 3 * j1 + i1), q = get(a, 3 * j2 + i2), s = get(a, 3 * j1 + i2), t = get(a, 3 * j2 + i1);
    return wmat{cfms(s, t, cmul(p, q))};
  }
  // a x b for b the inverse of a
  __device__ __forceinline__ wmat carry(const wmat& a, const wmat& x, const wmat& b) const { return mul(mul(a, x), b); }

  template <typename L>
  __device__ __forceinline__ wmat link(const typename vec2_of<L>::type* U, int mu, int s, int V) const {
    const cx<L> w = unpack(U[((size_t)mu * 9 + k) * V + s]);
    return wmat{cx<double>{real_d(w.re), real_d(w.im)}};
  }
  __device__ __forceinline__ wmat load(tagged f, int plane, int s, int V) const {
    const int4* p = f.p + (size_t)plane * 9 * V + s;
    const int4 v = p[(size_t)k * V];
    if (fx_is_raw(__int_as_float(p[0].x))) {
      cx<double> r = {__hiloint2double(v.y, v.x), __hiloint2double(v.w, v.z)};
      if (k == 0) r.re = fx_raw_first(make_int2(v.x, v.y));
      return wmat{cx<double>{fx_pow2(r.re, f.ex), fx_pow2(r.im, f.ex)}};
    }
    const cx<fx> w = unpack(v);
    return wmat{cx<double>{fx_to_double(w.re, f.ex), fx_to_double(w.im, f.ex)}};
  }
  __device__ __forceinline__ wmat load(tagged_c f, int plane, int s, int V) const { return wmat{cmul(load(f.f, plane, s, V).v, f.sc)}; }
  // In fixed point where it fits, as store(tagged).
  __device__ __forceinline__ void store(tagged f, int plane, int s, int V, const wmat& a) const {
    const double re = fx_pow2(a.v.re, -f.ex), im = fx_pow2(a.v.im, -f.ex);
    unsigned mag = 0;
    const cx<fx> w = {fx_of_double(re, mag), fx_of_double(im, mag)};
    const bool fits = __all_sync(mask, mag < f.lim);
    const int2 x = k == 0 ? fx_raw_first(re) : make_int2(__double2loint(re), __double2hiint(re));
    if ((threadIdx.x & 31) < 9)
      f.p[((size_t)plane * 9 + k) * V + s] = fits ? pack(w) : make_int4(x.x, x.y, __double2loint(im), __double2hiint(im));
  }
};
__device__ __forceinline__ wmat operator+(wmat a, wmat b) { return wmat{cadd(a.v, b.v)}; }
__device__ __forceinline__ wmat operator-(wmat a, wmat b) { return wmat{csub(a.v, b.v)}; }
__device__ __forceinline__ wmat operator*(double s, wmat a) { return wmat{cx<double>{s * a.v.re, s * a.v.im}}; }

// The formulas of k_update.cuh for plane p of site s.
template <typename L>
static __device__ __noinline__ void warp_plaq(unsigned mask, Geo g, const typename vec2_of<L>::type* U, tagged Pq, tagged Dq,
                                              int p, int s) {
  const warp_ops W(mask);
  const int mu = plane_mu(p), nu = plane_nu(p);
  int x[4];
  site_coords(g, s, x);
  const wmat A = W.mul(W.link<L>(U, mu, s, g.V), W.link<L>(U, nu, hop(g, s, x, mu, 1), g.V));
  const wmat B = W.mul(W.adj(W.link<L>(U, mu, hop(g, s, x, nu, 1), g.V)), W.adj(W.link<L>(U, nu, s, g.V)));
  const wmat P = W.mul(A, B), Pi = W.adj(P);
  // the force takes P^{-1} = P - D from the words: P as words only where P^{-1} fits as well
  const unsigned mag = max((unsigned)__double2hiint(Pi.v.re) & 0x7fffffffu, (unsigned)__double2hiint(Pi.v.im) & 0x7fffffffu);
  if (!__all_sync(mask, fx_mag_ok(mag))) Pq.lim = 0u;
  W.store(Pq, p, s, g.V, P);
  W.store(Dq, p, s, g.V, P - Pi);
}
template <typename L>
static __device__ __noinline__ void warp_clover(unsigned mask, Geo g, const typename vec2_of<L>::type* U, tagged Dq, tagged F,
                                                double scale, int p, int s) {
  const warp_ops W(mask);
  const int mu = plane_mu(p), nu = plane_nu(p);
  int x[4];
  site_coords(g, s, x);
  const int xmm = hop(g, s, x, mu, -1), xmn = hop(g, s, x, nu, -1);
  const int xmm_mn = hop2(g, s, x, mu, -1, nu, -1);
  wmat u = W.link<L>(U, mu, xmm, g.V);
  wmat acc = W.load(Dq, p, s, g.V) + W.carry(W.adj(u), W.load(Dq, p, xmm, g.V), u);
  u = W.link<L>(U, mu, xmm_mn, g.V);
  const wmat d = W.load(Dq, p, xmn, g.V) + W.carry(W.adj(u), W.load(Dq, p, xmm_mn, g.V), u);
  u = W.link<L>(U, nu, xmn, g.V);
  acc = acc + W.carry(W.adj(u), d, u);
  W.store(F, p, s, g.V, scale * acc);
}
template <typename L>
static __device__ __noinline__ void warp_force_wilson(unsigned mask, Geo g, const typename vec2_of<L>::type* U, tagged Dq,
                                                      tagged C, double b6, int p, int s) {
  const warp_ops W(mask);
  const wmat M = b6 * W.load(Dq, p, s, g.V), N = -1.0 * M;
  const wmat a = W.link<L>(U, plane_mu(p), s, g.V), u = W.link<L>(U, plane_nu(p), s, g.V);
  W.store(C, 4 * p + 0, s, g.V, N);
  W.store(C, 4 * p + 1, s, g.V, M);
  W.store(C, 4 * p + 2, s, g.V, W.carry(W.adj(a), N, a));
  W.store(C, 4 * p + 3, s, g.V, W.carry(W.adj(u), M, u));
}
template <typename L>
static __device__ __noinline__ void warp_force(unsigned mask, Geo g, const typename vec2_of<L>::type* U, tagged Pq, tagged Dq,
                                               tagged_c F, tagged C, double b6, int p, int s) {
  const warp_ops W(mask);
  const int mu = plane_mu(p), nu = plane_nu(p), pc = 5 - p;
  int x[4];
  site_coords(g, s, x);
  const int c1 = hop(g, s, x, mu, 1), c3 = hop(g, s, x, nu, 1);
  const wmat a = W.link<L>(U, mu, s, g.V), ai = W.adj(a), u = W.link<L>(U, nu, s, g.V), ui = W.adj(u);
  const wmat ab = W.mul(a, W.link<L>(U, nu, c1, g.V));
  const wmat D = W.load(Dq, p, s, g.V), P = W.load(Pq, p, s, g.V), Pi = P - D;
  const wmat G0 = W.load(F, pc, s, g.V), G1 = W.carry(a, W.load(F, pc, c1, g.V), ai);
  const wmat G2 = W.carry(ab, W.load(F, pc, hop(g, c1, x, nu, 1), g.V), W.adj(ab));
  const wmat G3 = W.carry(u, W.load(F, pc, c3, g.V), ui);
  const wmat G = G0 + G1 + G2 + W.carry(P, G3, Pi);
  const wmat K = W.mul(Pi, G) + W.mul(G, P), bD = b6 * D;
  const wmat s0 = (W.mul(D, G0) - W.mul(G0, D)) - bD, s2 = s0 + (W.mul(D, G1) - W.mul(G1, D));
  const wmat s3 = (W.mul(D, G3) - W.mul(G3, D)) + bD;
  W.store(C, 4 * p + 0, s, g.V, K + s0);
  W.store(C, 4 * p + 1, s, g.V, bD - K);
  W.store(C, 4 * p + 2, s, g.V, W.carry(ai, K + s2, a));
  W.store(C, 4 * p + 3, s, g.V, W.carry(ui, s3 - K, u));
}

// At the end of a kernel's body, by every thread with s < V: for each thread of
// the warp that failed, one(mask, its site) by the whole warp, or all(), each its
// own, where many did.
template <class One, class All>
__device__ __forceinline__ void general_path(bool bad, int s, int V, One one, All all) {
  const int s0 = s - (int)(threadIdx.x & 31), n = min(32, V - s0);
  const unsigned mask = n == 32 ? 0xffffffffu : (1u << n) - 1u;
  unsigned f = __ballot_sync(mask, bad);
  if (f == 0u) return;
  if (n >= 9 && __popc(f) <= WARP_GENERAL) {
    __syncwarp(mask);  // the failed thread's stores come before the ones that replace them
    for (; f; f &= f - 1u) one(mask, s0 + __ffs((int)f) - 1);
  } else if (bad) {
    all();
  }
}

}  // namespace clgc
