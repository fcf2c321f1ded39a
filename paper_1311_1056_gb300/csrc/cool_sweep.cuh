// cool_sweep.cuh -- the kernels of a cooling call, for link types double and
// df64 (sweeps in fixed point, cool_fx.cuh) and float (FP32 storage).
//
// Shape.  32 consecutive sites are a group; a block of 128 threads works on a
// group with one warp per direction mu.  In the gradient a thread takes the
// forward and the backward link of its direction and the four partial sums meet
// in shared memory; then one thread per site (gradient) or per site and sign
// (Omega) goes on.  In the apply a thread owns one link.  One thread per site
// all the way would be the same work in a chain four to eight times as long, and
// lattices below ~50,000 sites, a warp or two per scheduler, run at the length
// of that chain: gradient + Omega and apply 13 us each at 10x8x12x9, now ~8.
// Where the second half would leave most of the block idle and the lattice
// fills the GPU anyway, a block takes several groups before it (the wide shape); a
// site's numbers are the same either way.  FP32 storage, whose sums keep one
// order (sweep_add_f32), splits a site by the entries of G instead of by direction,
// and in the wide shape not at all.
//
// The rule (Sec. 4) needs sums over the lattice.  Every group (of large
// lattices: every few groups, cs_rounds) leaves one record; the block that
// finds, by a counter, that it is the last one sums the records in a fixed order
// and applies the rule.  No block waits.  (A launch of its own for the rule cost
// ~6 us a sweep.)  The records do not depend on how the groups are dealt to
// blocks, so a lone chain and a chain of a fused batch agree bit for bit.
#pragma once
#include <type_traits>

#include "cool_fx.cuh"
#include "cvt.cuh"
#include "link_fx.cuh"

namespace clgc {

const int CS_SITES = 32, CS_THREADS = 128, CS_NARROW_SITES = 24576;
__host__ __device__ inline int cs_groups(int V) { return (V + CS_SITES - 1) / CS_SITES; }
// Groups that a block of the wide shape takes at once.
template <typename L>
__host__ __device__ constexpr int cs_wide_grad() { return is_fx<L>() ? 2 : 4; }
template <typename L>
__host__ __device__ constexpr int cs_wide_omega() { return is_fx<L>() ? 3 : 4; }  // 3: what shared memory holds with the pipe
// Rounds of a block: the links of fixed-point forms keep at most ~2,048 records
// (which one block sums in ~3 us), one per warp; FP32 storage, whose kernels are
// short, at most 2,048 blocks of four groups a round (with the records' number
// for its blocks', 512 at 32^4: first gradient 0.134 against 0.091 ms).
template <typename L>
__host__ __device__ inline int cs_rounds(int V) {
  const int n = is_fx<L>() ? 2048 : 8192;
  return (cs_groups(V) + n - 1) / n;
}
// Blocks: gradient (width w: 1 or cs_wide_grad), gradient + Omega (width 1 or
// cs_wide_omega), apply (FP32 storage: width 1 or 4).
template <typename L>
__host__ __device__ inline int cs_grad_blocks(int V, int w) {
  const int n = w * cs_rounds<L>(V);
  return (cs_groups(V) + n - 1) / n;
}
__host__ __device__ inline int cs_grad_omega_blocks(int V, int w) { return (cs_groups(V) + w - 1) / w; }
template <typename L>
__host__ __device__ inline int cs_apply_blocks(int V, int w) { return cs_grad_blocks<L>(V, is_fx<L>() ? 1 : w); }
// Whether a lattice on its own runs the narrow shape.
inline bool cs_narrow(int V) { return V <= CS_NARROW_SITES; }

// What a sweep kernel works on.  U: the links; Ux: their fixed-point words
// (FP32 storage: U itself).
struct SweepArgs {
  const void* U;
  void* Ux;
  double* f;
  void *Om, *Omi;
  double2* rec;       // records of four doubles (sweep_grad_body)
  unsigned* ticket;   // blocks done, zero between launches
  CoolState* cs;
  CoolArgs ca;
};
// Number of sweeps that the host enqueues for a call.
__host__ __device__ inline int cs_sweeps(const CoolArgs& a) { return a.forced_sweeps >= 0 ? a.forced_sweeps : a.n_max; }

// One link from its fixed-point (or raw) words back to the link field.
template <class V2>
__device__ __forceinline__ void unload_link(V2* U, const int4* Ux, int mu, int s, int V) {
  mat<fx> u;
  fx_load_plain(u, Ux, mu, s, V);
  if (!fx_is_raw(u.e[0].re.l)) {
    fx_store_link(U, mu, s, V, u);
  } else {
    mat<double> d;
    load(d, tagged{const_cast<int4*>(Ux), 0}, mu, s, V);
    store_link(U, mu, s, V, d);
  }
}

// ------------------------------------------------------------------- rule
// The adaptive rule (Sec. 4): alpha_ad = alpha / D with D_0 = 1,
// D_1 = (1/3)<Tr U U^+> (normalised unitarity norm), D_2 = <|f_ax|>_{a,x}
// (or its RMS).  Sweep count: at least n_min, at most n_max; stop once the
// norm decreases by less than tol_rel of its distance from 1 or that distance
// is below d_floor; no sweep when D < d_guard; forced_sweeps >= 0 fixes the count.
// Both sides of the tol_rel test are differences of nearly equal norms, and chains
// do meet it within rounding: a count is reproducible for one build and form, and
// by one sweep sensitive to any change in the rounding of the links or of the sums.
// un: the norm; tot0, tot1: sum |f_ax|, sum f_ax^2; old: the state before.
// One thread runs this at the end of a kernel: the state comes in one read, and
// FP64 divisions (~0.5 us each) are left out where the divisor is known before.
__device__ __forceinline__ void cool_rule(double un, double tot0, double tot1, bool nonfinite, const CoolArgs& a,
                                          const CoolState& old, CoolState* cs, int first) {
  CoolState n = old;
  if (first) {
    n.alpha_ad = 0.0;
    n.alpha_ad_last = 0.0;
    n.un_prev = 0.0;
    n.sweeps = 0;
    n.done = 0;
    n.k = 0;
    n.nonfinite = 0;
  }
  if (n.done) return;
  double D = 1.0;
  if (a.mode == 1) D = un;
  if (a.mode == 2) D = tot0 * (0.5 * a.inv_links);
  if (a.mode == 3) D = sqrt(tot1 * (0.5 * a.inv_links));
  const int k = n.k;
  if (k == 0) n.un_before = un;
  n.un_after = un;
  n.D = D;
  bool stop;
  if (a.forced_sweeps >= 0) {
    stop = k >= a.forced_sweeps;
  } else {
    stop = k >= a.n_max;
    if (k >= a.n_min) {
      if (un - 1.0 < a.d_floor) stop = true;
      if (k >= 1 && (n.un_prev - un) < a.tol_rel * (n.un_prev - 1.0)) stop = true;
    }
  }
  if (D < a.d_guard) stop = true;
  if (nonfinite || !isfinite(un)) {
    n.nonfinite = 1;
    stop = true;
  }
  n.k = k + 1;
  if (stop) {
    n.done = 1;
  } else {
    n.alpha_ad = a.mode == 0 ? a.alpha : a.alpha / D;
    n.alpha_ad_last = n.alpha_ad;
    n.sweeps += 1;
    n.un_prev = un;
  }
  *cs = n;
}

struct SweepSums {
  double x = 0.0, y = 0.0, z = 0.0, w = 0.0;  // sum |f|, sum f^2, (1/3) sum Tr U U^+, nonfinite
};
__device__ __forceinline__ void sweep_record(const SweepArgs& a, int r, double x, double y, double z, double w) {
  __stcg(a.rec + 2 * r, make_double2(x, y));
  __stcg(a.rec + 2 * r + 1, make_double2(z, w));
}
// Norm accumulators of the single-pass sweeps' applies: integers, so the sum
// does not depend on the order of the blocks and needs no records.  They sit
// behind the records; the first gradient's last block zeroes them, every later
// rule takes and zeroes them.
struct SweepNorm {
  unsigned long long hi, lo;  // sum over blocks of acc >> 20 and of its low 20 bits
  double far;                 // FP32 storage: sites beyond the integers' range
  unsigned wild, pad;         // fixed point: blocks with links out of range
};
__device__ __forceinline__ SweepNorm* sweep_norm(const SweepArgs& a, int V) {
  return reinterpret_cast<SweepNorm*>(a.rec + 2 * (cs_groups(V) + 4));
}
// Whether this block is the last of nb.  Thread 0's writes before are visible
// to the last block; writes of other threads need a fence and a barrier before.
__device__ __forceinline__ bool sweep_last(const SweepArgs& a, int nb) {
  __shared__ unsigned last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(a.ticket, 1u) == (unsigned)(nb - 1);
    __threadfence();
  }
  __syncthreads();
  return last != 0;
}
// After the block's records: in the last of nb blocks sums the nrec records and
// applies the rule.  with_f: D_2 rules, which need sum |f| and sum f^2.
__device__ __forceinline__ void sweep_rule(const Geo& g, const SweepArgs& a, bool with_f, int nb, int nrec, int first) {
  __shared__ double part[CS_THREADS / 32][4];
  if (!sweep_last(a, nb)) return;
  CoolState old;
  if (threadIdx.x == 0) old = *a.cs;
  SweepSums t;
#pragma unroll 8
  for (int b = threadIdx.x; b < nrec; b += CS_THREADS) {
    if (with_f) {
      const double2 r = __ldcg(a.rec + 2 * b);
      t.x += r.x;
      t.y += r.y;
    }
    const double2 r = __ldcg(a.rec + 2 * b + 1);
    t.z += r.x;
    t.w += r.y;
  }
  const bool bad = t.w != 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (with_f) {
      t.x += __shfl_down_sync(0xffffffffu, t.x, o);
      t.y += __shfl_down_sync(0xffffffffu, t.y, o);
    }
    t.z += __shfl_down_sync(0xffffffffu, t.z, o);
  }
  if ((threadIdx.x & 31) == 0) {
    part[threadIdx.x >> 5][0] = t.x;
    part[threadIdx.x >> 5][1] = t.y;
    part[threadIdx.x >> 5][2] = t.z;
  }
  const bool nonfinite = __syncthreads_or(bad) != 0;
  if (threadIdx.x != 0) return;
  double tot[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) tot[q] = (part[0][q] + part[1][q]) + (part[2][q] + part[3][q]);
  cool_rule(tot[2] * a.ca.inv_links, tot[0], tot[1], nonfinite, a.ca, old, a.cs, first);
  if (first) *sweep_norm(a, g.V) = SweepNorm{0ull, 0ull, 0.0, 0u, 0u};
  *a.ticket = 0u;
}

// --------------------------------------------------------------- gradient
// The gradient between its two halves, in shared memory.  Fixed point: partial
// sums of one direction, 60-bit integers.  FP32 storage: a site's sums, floats.
template <typename L>
struct sweep_real { typedef typename std::conditional<is_fx<L>(), long long, float>::type type; };
// N: 9 numbers, g00, g11, g22, then re / im of g01, g02, g12; 12 with the norm
// (the three diagonals of the forward links).
template <typename L, int N>
struct SweepPart {
  static const int WIDTH = is_fx<L>() ? CS_THREADS : CS_SITES;
  typename sweep_real<L>::type q[N][WIDTH];
  // fixed point: largest row or column norm (squared); negative: of a direction whose
  // sums are in sixteenths; infinite: not representable
  float top[is_fx<L>() ? CS_THREADS : 1];
};

// FP32 storage.  The rule compares differences of norms, themselves sums of
// rounded floats, with a threshold that chains often meet within rounding, so
// a site's numbers are summed in one order in every shape: the forward links
// mu = 0 .. 3, then the backward ones.  (Summed direction by direction the same
// chains stopped a sweep earlier or later now and then.)
// One column k of a link's rows (or conjugated columns) a, b, c: d += |c|^2, o += a conj(b).
__device__ __forceinline__ void sweep_add_f32(float& d, cx<float>& o, cx<float> a, cx<float> b, cx<float> c) {
  d = fmaf(c.re, c.re, fmaf(c.im, c.im, d));
  o = cfma(a, cx<float>{b.re, -b.im}, o);
}
__device__ __forceinline__ void sweep_sub_f32(float& d, cx<float>& o, cx<float> a, cx<float> b, cx<float> c) {
  d = fmaf(-c.re, c.re, fmaf(-c.im, c.im, d));
  o = cfms(cx<float>{a.re, -a.im}, b, o);
}
// Rows of pair p: g01 with g00, g12 with g11, g02 with g22.
__host__ __device__ constexpr int pair_a(int p) { return p == 1 ? 1 : 0; }
__host__ __device__ constexpr int pair_b(int p) { return p == 0 ? 1 : 2; }
__host__ __device__ constexpr int pair_off(int p) { return p == 0 ? 3 : p == 1 ? 7 : 5; }  // its slot among the nine numbers
// Pair P of a site, for the narrow shape, a warp a pair (9 chains of 48 dependent
// multiply-adds, a third of them a warp's).  fwd: the diagonal after the forward links.
template <int P>
__device__ __forceinline__ void sweep_pair_f32(float& d, float& fwd, cx<float>& o, const Geo& g, const float2* __restrict__ U, int s) {
  constexpr int A = pair_a(P), B = pair_b(P);
  int x[4];
  site_coords(g, s, x);
  d = 0.0f;
  o = cx<float>{0.0f, 0.0f};
#pragma unroll
  for (int dir = 0; dir < 8; ++dir) {
    const int mu = dir & 3;
    const float2* p = U + (size_t)mu * 9 * g.V + (dir < 4 ? s : hop(g, s, x, mu, -1));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cx<float> a = unpack(__ldg(p + (size_t)(dir < 4 ? 3 * A + k : 3 * k + A) * g.V));
      const cx<float> b = unpack(__ldg(p + (size_t)(dir < 4 ? 3 * B + k : 3 * k + B) * g.V));
      if (dir < 4)
        sweep_add_f32(d, o, a, b, P == 2 ? b : a);
      else
        sweep_sub_f32(d, o, a, b, P == 2 ? b : a);
    }
    if (dir == 3) fwd = d;
  }
}
// The wide shape's site: all of it by one thread; q[9] the norm.
__device__ __forceinline__ void sweep_sums_f32(float* q, const Geo& g, const float2* __restrict__ U, int s) {
  int x[4];
  site_coords(g, s, x);
  float d[3] = {0.0f, 0.0f, 0.0f};
  cx<float> o[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
  mat<float> u;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    load(u, U, mu, s, g.V);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int p = 0; p < 3; ++p)
        sweep_add_f32(d[p], o[p], u.e[3 * pair_a(p) + k], u.e[3 * pair_b(p) + k], u.e[3 * p + k]);
  }
  q[9] = d[0] + d[1] + d[2];
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    load(u, U, mu, hop(g, s, x, mu, -1), g.V);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int p = 0; p < 3; ++p)
        sweep_sub_f32(d[p], o[p], u.e[3 * k + pair_a(p)], u.e[3 * k + pair_b(p)], u.e[3 * k + p]);
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    q[p] = d[p];
    q[pair_off(p)] = o[p].re;
    q[pair_off(p) + 1] = o[p].im;
  }
}

// Entries beyond the fixed-point bound, up to 2^K times it (chains whose links
// have skirts keep a few such): the link times 2^-K, from its words or doubles.
template <int K>
__device__ __forceinline__ bool fx_load_wild(mat<fx>& u, const int4* Ux, int mu, int s, int V) {
  fx_load_plain(u, Ux, mu, s, V);
  unsigned mag = 0;
  if (fx_is_raw(u.e[0].re.l)) {
    mat<double> d;
    load(d, tagged{const_cast<int4*>(Ux), 0}, mu, s, V);
#pragma unroll
    for (int k = 0; k < 9; ++k)
      u.e[k] = cx<fx>{fx_of_double(fx_pow2(d.e[k].re, -K), mag), fx_of_double(fx_pow2(d.e[k].im, -K), mag)};
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) u.e[k] = cx<fx>{fx_of_bits(fx_bits(u.e[k].re) >> K), fx_of_bits(fx_bits(u.e[k].im) >> K)};
  }
  return fx_mag_ok(mag);
}
// A thread's part of the gradient where a link of it is beyond the bound or a sum
// beyond 8: both links times 1/4, the sums in sixteenths.  (In FP64 the site's eight
// links are one thread's chain of ~600 instructions: 20 us a sweep for the whole
// launch, and at a unitarity norm of 1.2 all sites': 24^4, five sweeps, 10.0 ms
// against 4.4.)
template <typename L, bool FIRST>
static __device__ __noinline__ void sweep_part_wild(long long* q, int n, float* top, const void* U, const int4* Ux, int mu, int s, int sb,
                                                    int V) {
  const auto get = [&](mat<fx>& u, int site) {
    if constexpr (FIRST) {  // the neighbour's words may not be there yet
      mat<double> d;
      load_link_d<L>(d, (const typename vec2_of<L>::type*)U, mu, site, V);
      unsigned mag = 0;
#pragma unroll
      for (int k = 0; k < 9; ++k) u.e[k] = cx<fx>{fx_of_double(fx_pow2(d.e[k].re, -2), mag), fx_of_double(fx_pow2(d.e[k].im, -2), mag)};
      return fx_mag_ok(mag);
    } else {
      return fx_load_wild<2>(u, Ux, mu, site, V);
    }
  };
  fx_acc D[3], O[6];
  float nf[3] = {0.0f, 0.0f, 0.0f}, nb[3] = {0.0f, 0.0f, 0.0f}, m = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) D[i] = fx_zero();
#pragma unroll
  for (int i = 0; i < 6; ++i) O[i] = fx_zero();
  mat<fx> u;
  *top = __int_as_float(0x7f800000);
  if (!get(u, s)) return;
#pragma unroll
  for (int k = 0; k < 3; ++k) fx_outer(D, O, nf, u.e[k], u.e[3 + k], u.e[6 + k], false);
  if (n > 9)
#pragma unroll
    for (int i = 0; i < 3; ++i) q[(9 + i) * CS_THREADS] = fx_sum<true>(D[i]) - (1 << 29);
  if (!get(u, sb)) return;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cx<fx> a = u.e[3 * k], b = u.e[3 * k + 1], c = u.e[3 * k + 2];
    fx_outer(D, O, nb, cx<fx>{a.re, -a.im}, cx<fx>{b.re, -b.im}, cx<fx>{c.re, -c.im}, true);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q[i * CS_THREADS] = fx_sum<true>(D[i]) - (1 << 29);
    m = fmaxf(m, fmaxf(nf[i], nb[i]));
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) q[(3 + i) * CS_THREADS] = fx_sum<true>(O[i]) - (1 << 29);
  if (m < 7.6f * 0x1p60f) *top = -16.0f * 0x1p-60f * m;
}

// First half: this thread's direction (fixed point) or pair (FP32 storage), a warp
// each, and site.  FIRST: the links are read from U and (fixed point) their words
// written to Ux.
// PIPE: the links come through a pipe, the forward one asked for by
// the call for the group before (next; the first group's by the caller), so that each
// link's load runs under the outer products of the one before (gradient + Omega
// of a 32^4 step of ten sweeps 2.53 -> 2.37 ms).
__device__ __forceinline__ void sweep_ask(fx_pipe<1>& P, const Geo& g, const SweepArgs& a, int group) {
  const int mu = threadIdx.x >> 5, s = group * CS_SITES + (threadIdx.x & 31);
  if (s < g.V) P.ask((const int4*)a.Ux, mu, s, g.V);
}
template <typename L, bool FIRST, bool PIPE, int N>
__device__ __forceinline__ void sweep_part(SweepPart<L, N>& sm, const Geo& g, const SweepArgs& a, int group, fx_pipe<1>& P,
                                           int next) {
  typedef typename vec2_of<L>::type V2;
  const int mu = threadIdx.x >> 5, s = group * CS_SITES + (threadIdx.x & 31), t = threadIdx.x;
  if (s >= g.V) return;
  if constexpr (is_fx<L>()) {
    int x[4];
    site_coords(g, s, x);
    const int sb = hop(g, s, x, mu, -1);
    const V2* U = (const V2*)a.U;
    int4* Ux = (int4*)a.Ux;
    fx_acc D[3], O[6];
    float nf[3] = {0.0f, 0.0f, 0.0f}, nb[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < 3; ++i) D[i] = fx_zero();
#pragma unroll
    for (int i = 0; i < 6; ++i) O[i] = fx_zero();
    mat<fx> u;
    fx_chk ck;
    bool ok = true;
    if constexpr (FIRST) {
      ok = fx_load_link<L>(u, U, mu, s, g.V);
      if (ok) {
        store<fx>(Ux, mu, s, g.V, u);
      } else {
        mat<double> d;
        load_link_d<L>(d, U, mu, s, g.V);
        store(tagged{Ux, 0}, mu, s, g.V, d);
      }
    } else if constexpr (PIPE) {
      P.take(u, ck);
      P.ask(Ux, mu, sb, g.V);
    } else {
      fx_load(u, Ux, mu, s, g.V, ck);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) fx_outer(D, O, nf, u.e[k], u.e[3 + k], u.e[6 + k], false);
    if constexpr (N > 9) {
#pragma unroll
      for (int i = 0; i < 3; ++i) sm.q[9 + i][t] = fx_sum<true>(D[i]) - (1 << 29);
    }
    if constexpr (FIRST) {
      const bool b = fx_load_link<L>(u, U, mu, sb, g.V);
      ok = ok && b;
    } else if constexpr (PIPE) {
      P.take(u, ck);
      if (next >= 0) sweep_ask(P, g, a, next);
    } else {
      fx_load(u, Ux, mu, sb, g.V, ck);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cx<fx> p = u.e[3 * k], q = u.e[3 * k + 1], r = u.e[3 * k + 2];
      fx_outer(D, O, nb, cx<fx>{p.re, -p.im}, cx<fx>{q.re, -q.im}, cx<fx>{r.re, -r.im}, true);
    }
    float top = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      sm.q[i][t] = fx_sum<true>(D[i]) - (1 << 29);
      top = fmaxf(top, fmaxf(nf[i], nb[i]));
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) sm.q[3 + i][t] = fx_sum<true>(O[i]) - (1 << 29);
    top *= 0x1p-60f;
    sm.top[t] = ok && !ck.bad() && top < 7.6f ? top : __int_as_float(0x7f800000);
    if (!ok || ck.bad() || !(top < 7.6f)) sweep_part_wild<L, FIRST>(&sm.q[0][t], N, &sm.top[t], a.U, Ux, mu, s, sb, g.V);
  } else if (mu < 3) {
    float d, fwd;
    cx<float> o;
    if (mu == 0) sweep_pair_f32<0>(d, fwd, o, g, (const V2*)a.U, s);
    if (mu == 1) sweep_pair_f32<1>(d, fwd, o, g, (const V2*)a.U, s);
    if (mu == 2) sweep_pair_f32<2>(d, fwd, o, g, (const V2*)a.U, s);
    const int l = t & 31;
    sm.q[mu][l] = d;
    sm.q[pair_off(mu)][l] = o.re;
    sm.q[pair_off(mu) + 1][l] = o.im;
    if constexpr (N > 9) sm.q[9 + mu][l] = fwd;
  }
}
// Second half (after a barrier), one thread per site: the sums over directions.
template <typename L, int N>
__device__ __forceinline__ typename sweep_real<L>::type sweep_sum(const SweepPart<L, N>& sm, int q) {
  const int l = threadIdx.x & 31;
  return ((sm.q[q][l] + sm.q[q][32 + l]) + sm.q[q][64 + l]) + sm.q[q][96 + l];
}
// The sum of number q times 2^-n, for sites with directions in sixteenths.
template <typename L, int N>
static __device__ __noinline__ long long sweep_sum_wild(const SweepPart<L, N>& sm, int q, int n) {
  long long v = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const int l = (threadIdx.x & 31) + 32 * mu, k = sm.top[l] < 0.0f ? n - 4 : n;
    v += k >= 0 ? sm.q[q][l] >> k : sm.q[q][l] << -k;
  }
  return v;
}
// The sum of the norms' diagonals, Tr U U^+ over the four forward links, likewise.
template <typename L, int N>
static __device__ __noinline__ double sweep_norm_wild(const SweepPart<L, N>& sm, int n) {
  double un = 0.0;
  for (int i = 0; i < 3; ++i) un += fx_bits_to_double(sweep_sum_wild(sm, 9 + i, n), n);
  return un;
}
template <typename L, int N>
__device__ __forceinline__ bool sweep_gradient(fx_gradient& G, const SweepPart<L, N>& sm) {
  const int l = threadIdx.x & 31;
  // the sums over the four directions must stay below 8
  const float t0 = sm.top[l], t1 = sm.top[32 + l], t2 = sm.top[64 + l], t3 = sm.top[96 + l];
  const bool tame = fminf(fminf(t0, t1), fminf(t2, t3)) >= 0.0f && ((t0 + t1) + t2) + t3 < 7.6f;
#pragma unroll
  for (int i = 0; i < 3; ++i) G.d[i] = sweep_sum(sm, i);
#pragma unroll
  for (int i = 0; i < 6; ++i) G.o[i] = sweep_sum(sm, 3 + i);
  // |G| below 1, as everything formed from it expects: an eighth of it if need be
  bool one = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) one = one && fx_below_one(G.d[k]) && fx_below_one(G.o[2 * k]) && fx_below_one(G.o[2 * k + 1]);
  G.e = one ? 0 : 3;
  G.wild = 0;
  if (!one) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      G.d[k] >>= 3;
      G.o[2 * k] >>= 3;
      G.o[2 * k + 1] >>= 3;
    }
  }
  if (!tame) {
    const float top = ((fabsf(t0) + fabsf(t1)) + fabsf(t2)) + fabsf(t3);
    if (!(top < 1024.0f)) return false;
    const int n = max(1, ((__float_as_int(top) >> 23) & 0xff) - 126);  // top 2^-n in [1/2, 1)
#pragma unroll
    for (int i = 0; i < 3; ++i) G.d[i] = sweep_sum_wild(sm, i, n);
#pragma unroll
    for (int i = 0; i < 6; ++i) G.o[i] = sweep_sum_wild(sm, 3 + i, n);
    G.e = G.wild = n;
  }
  return true;
}
__device__ __forceinline__ void sweep_f(float* fa, const float* q) {
  fa[0] = 4.0f * q[3];
  fa[1] = -(4.0f * q[4]);
  fa[2] = 2.0f * (q[0] - q[1]);
  fa[3] = 4.0f * q[5];
  fa[4] = -(4.0f * q[6]);
  fa[5] = 4.0f * q[7];
  fa[6] = -(4.0f * q[8]);
  fa[7] = 2.0f * 0.57735026918962576451f * (q[0] + q[1] - 2.0f * q[2]);
}

// f_ax = 2 Tr[lambda_a G_x] of one site in FP64 (the general path); returns
// the sum over the four links at x of Tr U U^+.
template <class FU>
__device__ __forceinline__ double cool_grad_site(const Geo& g, FU U, int s, double* fa) {
  int x[4];
  site_coords(g, s, x);
  double d[3] = {0.0, 0.0, 0.0}, un = 0.0;
  cx<double> o[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 1
  for (int dir = 0; dir < 8; ++dir) {
    const int mu = dir & 3;
    mat<double> u, w;
    load(u, U, mu, dir < 4 ? s : hop(g, s, x, mu, -1), g.V);
    const double sg = dir < 4 ? 1.0 : -1.0;
    if (dir == 4) un = d[0] + d[1] + d[2];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k)  // rows of U, or conjugated columns
        w.e[3 * i + k] = dir < 4 ? u.e[3 * i + k] : cx<double>{u.e[3 * k + i].re, -u.e[3 * k + i].im};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cx<double> r[3] = {w.e[k], w.e[3 + k], w.e[6 + k]};
#pragma unroll
      for (int i = 0; i < 3; ++i) d[i] = fma(sg * r[i].re, r[i].re, fma(sg * r[i].im, r[i].im, d[i]));
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int i = q < 2 ? 0 : 1, j = q == 0 ? 1 : 2;
        o[q] = cfma(cx<double>{sg * r[i].re, sg * r[i].im}, cx<double>{r[j].re, -r[j].im}, o[q]);
      }
    }
  }
  fa[0] = 4.0 * o[0].re;
  fa[1] = -(4.0 * o[0].im);
  fa[2] = 2.0 * (d[0] - d[1]);
  fa[3] = 4.0 * o[1].re;
  fa[4] = -(4.0 * o[1].im);
  fa[5] = 4.0 * o[2].re;
  fa[6] = -(4.0 * o[2].im);
  fa[7] = 2.0 * 0.57735026918962576451 * (d[0] + d[1] - 2.0 * d[2]);
  return un;
}
template <typename L, bool FIRST>
static __device__ __noinline__ double general_cool_grad(const Geo g, const void* U, void* Ux, int s, double* fa) {
  if constexpr (FIRST) return cool_grad_site(g, link_field<L>{(const typename vec2_of<L>::type*)U}, s, fa);
  return cool_grad_site(g, tagged{(int4*)Ux, 0}, s, fa);
}

// The gradient f into [a][V] (FP64), and the rule.  FIRST: the call's first
// gradient, which always runs.  rule = false: f alone (a diagnostic).
template <typename L, bool FIRST>
__device__ __forceinline__ void sweep_grad_site(SweepSums& v, const SweepPart<L, 12>& sm, const float* q, const Geo& g,
                                                const SweepArgs& a, int s, bool with_f) {
  {
    double fa[8];
    if constexpr (is_fx<L>()) {
      fx_gradient G;
      double un;
      if (sweep_gradient(G, sm)) {
        long long o = 0;
        fx_acc sq = fx_zero();  // sum (f / 4)^2: six below 1, and the diagonal's two, which are
                                // (sum d^2 - (sum d)^2 / 3) / 2 < 4 / 3 together: below 8
        fx_chk ck;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          o += G.o[k] < 0 ? -G.o[k] : G.o[k];
          const fx w = fx_of_bits(G.o[k]);
          fx_mac(sq, fx_lhs(w), fx_rhs(w));
          const double d = fx_bits_to_double(G.o[k], 2 + G.e);
          fa[k < 2 ? k : k + 1] = (k & 1) ? -d : d;
        }
        const long long d01 = G.d[0] - G.d[1], d2 = G.d[0] + G.d[1] - 2 * G.d[2];
        fa[2] = fx_bits_to_double(d01, 1 + G.e);
        fa[7] = fx_bits_to_double(d2, 1 + G.e) * 0.57735026918962576451;
        if (with_f) {
          v.x += fx_bits_to_double(o, 2 + G.e) + (fabs(fa[2]) + fabs(fa[7]));
          // (f_2 / 4)^2 + (f_7 / 4)^2 with f_2 / 4 = d01 / 2, f_7 / 4 = d2 / (2 sqrt 3)
          const fx w2 = fx_of_bits(d01 >> 1);
          unsigned mag = 0;
          const fx c7 = fx_of_double(0.28867513459481288225, mag);
          fx_acc z = fx_zero();
          fx_mac(z, fx_lhs(c7), fx_rhs(fx_of_bits(d2 >> 2)));
          const fx w7 = fx_twice(fx_twice(fx_get<FX_WIDE>(z, ck)));
          fx_mac(sq, fx_lhs(w2), fx_rhs(w2));
          fx_mac(sq, fx_lhs(w7), fx_rhs(w7));
          v.y += fx_bits_to_double(fx_sum(sq) - (1 << 29), 4 + 2 * G.e);
        }
        // the unitarity norm; later gradients of D_2 calls need it too
        long long dev = 0;  // of the three diagonals from 4, 2^-58
#pragma unroll
        for (int i = 0; i < 3; ++i) dev += (sweep_sum(sm, 9 + i) - (4ll << 60)) >> 2;
        un = G.wild ? sweep_norm_wild(sm, G.wild) : 12.0 + fx_bits_to_double(dev, 2);
      } else {
        double fg[8];
        un = general_cool_grad<L, FIRST>(g, a.U, a.Ux, s, fg);
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          fa[k] = fg[k];
          t += fabs(fg[k]);
          v.y = fma(fg[k], fg[k], v.y);
        }
        v.x += t;
        v.w += isfinite(un) && isfinite(t) ? 0.0 : 1.0;
      }
      v.z += un * (1.0 / 3.0);
    } else {
      float ff[8];
      sweep_f(ff, q);
      const float un = q[9];
      bool ok = isfinite(un);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        fa[k] = cvt<double>(ff[k]);
        ok = ok && isfinite(ff[k]);
        if (with_f) {
          v.x += fabs(fa[k]);
          v.y = fma(fa[k], fa[k], v.y);
        }
      }
      v.z += cvt<double>(un) * (1.0 / 3.0);
      v.w += ok ? 0.0 : 1.0;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) a.f[(size_t)k * g.V + s] = fa[k];
  }
}
// W: groups at once.  Record W vb + w of a block is that of its warp w: the
// groups W (R vb + j) + w, j < R = cs_rounds.  FP32 storage beyond 2,048 groups:
// record vb, the block's.
template <typename L, bool FIRST, int W>
__device__ __forceinline__ void sweep_grad_body(const Geo& g, const SweepArgs& a, int vb, bool rule) {
  if (!FIRST && a.cs->done) return;
  // FP32 storage in the wide shape: a thread forms its site's sums itself
  constexpr bool ALONE = !is_fx<L>() && W > 1;
  __shared__ SweepPart<L, 12> sm[ALONE ? 1 : W];
  SweepSums v;
  const bool with_f = a.ca.mode >= 2;
  const int ng = cs_groups(g.V), R = cs_rounds<L>(g.V), w = threadIdx.x >> 5;
  constexpr bool PIPE = is_fx<L>() && !FIRST && W > 1;
  __shared__ int4 slot[PIPE ? fx_pipe<1>::WORDS : 1];
  fx_pipe<1> P(slot);
  if (PIPE) sweep_ask(P, g, a, W * R * vb);
  for (int j = 0; j < R; ++j) {
    const int g0 = W * (R * vb + j);
    const int s = (g0 + w) * CS_SITES + ((int)threadIdx.x & 31);
    float q[10];
    if constexpr (ALONE) {
      if (s < g.V) sweep_sums_f32(q, g, (const float2*)a.U, s);
    } else {
      if (j > 0) __syncthreads();
#pragma unroll 1
      for (int p = 0; p < W; ++p) sweep_part<L, FIRST, PIPE, 12>(sm[p], g, a, g0 + p, P, p + 1 < W || j + 1 < R ? g0 + p + 1 : -1);
      __syncthreads();
      if constexpr (!is_fx<L>())
        if (w < W && s < g.V) {
          const int l = threadIdx.x & 31;
#pragma unroll
          for (int i = 0; i < 9; ++i) q[i] = sm[w].q[i][l];
          q[9] = (sm[w].q[9][l] + sm[w].q[10][l]) + sm[w].q[11][l];
        }
    }
    if (w < W && s < g.V) sweep_grad_site<L, FIRST>(v, sm[ALONE ? 0 : w], q, g, a, s, with_f);
  }
  if (!rule) return;
  const bool one = !is_fx<L>() && ng > 2048;  // one record for the block
  if (w < W) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (with_f) {
        v.x += __shfl_down_sync(0xffffffffu, v.x, o);
        v.y += __shfl_down_sync(0xffffffffu, v.y, o);
      }
      v.z += __shfl_down_sync(0xffffffffu, v.z, o);
    }
    v.w = __any_sync(0xffffffffu, v.w != 0.0) ? 1.0 : 0.0;
    if (!one && (threadIdx.x & 31) == 0 && (R > 1 || W * vb + w < ng)) sweep_record(a, W * vb + w, v.x, v.y, v.z, v.w);
  }
  if constexpr (ALONE) {
    if (one) {
      __shared__ SweepSums part[W];
      if ((threadIdx.x & 31) == 0) part[w] = v;
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int q = 1; q < W; ++q) {
          v.x += part[q].x;
          v.y += part[q].y;
          v.z += part[q].z;
          v.w += part[q].w;
        }
        sweep_record(a, vb, v.x, v.y, v.z, v.w);
      }
    }
  }
  if (W > 1) {
    __threadfence();
    __syncthreads();
  }
  const int nb = cs_grad_blocks<L>(g.V, W);
  sweep_rule(g, a, with_f, nb, one ? nb : R > 1 ? W * nb : ng, FIRST ? 1 : 0);
}


// ------------------------------------------------------------------ Omega
// Packed Hermitian field: planes d0, d1, d2, re01, im01, re02, im02, re12, im12.
template <typename T>
__device__ __forceinline__ void store_herm(T* P, int s, int V, const herm& h) {
  P[0 * (size_t)V + s] = cvt<T>(h.d0);
  P[1 * (size_t)V + s] = cvt<T>(h.d1);
  P[2 * (size_t)V + s] = cvt<T>(h.d2);
  P[3 * (size_t)V + s] = cvt<T>(h.o01.re);
  P[4 * (size_t)V + s] = cvt<T>(h.o01.im);
  P[5 * (size_t)V + s] = cvt<T>(h.o02.re);
  P[6 * (size_t)V + s] = cvt<T>(h.o02.im);
  P[7 * (size_t)V + s] = cvt<T>(h.o12.re);
  P[8 * (size_t)V + s] = cvt<T>(h.o12.im);
}
template <typename T>
__device__ __forceinline__ void load_herm_mat(mat<T>& m, const T* __restrict__ P, int s, int V) {
  T d0 = __ldg(P + s), d1 = __ldg(P + (size_t)V + s), d2 = __ldg(P + 2 * (size_t)V + s);
  T a = __ldg(P + 3 * (size_t)V + s), b = __ldg(P + 4 * (size_t)V + s);
  T c = __ldg(P + 5 * (size_t)V + s), d = __ldg(P + 6 * (size_t)V + s);
  T e = __ldg(P + 7 * (size_t)V + s), f = __ldg(P + 8 * (size_t)V + s);
  m.e[0] = cx<T>{d0, T(0)};
  m.e[4] = cx<T>{d1, T(0)};
  m.e[8] = cx<T>{d2, T(0)};
  m.e[1] = cx<T>{a, b};
  m.e[3] = cx<T>{a, -b};
  m.e[2] = cx<T>{c, d};
  m.e[6] = cx<T>{c, -d};
  m.e[5] = cx<T>{e, f};
  m.e[7] = cx<T>{e, -f};
}
// H = c * sum_a g_a lambda_a (Hermitian, traceless), g real.
__device__ __forceinline__ herm herm_from_algebra(const double* g, double c) {
  const double r3 = 0.57735026918962576451;
  herm h;
  h.d0 = c * (g[2] + g[7] * r3);
  h.d1 = c * (-g[2] + g[7] * r3);
  h.d2 = c * (-2.0 * g[7] * r3);
  h.o01 = cx<double>{c * g[0], -c * g[1]};
  h.o02 = cx<double>{c * g[3], -c * g[4]};
  h.o12 = cx<double>{c * g[5], -c * g[6]};
  return h;
}
// The general path of either field, in FP64.
static __device__ __noinline__ void general_omega(const double* fa, double c, int2* Om, int2* Omi, int s, int V) {
  const herm h = herm_from_algebra(fa, c);
  herm om, omi;
  expm_hermitian_pair(om, omi, h);
  store_herm(tagged_herm{Om}, s, V, om);
  store_herm(tagged_herm{Omi}, s, V, omi);
}
static __device__ __noinline__ void general_omega_f32(const double* fa, double c, float* Om, float* Omi, int s, int V) {
  const herm h = herm_from_algebra(fa, c);
  herm om, omi;
  expm_hermitian_pair(om, omi, h, TAYLOR_TOL_FP32_STORAGE);
  store_herm(Om, s, V, om);
  store_herm(Omi, s, V, omi);
}

// exp(H) (sign 0), exp(-H) (1) or both (2) of a site into their fields; false
// when the site needs the general path.
template <typename L>
__device__ __forceinline__ bool sweep_omega(const fx_herm& H, const SweepArgs& a, int s, int V, int sign) {
  fx_exp_series S;
  if (!fx_exp_setup(S, H, is_fx<L>() ? TAYLOR_TOL_FP64 : TAYLOR_TOL_FP32_STORAGE)) return false;
#pragma unroll 1
  for (int k = sign == 1 ? 1 : 0; k <= (sign == 0 ? 0 : 1); ++k) {
    fx_herm om;
    fx_exp_sum(om, S, H, k == 1);
    void* P = k == 1 ? a.Omi : a.Om;
    if constexpr (is_fx<L>())
      fx_store_herm((int2*)P, s, V, om);
    else
      fx_store_herm((float*)P, s, V, om);
  }
  return true;
}

// Omega_x = exp(-eps alpha_ad f_ax lambda_a) and its inverse from f; one thread
// per site or (SPLIT) per site and sign, the inverses in the block's upper half.
template <typename L, bool SPLIT>
__device__ __forceinline__ void sweep_omega_body(const Geo& g, const SweepArgs& a, int vb) {
  if (a.cs->done) return;
  const int n = SPLIT ? CS_THREADS / 2 : CS_THREADS, s = vb * n + (int)threadIdx.x % n;
  if (s >= g.V) return;
  const int sign = SPLIT ? (int)threadIdx.x / n : 2;
  const double c = -a.ca.eps * a.cs->alpha_ad;
  double fa[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) fa[k] = __ldg(a.f + (size_t)k * g.V + s);
  fx_herm H;
  if (fx_herm_of_f(H, fa, c) && sweep_omega<L>(H, a, s, g.V, sign)) return;
  if (sign == 1) return;  // the other half takes the same way out and writes both
  double fg[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) fg[k] = fa[k];
  if constexpr (is_fx<L>())
    general_omega(fg, c, (int2*)a.Om, (int2*)a.Omi, s, g.V);
  else
    general_omega_f32(fg, c, (float*)a.Om, (float*)a.Omi, s, g.V);
}
__host__ __device__ inline int cs_omega_blocks(int V, bool split) {
  const int n = split ? CS_THREADS / 2 : CS_THREADS;
  return (V + n - 1) / n;
}

// Single-pass sweep of the D_0 / D_1 rules: their strength needs only the
// unitarity norm, which the previous sweep's apply summed, so the gradient
// goes straight into Omega.
// W = 1: two warps take the signs; W > 1: a thread per site forms both.
template <typename L, int W>
__device__ __forceinline__ void sweep_grad_omega_body(const Geo& g, const SweepArgs& a, int vb) {
  if (a.cs->done) return;
  constexpr bool ALONE = !is_fx<L>() && W > 1;
  __shared__ SweepPart<L, 9> sms[ALONE ? 1 : W];
  if constexpr (!ALONE) {
    constexpr bool PIPE = is_fx<L>() && W > 1;
    __shared__ int4 slot[PIPE ? fx_pipe<1>::WORDS : 1];
    fx_pipe<1> P(slot);
    if (PIPE) sweep_ask(P, g, a, W * vb);
#pragma unroll 1
    for (int p = 0; p < W; ++p) sweep_part<L, false, PIPE, 9>(sms[p], g, a, W * vb + p, P, p + 1 < W ? W * vb + p + 1 : -1);
    __syncthreads();
  }
  const int q = W == 1 ? 0 : threadIdx.x >> 5, sign = W == 1 ? (int)(threadIdx.x >> 5) : 2;
  const SweepPart<L, 9>& sm = sms[ALONE ? 0 : q];
  const int s = (W * vb + q) * CS_SITES + ((int)threadIdx.x & 31);
  if ((W == 1 ? threadIdx.x >= 64 : q >= W) || s >= g.V) return;
  const double c = -a.ca.eps * a.cs->alpha_ad;
  fx_herm H;
  bool ok;
  float ff[8];
  if constexpr (is_fx<L>()) {
    fx_gradient G;
    ok = sweep_gradient(G, sm) && fx_herm_of_gradient(H, G, c);
  } else {
    float r[10];
    if constexpr (ALONE) {
      sweep_sums_f32(r, g, (const float2*)a.U, s);
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) r[i] = sm.q[i][threadIdx.x & 31];
    }
    sweep_f(ff, r);
    ok = fx_herm_of_f(H, ff, c);
  }
  if (ok && sweep_omega<L>(H, a, s, g.V, sign)) return;
  if (sign == 1) return;
  double fg[8];
  if constexpr (is_fx<L>()) {
    general_cool_grad<L, false>(g, a.U, a.Ux, s, fg);
    general_omega(fg, c, (int2*)a.Om, (int2*)a.Omi, s, g.V);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) fg[k] = cvt<double>(ff[k]);
    general_omega_f32(fg, c, (float*)a.Om, (float*)a.Omi, s, g.V);
  }
}

// ------------------------------------------------------------------ apply
// Fixed point, general path of one link; returns Tr U U^+.
static __device__ __noinline__ double general_cool_apply(const Geo g, int4* Ux, int2* Om, int2* Omi, int mu, int s, int sp) {
  mat<double> o, oi, u, t;
  load_herm_mat(o, tagged_herm{Om}, s, g.V);
  load_herm_mat(oi, tagged_herm{Omi}, sp, g.V);
  load(u, tagged{Ux, 0}, mu, s, g.V);
  mul_herm_left(t, o, u);
  mul_herm_right(u, t, oi);
  store(tagged{Ux, 0}, mu, s, g.V, u);
  return norm2(u);
}
// U_{x,mu} <- Omega_x U_{x,mu} Omega_{x+mu}^{-1}, all links at once (in place:
// every link is read and written by the same thread).  RULE: the single-pass
// sweeps' rule from the new links' norm.  last: the call's last enqueued sweep,
// which leaves the links in U (fixed point): its own results, or, when the
// rule has stopped the call after at least one sweep, what the words hold.
// Norms are summed as integers, exactly, within a record: a link's Tr U U^+ - 3
// (below 1.9) in units of 2^(sh - 60), so that R groups of 128 links fit; links
// beyond that (wild) in FP64.
// The apply is linear in the link: one beyond the bound goes through it times
// 1/8, and back into fixed point where it fits.  Returns Tr U U^+.
static __device__ __noinline__ double far_cool_apply(const Geo g, int4* Ux, int2* Om, int2* Omi, int mu, int s, int sp) {
  fx_chk ck;
  fx_herm o, oi;
  mat<fx> u;
  fx_load_herm(o, Om, s, g.V, ck);
  fx_load_herm(oi, Omi, sp, g.V, ck);
  if (!fx_load_wild<3>(u, Ux, mu, s, g.V)) ck.fail();
  fx_apply_ops ops;
  fx_lhs(ops, o);
  long long dev = 0;
  fx_apply_link<true>(u, ops, oi, ck, dev);
  if (ck.bad()) return general_cool_apply(g, Ux, Om, Omi, mu, s, sp);
  int top = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) top = max(top, max(abs(u.e[k].re.h), abs(u.e[k].im.h)));
  const bool fits = top < (int)(1.4375 / 8 * (1 << 30)) - 1;
  int4* p = Ux + (size_t)mu * 9 * g.V + s;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const long long re = fx_bits(u.e[k].re), im = fx_bits(u.e[k].im);
    if (fits) {
      p[(size_t)k * g.V] = pack(cx<fx>{fx_of_bits(re << 3), fx_of_bits(im << 3)});
    } else {
      const double x = fx_bits_to_double(re, 3), y = fx_bits_to_double(im, 3);
      const int2 w = k == 0 ? fx_raw_first(x) : make_int2(__double2loint(x), __double2hiint(x));
      p[(size_t)k * g.V] = make_int4(w.x, w.y, __double2loint(y), __double2hiint(y));
    }
  }
  return 192.0 + fx_bits_to_double(dev, 6);  // dev: Tr (U / 8) (U / 8)^+ - 3
}
// A thread's next link and its two Omegas on their way into shared memory while
// it works on the current ones (lattices where a block takes several groups:
// apply of a 32^4 step of ten sweeps 4.03 -> 3.74 ms; now 3.63).
// Item k of a thread at sm[k CS_THREADS + thread]; a thread's own, no barrier.
struct sweep_pipe {
  int4* sm;
  __device__ __forceinline__ void ask(const SweepArgs& a, int mu, int s, int sp, int V) const {
    const int4* u = (const int4*)a.Ux + (size_t)mu * 9 * V + s;
    const int2 *o = (const int2*)a.Om + s, *oi = (const int2*)a.Omi + sp;
    const unsigned d = (unsigned)__cvta_generic_to_shared(sm);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + k * CS_THREADS * 16), "l"(u + (size_t)k * V) : "memory");
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + (9 + k) * CS_THREADS * 16), "l"(o + (size_t)k * V) : "memory");
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + (9 + k) * CS_THREADS * 16 + 8), "l"(oi + (size_t)k * V) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void take(mat<fx>& u, fx_herm& o, fx_herm& oi, fx_chk& ck) const {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    int4 h[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      u.e[k] = unpack(sm[k * CS_THREADS]);
      h[k] = sm[(9 + k) * CS_THREADS];
    }
    int2 w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = make_int2(h[k].x, h[k].y);
    fx_unpack_herm(o, w, ck);
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = make_int2(h[k].z, h[k].w);
    fx_unpack_herm(oi, w, ck);
  }
};
template <typename L, bool RULE>
__device__ __forceinline__ void sweep_apply_body(const Geo& g, const SweepArgs& a, int vb, bool last) {
  typedef typename vec2_of<L>::type V2;
  const int mu = threadIdx.x >> 5, R = cs_rounds<L>(g.V);
  V2* U = (V2*)const_cast<void*>(a.U);
  const bool stopped = a.cs && a.cs->done;
  if (stopped && !(last && a.cs->sweeps > 0)) return;
  const int sh = 6 + (R > 1 ? 32 - __clz(R - 1) : 0);
  long long acc = 0;
  double wild = 0.0;
  int nwild = 0;
  __shared__ int4 sm[18 * CS_THREADS];
  const sweep_pipe P = {sm + threadIdx.x};
  int sp0 = 0;  // the next site's neighbour, asked for already
  if (R > 1 && !stopped) {
    const int s = R * vb * CS_SITES + ((int)threadIdx.x & 31);
    if (s < g.V) {
      int x[4];
      site_coords(g, s, x);
      sp0 = hop(g, s, x, mu, 1);
      P.ask(a, mu, s, sp0, g.V);
    }
  }
  for (int j = 0; j < R; ++j) {
    const int s = (R * vb + j) * CS_SITES + ((int)threadIdx.x & 31);
    if (s >= g.V) break;
    if (stopped) {
      unload_link(U, (const int4*)a.Ux, mu, s, g.V);
      continue;
    }
    int x[4];
    int sp = sp0;
    int4* Ux = (int4*)a.Ux;
    fx_chk ck;
    fx_herm o, oi;
    mat<fx> u;
    if (R > 1) {
      P.take(u, o, oi, ck);
      const int s1 = s + CS_SITES;
      if (j + 1 < R && s1 < g.V) {
        site_coords(g, s1, x);
        sp0 = hop(g, s1, x, mu, 1);
        P.ask(a, mu, s1, sp0, g.V);
      }
    } else {
      site_coords(g, s, x);
      sp = hop(g, s, x, mu, 1);
      fx_load_herm(o, (const int2*)a.Om, s, g.V, ck);
      fx_load_herm(oi, (const int2*)a.Omi, sp, g.V, ck);
      fx_load_plain(u, Ux, mu, s, g.V);
    }
    long long dev = 0;
    if (fx_is_raw(u.e[0].re.l)) {
      ck.fail();
    } else {
      fx_apply_ops ops;
      fx_lhs(ops, o);
      fx_apply_link<RULE>(u, ops, oi, ck, dev);
    }
    if (!ck.bad()) {
      if (last) fx_store_link(U, mu, s, g.V, u);
      if (!last || !RULE) store<fx>(Ux, mu, s, g.V, u);  // D_2 calls end with a gradient
      acc += dev >> sh;
    } else {
      wild += far_cool_apply(g, Ux, (int2*)a.Om, (int2*)a.Omi, mu, s, sp) - 3.0;
      nwild = 1;
      if (last) unload_link(U, Ux, mu, s, g.V);
    }
  }
  if constexpr (RULE) {
    if (stopped) return;
    __shared__ long long sums[CS_THREADS / 32];
    __shared__ double wilds[CS_THREADS / 32];
    const auto warp_sum = [](double w) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
      return w;
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    const bool any_warp = __any_sync(0xffffffffu, nwild != 0);
    const double w = any_warp ? warp_sum(wild) : 0.0;
    if ((threadIdx.x & 31) == 0) {
      sums[threadIdx.x >> 5] = acc;
      wilds[threadIdx.x >> 5] = w;
    }
    const int any = __syncthreads_or(nwild);
    SweepNorm* n = sweep_norm(a, g.V);
    if (threadIdx.x == 0) {
      const long long t = sums[0] + sums[1] + sums[2] + sums[3];
      atomicAdd(&n->hi, (unsigned long long)(t >> 20));
      atomicAdd(&n->lo, (unsigned long long)(t & 0xfffff));
      if (any) atomicAdd(&n->wild, 1u);
      __stcg(a.rec + 2 * vb, make_double2(any ? (wilds[0] + wilds[1]) + (wilds[2] + wilds[3]) : 0.0, 0.0));
    }
    const int nb = cs_apply_blocks<L>(g.V, 1);
    if (!sweep_last(a, nb)) return;
    double far = 0.0;  // links beyond the bound, by the whole block
    if (__ldcg(&n->wild) != 0u) {
      for (int b = threadIdx.x; b < nb; b += CS_THREADS) far += __ldcg(a.rec + 2 * b).x;
      far = warp_sum(far);
      if ((threadIdx.x & 31) == 0) wilds[threadIdx.x >> 5] = far;
      __syncthreads();
      far = (wilds[0] + wilds[1]) + (wilds[2] + wilds[3]);
    }
    if (threadIdx.x != 0) return;
    const CoolState old = *a.cs;
    const long long hi = (long long)__ldcg(&n->hi), lo = (long long)__ldcg(&n->lo);
    const double dev = fx_bits_to_double(hi, sh + 20) + fx_bits_to_double(lo, sh) + far;
    cool_rule(1.0 + dev * ((1.0 / 3.0) * a.ca.inv_links), 0.0, 0.0, false, a.ca, old, a.cs, 0);
    *n = SweepNorm{0ull, 0ull, 0.0, 0u, 0u};
    *a.ticket = 0u;
  }
}

// FP32 storage: the apply of one link; returns Tr U U^+.
__device__ __forceinline__ float sweep_apply_f32(float2* U, const mat<float>& o, const float* Omi, const Geo& g, int mu, int s,
                                                 const int* x) {
  mat<float> oi, u, w;
  load_herm_mat(oi, Omi, hop(g, s, x, mu, 1), g.V);
  load(u, U, mu, s, g.V);
  mul_herm_left(w, o, u);
  mul_herm_right(u, w, oi);
  store(U, mu, s, g.V, u);
  return norm2(u);
}
// W = 1: a group, a warp per direction; W = 4: a thread per site, which loads
// Omega_x once, cs_rounds rounds of 128 sites (32^4, ten sweeps: 1.20 ms against
// 1.25; 16^4: 0.153 against 0.173).  RULE as above; a site's norm is the float sum over mu = 0 .. 3
// (the order matters, see sweep_add_f32), the lattice's an exact one: integers
// in units of 2^-36, which hold every float above 2^-12; sites of norm beyond
// 1,024 (or not finite) in FP64.
template <bool RULE, int W>
__device__ __forceinline__ void sweep_apply_f32_body(const Geo& g, const SweepArgs& a, int vb) {
  if (a.cs && a.cs->done) return;
  float2* U = (float2*)const_cast<void*>(a.U);
  const float *Om = (const float*)a.Om, *Omi = (const float*)a.Omi;
  long long acc = 0;
  double far = 0.0;
  int nfar = 0;
  const auto site = [&](float un) {
    if (un < 1024.0f) {
      acc += __float2ll_rn(un * 0x1p36f) - (12ll << 36);
    } else {
      far += cvt<double>(un) - 12.0;
      nfar = 1;
    }
  };
  mat<float> o;
  int x[4];
  if (W > 1) {
    const int R = cs_rounds<float>(g.V);
    for (int j = 0; j < R; ++j) {
      const int s = (R * vb + j) * CS_THREADS + (int)threadIdx.x;
      if (s >= g.V) break;
      site_coords(g, s, x);
      load_herm_mat(o, Om, s, g.V);
      float un = 0.0f;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) un += sweep_apply_f32(U, o, Omi, g, mu, s, x);
      if (RULE) site(un);
    }
  } else {
    __shared__ float n[4][CS_SITES];
    const int mu = threadIdx.x >> 5, l = threadIdx.x & 31, s = vb * CS_SITES + l;
    if (s < g.V) {
      site_coords(g, s, x);
      load_herm_mat(o, Om, s, g.V);
      n[mu][l] = sweep_apply_f32(U, o, Omi, g, mu, s, x);
    }
    if (RULE) {
      __syncthreads();
      if (mu == 0 && s < g.V) site(((n[0][l] + n[1][l]) + n[2][l]) + n[3][l]);
    }
  }
  if constexpr (RULE) {
    __shared__ long long sums[CS_THREADS / 32];
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, k);
    if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = acc;
    SweepNorm* n = sweep_norm(a, g.V);
    if (nfar) atomicAdd(&n->far, far);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const long long t = sums[0] + sums[1] + sums[2] + sums[3];
      atomicAdd(&n->hi, (unsigned long long)(t >> 20));
      atomicAdd(&n->lo, (unsigned long long)(t & 0xfffff));
    }
    if (!sweep_last(a, cs_apply_blocks<float>(g.V, W))) return;
    if (threadIdx.x != 0) return;
    const CoolState old = *a.cs;
    const long long hi = (long long)__ldcg(&n->hi), lo = (long long)__ldcg(&n->lo);
    const double dev = fx_bits_to_double(hi, 44) + fx_bits_to_double(lo, 24) + __ldcg(&n->far);
    cool_rule(1.0 + dev * ((1.0 / 3.0) * a.ca.inv_links), 0.0, 0.0, false, a.ca, old, a.cs, 0);
    *n = SweepNorm{0ull, 0ull, 0.0, 0u, 0u};
    *a.ticket = 0u;
  }
}

// The apply of either field; wide: FP32 storage at W = 4.
template <typename L, bool RULE, bool WIDE>
__device__ __forceinline__ void sweep_apply(const Geo& g, const SweepArgs& a, int vb, bool last) {
  if constexpr (is_fx<L>())
    sweep_apply_body<L, RULE>(g, a, vb, last);
  else
    sweep_apply_f32_body<RULE, WIDE ? 4 : 1>(g, a, vb);
}

}  // namespace clgc
