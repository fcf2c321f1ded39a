// kernels.cu -- starts, layout conversion, clover field, gauge cooling and
// observables.  The CL update kernel itself is in k_update.cuh
// (instantiated by k_update_f64.cu / k_update_f32.cu).
#include <type_traits>

#include "cool_sweep.cuh"
#include "cvt.cuh"
#include "expm.cuh"
#include "fixed.cuh"
#include "launch.h"
#include "lattice.cuh"
#include "noise_fx.cuh"
#include "philox.cuh"
#include "su3.cuh"

namespace clgc {

// Resident blocks of CS_THREADS threads the apply is built for.
#define CS_APPLY_BLOCKS(L) (is_fx<L>() ? 3 : 7)

namespace {

const double KAPPA_Q = -1.0 / (256.0 * 9.86960440108935861883);  // -1/(256 pi^2)

Geo to_geo(const GeoH& h) { return make_geo(h.L, h.V); }

inline dim3 grid_sites(int V, int planes = 1) {
  return dim3((unsigned)((V + RED_THREADS - 1) / RED_THREADS), (unsigned)planes);
}

// Fixed-order block reduction of NQ doubles (slot MAXSLOT takes the max)
// into the block's record rec[0 .. NQ-1].
template <int NQ, int MAXSLOT>
__device__ __forceinline__ void block_reduce_store(double* v, double* rec) {
  __shared__ double sm[RED_THREADS / 32][NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      double o = __shfl_down_sync(0xffffffffu, v[q], off);
      v[q] = (q == MAXSLOT) ? fmax(v[q], o) : v[q] + o;
    }
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NQ; ++q) sm[w][q] = v[q];
  __syncthreads();
  if (threadIdx.x < NQ) {
    int q = threadIdx.x;
    double s = sm[0][q];
    for (int k = 1; k < RED_THREADS / 32; ++k) s = (q == MAXSLOT) ? fmax(s, sm[k][q]) : s + sm[k][q];
    rec[q] = s;
  }
}

// Single-block fixed-order sum of nb records of NQ doubles.
template <int NQ, int MAXSLOT>
__device__ __forceinline__ void reduce_partials(const double* partials, int nb, double* out) {
  __shared__ double sm[256][NQ];
  double v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double x = partials[(size_t)b * NQ + q];
      v[q] = (q == MAXSLOT) ? fmax(v[q], x) : v[q] + x;
    }
#pragma unroll
  for (int q = 0; q < NQ; ++q) sm[threadIdx.x][q] = v[q];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        sm[threadIdx.x][q] = (q == MAXSLOT) ? fmax(sm[threadIdx.x][q], sm[threadIdx.x + w][q])
                                            : sm[threadIdx.x][q] + sm[threadIdx.x + w][q];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int q = 0; q < NQ; ++q) out[q] = sm[0][q];
}

template <typename T>
__device__ __forceinline__ bool finite_mat(const mat<T>& a) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) ok = ok && isfinite(a.e[k].re) && isfinite(a.e[k].im);
  return ok;
}

// --------------------------------------------------------------- starts
template <typename T>
__global__ void k_cold(Geo g, typename vec2_of<T>::type* U) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  mat<T> I;
  set_ident(I);
  store(U, blockIdx.y, s, g.V, I);
}

// Haar SU(3): Gram-Schmidt on the rows of a complex Gaussian matrix (Philox
// stream 2) gives Haar U(3); the principal cube root of the determinant maps
// it to SU(3).
template <typename T>
__global__ void k_hot(Geo g, typename vec2_of<T>::type* U, uint64_t seed) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int mu = blockIdx.y;
  double z[18];
  normals_f64<9>(z, seed, 0u, (uint32_t)s, (uint32_t)mu, STREAM_HOT);
  mat<double> m;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k] = cx<double>{z[2 * k], z[2 * k + 1]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int k = 0; k < i; ++k) {
      cx<double> ip = {0.0, 0.0};  // <row_k, row_i>
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cx<double> ck = {m.e[3 * k + j].re, -m.e[3 * k + j].im};
        ip = cfma(ck, m.e[3 * i + j], ip);
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) m.e[3 * i + j] = cfms(ip, m.e[3 * k + j], m.e[3 * i + j]);
    }
    double n = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) n = fma(m.e[3 * i + j].re, m.e[3 * i + j].re, fma(m.e[3 * i + j].im, m.e[3 * i + j].im, n));
    double inv = 1.0 / sqrt(n);
#pragma unroll
    for (int j = 0; j < 3; ++j) { m.e[3 * i + j].re *= inv; m.e[3 * i + j].im *= inv; }
  }
  cx<double> zf = det_inv_cuberoot(det(m));
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k] = cmul(m.e[k], zf);
  mat<T> t;
  convert(t, m);
  store(U, mu, s, g.V, t);
}

// Omega_x = exp(i w_a lambda_a) with w_a = i sigma g_a, i.e. exp(-sigma g_a lambda_a).
template <typename T>
__global__ void k_gauge_omega(Geo g, T* Om, T* Omi, uint64_t seed, double sigma) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  double r[8];
  normals_f64<4>(r, seed, 0u, (uint32_t)s, 0u, STREAM_GAUGE);
  herm h = herm_from_algebra(r, -sigma), om, omi;
  expm_hermitian_pair(om, omi, h, taylor_tol<T>());
  if constexpr (is_fx<T>()) {
    store_herm(tagged_herm{(int2*)Om}, s, g.V, om);
    store_herm(tagged_herm{(int2*)Omi}, s, g.V, omi);
  } else {
    store_herm(Om, s, g.V, om);
    store_herm(Omi, s, g.V, omi);
  }
}

// The CL noise of links (site0 + i, mu) as form T draws it (a diagnostic).
template <typename T>
__global__ void k_noise_sample(int site0, int n, uint64_t seed, uint32_t step, uint32_t mu, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t s = (uint32_t)(site0 + i);
  if constexpr (is_fx<T>()) {
    fx e[8];
    normals_fx<4>(e, seed, step, s, mu, STREAM_CL);
#pragma unroll
    for (int j = 0; j < 8; ++j) out[8 * (size_t)i + j] = fx_to_double(e[j], 3);
  } else {
    float e[8];
    normals_f32<4>(e, seed, step, s, mu, STREAM_CL);
#pragma unroll
    for (int j = 0; j < 8; ++j) out[8 * (size_t)i + j] = (double)e[j];
  }
}

// ------------------------------------------------------------ conversion
// AoS [site][plane][row][col]{re,im} doubles <-> SoA planes of T2, through a
// shared-memory transpose of CONV_SITES sites: the AoS side (often the host's
// page-locked memory, read or written over the host link) is one contiguous
// run per block, and the SoA side is CONV_SITES consecutive sites per row.
// The tile's pitch is odd in 16-byte units, so the column-wise accesses of a
// quarter warp hit distinct banks.  16-byte accesses with a tile's loads in
// flight at once where the buffer is aligned: both directions then run at the
// host link's rate (24^3 x 32 links from / to page-locked memory 1.22 / 1.33 ms,
// the copy engine's 1.23 / 1.34; out in 8-byte writes 1.82 ms).
const int CONV_SITES = 32, CONV_MAX_ROWS = 54;  // up to 6 planes
const int CONV_BATCH = 5;  // AoS loads in flight per thread (36 rows: the whole tile)
__host__ __device__ constexpr int conv_pitch(int rows) { return rows + 1 + (rows & 1); }

template <typename T>
__global__ void __launch_bounds__(256) k_aos_to_soa(Geo g, const double* __restrict__ aos,
                                                    typename vec2_of<T>::type* U, int nplanes) {
  __shared__ double2 buf[CONV_SITES * conv_pitch(CONV_MAX_ROWS)];
  const int R = 9 * nplanes, pitch = conv_pitch(R);
  const int s0 = blockIdx.x * CONV_SITES;
  const int ns = min(CONV_SITES, g.V - s0), n = ns * R;
  const double* src = aos + 2 * (size_t)s0 * R;
  // a caller's buffer need only be aligned to 8 bytes
  const bool wide = (reinterpret_cast<size_t>(src) & 15) == 0;
  for (int e0 = threadIdx.x; e0 < n; e0 += CONV_BATCH * 256) {
    double2 v[CONV_BATCH];
#pragma unroll
    for (int q = 0; q < CONV_BATCH; ++q) {
      const int e = e0 + q * 256;
      if (e < n) v[q] = wide ? __ldcs(reinterpret_cast<const double2*>(src) + e) : make_double2(src[2 * e], src[2 * e + 1]);
    }
#pragma unroll
    for (int q = 0; q < CONV_BATCH; ++q) {
      const int e = e0 + q * 256;
      const int j = e / R, r = e - j * R;
      if (e < n) buf[j * pitch + r] = v[q];
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < R * CONV_SITES; e += blockDim.x) {
    const int r = e / CONV_SITES, j = e - r * CONV_SITES;
    if (j < ns) {
      const double2 v = buf[j * pitch + r];
      U[(size_t)r * g.V + s0 + j] = pack(cx<T>{(T)v.x, (T)v.y});
    }
  }
}
template <typename T>
__global__ void __launch_bounds__(256) k_soa_to_aos(Geo g, const typename vec2_of<T>::type* __restrict__ U,
                                                    double* aos, int nplanes) {
  __shared__ double2 buf[CONV_SITES * conv_pitch(CONV_MAX_ROWS)];
  const int R = 9 * nplanes, pitch = conv_pitch(R);
  const int s0 = blockIdx.x * CONV_SITES;
  const int ns = min(CONV_SITES, g.V - s0);
  for (int e = threadIdx.x; e < R * CONV_SITES; e += blockDim.x) {
    const int r = e / CONV_SITES, j = e - r * CONV_SITES;
    if (j < ns) {
      const cx<T> c = unpack(U[(size_t)r * g.V + s0 + j]);
      buf[j * pitch + r] = make_double2((double)c.re, (double)c.im);
    }
  }
  __syncthreads();
  double* dst = aos + 2 * (size_t)s0 * R;
  const bool wide = (reinterpret_cast<size_t>(dst) & 15) == 0;
  for (int e = threadIdx.x; e < ns * R; e += blockDim.x) {
    const int j = e / R, r = e - j * R;
    const double2 v = buf[j * pitch + r];
    if (wide) {
      __stcs(reinterpret_cast<double2*>(dst) + e, v);
    } else {
      dst[2 * e] = v.x;
      dst[2 * e + 1] = v.y;
    }
  }
}

// --------------------------------------------------------------- cooling
// The kernels of cool_sweep.cuh, one launch per lattice.
template <typename L, bool FIRST, int W>
__global__ void __launch_bounds__(CS_THREADS, is_fx<L>() ? 4 : 0) k_cool_grad(Geo g, SweepArgs a, int rule) {
  sweep_grad_body<L, FIRST, W>(g, a, blockIdx.x, rule != 0);
}
template <typename L, bool SPLIT>
__global__ void __launch_bounds__(CS_THREADS) k_cool_omega(Geo g, SweepArgs a) {
  sweep_omega_body<L, SPLIT>(g, a, blockIdx.x);
}
template <typename L, int W>
__global__ void __launch_bounds__(CS_THREADS) k_cool_grad_omega(Geo g, SweepArgs a) {
  sweep_grad_omega_body<L, W>(g, a, blockIdx.x);
}
template <typename L, bool RULE, bool WIDE>
__global__ void __launch_bounds__(CS_THREADS, CS_APPLY_BLOCKS(L)) k_cool_apply(Geo g, SweepArgs a, int last) {
  sweep_apply<L, RULE, WIDE>(g, a, blockIdx.x, last != 0);
}
// The links' fixed-point words, for an apply without a gradient before it.
template <typename L>
__global__ void __launch_bounds__(CS_THREADS) k_cool_load(Geo g, const typename vec2_of<L>::type* __restrict__ U, int4* Ux) {
  const int mu = threadIdx.x >> 5, s = blockIdx.x * CS_SITES + ((int)threadIdx.x & 31);
  if (s >= g.V) return;
  mat<fx> u;
  if (fx_load_link<L>(u, U, mu, s, g.V)) {
    store<fx>(Ux, mu, s, g.V, u);
  } else {
    mat<double> d;
    load_link_d<L>(d, U, mu, s, g.V);
    store(tagged{Ux, 0}, mu, s, g.V, d);
  }
}

// ----------------------------------------------------------- observables
// Per site: Tr P / 3 and Tr P + Tr P^{-1} of the six plaquettes (from the
// plaquette pass's P and D = P - P^{-1}), (1/3) Tr U U^+ of the four links,
// max |det U - 1|^2, nonfinite count and q_L(x) = kappa [Tr F01 F23 - Tr F02 F13
// + Tr F03 F12] of the clover field.  Sums of a site run in fixed point and
// are widened to FP64 once (GB300's FP64 rate again: 430 us at 16^4 with the
// plaquettes, determinants and traces formed in FP64).

// One link's Tr U U^+ - 3 (60-bit integer, within 1.95 of zero: four are added)
// and |det U - 1|^2; false out of range.
__device__ __forceinline__ bool obs_link(const mat<fx>& u, long long& dev, double& det2) {
  fx_chk ck;
  fx_acc n = fx_zero();
  float nf = 0.0f;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    fx_mac(n, fx_lhs(u.e[k].re), fx_rhs(u.e[k].re));
    fx_mac(n, fx_lhs(u.e[k].im), fx_rhs(u.e[k].im));
    nf = fmaf((float)u.e[k].re.h, (float)u.e[k].re.h, fmaf((float)u.e[k].im.h, (float)u.e[k].im.h, nf));
  }
  const cx<fx> e = fx_det_minus_one(u, ck);
  if (ck.bad() || !(nf > 1.05f * 0x1p60f && nf < 4.9f * 0x1p60f)) return false;
  dev += fx_sum(n) - ((3ll << 60) + (1 << 29));
  const double re = fx_to_double(e.re), im = fx_to_double(e.im);
  det2 = fmax(det2, fma(re, re, im * im));
  return true;
}
// The same of a link beyond the range (or not finite), in FP64; returns Tr U U^+.
template <typename T>
static __device__ __noinline__ double general_obs_link(const typename vec2_of<T>::type* U, int mu, int s, int V, double* det2,
                                                       double* bad) {
  mat<double> u;
  load_link_d<T>(u, U, mu, s, V);
  if (!finite_mat(u)) *bad = 1.0;
  const cx<double> d = det(u);
  const double h = hypot(d.re - 1.0, d.im);
  *det2 = fmax(*det2, h * h);
  return norm2(u);
}
// Tr of a stored matrix times 1/4 as a 60-bit integer (FP32 storage: of its float
// trace).  Six of them are added: each below 5.3 / 4 (fixed point: 3 1.4375 / 4).
__device__ __forceinline__ bool obs_trace(long long& re, long long& im, const float2* f, int p, int s, int V) {
  float tr = 0.0f, ti = 0.0f;
#pragma unroll
  for (int k = 0; k < 9; k += 4) {
    const float2 w = __ldg(f + ((size_t)p * 9 + k) * V + s);
    tr += w.x;
    ti += w.y;
  }
  if (!(fabsf(tr) < 5.3f && fabsf(ti) < 5.3f)) return false;
  re = fx_bits(fx_of_float(0.25f * tr));
  im = fx_bits(fx_of_float(0.25f * ti));
  return true;
}
__device__ __forceinline__ bool obs_trace(long long& re, long long& im, const int4* P, int p, int s, int V) {
  bool ok = true;
  re = im = 0;
#pragma unroll
  for (int k = 0; k < 9; k += 4) {
    const cx<fx> w = unpack(__ldg(P + ((size_t)p * 9 + k) * V + s));
    if (k == 0 && fx_is_raw(w.re.l)) ok = false;
    re += fx_bits(w.re) >> 2;
    im += fx_bits(w.im) >> 2;
  }
  return ok;
}
static __device__ __noinline__ void general_obs_trace(const int4* f, int p, int s, int V, int ex, double* out) {
  mat<double> m;
  load(m, tagged{const_cast<int4*>(f), ex}, p, s, V);
  const cx<double> t = trace(m);
  out[0] = t.re;
  out[1] = t.im;
}
static __device__ __noinline__ void general_obs_trace(const float2* f, int p, int s, int V, int, double* out) {
  mat<float> m;
  load(m, f, p, s, V);
  const cx<float> t = trace(m);
  out[0] = (double)t.re;
  out[1] = (double)t.im;
}
// Tr F_p F_{5-p} in FP64.
static __device__ __noinline__ void general_obs_ff(const int4* F, int p, int s, int V, int ex, double* out) {
  mat<double> F1, F2;
  load(F1, tagged{const_cast<int4*>(F), ex}, p, s, V);
  load(F2, tagged{const_cast<int4*>(F), ex}, 5 - p, s, V);
  const cx<double> t = trace_mul(F1, F2);
  out[0] = t.re;
  out[1] = t.im;
}

// The type of the plaquette and clover fields' words.
template <typename T>
struct obs_word { typedef typename std::conditional<is_fx<T>(), int4, float2>::type type; };
template <typename T>
__global__ void __launch_bounds__(RED_THREADS) k_obs(Geo g, const typename vec2_of<T>::type* __restrict__ U,
                                                    const int4* __restrict__ Ux,
                                                    const typename obs_word<T>::type* __restrict__ Pq,
                                                    const typename obs_word<T>::type* __restrict__ Dq,
                                                    const typename obs_word<T>::type* __restrict__ F,
                                                    double* partials, double* q_site, const unsigned* top) {
  constexpr bool FX = is_fx<T>();
  double v[NQ_OBS];
#pragma unroll
  for (int q = 0; q < NQ_OBS; ++q) v[q] = 0.0;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < g.V; s += gridDim.x * blockDim.x) {
    // links
    long long dev = 0;
    double wild = 0.0, det2 = 0.0, bad = 0.0;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      mat<fx> u;
      bool in;
      if constexpr (FX) {
        load<fx>(u, Ux, mu, s, g.V);
        in = !fx_is_raw(u.e[0].re.l);
      } else {
        mat<T> w;
        load(w, U, mu, s, g.V);
        in = true;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          in = in && fabsf((float)w.e[k].re) < 1.4375f && fabsf((float)w.e[k].im) < 1.4375f;
          u.e[k] = cx<fx>{fx_of_float((float)w.e[k].re), fx_of_float((float)w.e[k].im)};
        }
      }
      if (!in || !obs_link(u, dev, det2)) wild += general_obs_link<T>(U, mu, s, g.V, &det2, &bad) - 3.0;
    }
    v[4] += (12.0 + (fx_bits_to_double(dev) + wild)) * (1.0 / 3.0);
    v[7] = fmax(v[7], det2);
    v[8] += bad;
    // plaquettes: Tr P and Tr P^{-1} = Tr P - Tr D (the fixed-point D is halved)
    long long pr = 0, pi = 0, dr = 0, di = 0;  // units of 2^-58
    double wp[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      long long a, b, c, d;
      if (obs_trace(a, b, Pq, p, s, g.V) && obs_trace(c, d, Dq, p, s, g.V)) {
        pr += a;
        pi += b;
        dr += c;
        di += d;
      } else {
        double t[2];
        general_obs_trace(Pq, p, s, g.V, 0, t);
        wp[0] += t[0];
        wp[1] += t[1];
        general_obs_trace(Dq, p, s, g.V, 1, t);
        wp[2] += t[0];
        wp[3] += t[1];
      }
    }
    const double tr = fx_bits_to_double(pr, 2) + wp[0], ti = fx_bits_to_double(pi, 2) + wp[1];
    v[0] += tr * (1.0 / 3.0);
    v[1] += ti * (1.0 / 3.0);
    v[2] += 2.0 * tr - (fx_bits_to_double(dr, FX ? 3 : 2) + wp[2]);
    v[3] += 2.0 * ti - (fx_bits_to_double(di, FX ? 3 : 2) + wp[3]);
    // topological charge density (fixed point: F is an eighth of the clover field)
    cx<double> q = {0.0, 0.0};
    if constexpr (FX) {
      fx_acc re = fx_zero(), im = fx_zero();
      fx_chk ck;
      const int shift = fx_field_shift(top);
      float nf = 0.0f;  // sum of |F|^2, twice a bound of the traces' sum
#pragma unroll 1
      for (int p = 0; p < 3; ++p) {  // the planes 1 and 4 are both stored negated
        mat<fx> F1, F2;
        fx_load(F1, F, p, s, g.V, ck);
        fx_load(F2, F, 5 - p, s, g.V, ck);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const cx<fx> x = F1.e[3 * i + k], y = F2.e[3 * k + i];
            fx_cmac(re, im, p == 1 ? fx_lhs_neg(x) : fx_lhs(x), fx_rhs(y));
            nf = fmaf((float)x.re.h, (float)x.re.h, fmaf((float)x.im.h, (float)x.im.h, nf));
            nf = fmaf((float)y.re.h, (float)y.re.h, fmaf((float)y.im.h, (float)y.im.h, nf));
          }
      }
      if (!ck.bad() && nf < 15.0f * 0x1p60f) {
        q.re = fx_bits_to_double(fx_sum<true>(re) - (1 << 29), -2 * shift);
        q.im = fx_bits_to_double(fx_sum<true>(im) - (1 << 29), -2 * shift);
      } else {
        for (int p = 0; p < 3; ++p) {
          double t[2];
          general_obs_ff(F, p, s, g.V, -shift, t);
          q.re += p == 1 ? -t[0] : t[0];
          q.im += p == 1 ? -t[1] : t[1];
        }
      }
      q.re *= 64.0 * KAPPA_Q;
      q.im *= 64.0 * KAPPA_Q;
    } else {
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        mat<T> F1, F2;
        load(F1, F, p, s, g.V);
        load(F2, F, 5 - p, s, g.V);
        const cx<T> t = trace_mul(F1, F2);
        q.re += p == 1 ? -cvt<double>(t.re) : cvt<double>(t.re);
        q.im += p == 1 ? -cvt<double>(t.im) : cvt<double>(t.im);
      }
      q.re *= KAPPA_Q;
      q.im *= KAPPA_Q;
    }
    v[5] += q.re;
    v[6] += q.im;
    if (q_site) {
      q_site[2 * (size_t)s] = q.re;
      q_site[2 * (size_t)s + 1] = q.im;
    }
  }
  block_reduce_store<NQ_OBS, 7>(v, partials + (size_t)blockIdx.x * NQ_OBS);
}

__global__ void k_obs_final(Geo g, const double* partials, int nb, double beta, double th_re,
                            double th_im, ObsOut* out) {
  __shared__ double tot[NQ_OBS];
  reduce_partials<NQ_OBS, 7>(partials, nb, tot);
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double V = (double)g.V, np = 6.0 * V;
  out->plaq_re = tot[0] / np;
  out->plaq_im = tot[1] / np;
  out->un = tot[4] / (4.0 * V);
  out->q_re = tot[5];
  out->q_im = tot[6];
  out->sw_re = beta * np - beta / 6.0 * tot[2];
  out->sw_im = -beta / 6.0 * tot[3];
  // S = S_W - i theta Q
  out->s_re = out->sw_re + th_re * tot[6] + th_im * tot[5];
  out->s_im = out->sw_im - th_re * tot[5] + th_im * tot[6];
  out->max_det_dev = sqrt(tot[7]);
  out->nonfinite = tot[8];
}

// Self-test of the integer-pipe conversions (cvt.cuh) against the hardware
// ones, bit for bit (NaN against NaN).  Case i draws 64 random bits by the
// SplitMix64 finaliser of seed + i: all 32-bit float patterns (every exponent,
// subnormals, infinities, NaNs) for f2d; for d2f doubles whose exponent spans
// the float range and both its ends (underflow to zero, overflow to inf),
// every fourth an exact rounding tie, every eighth a full random pattern.
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__global__ void k_selftest_convert(uint64_t seed, long long n, unsigned long long* bad) {
  unsigned long long b0 = 0, b1 = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const uint64_t r = splitmix64(seed + (uint64_t)i), q = splitmix64(r);
    const float f = __uint_as_float((unsigned)r);
    const double a = f2d(f), b = (double)f;
    if (!(isnan(a) && isnan(b)) && __double_as_longlong(a) != __double_as_longlong(b)) ++b0;
    uint64_t bits;
    if ((i & 7) == 7) {
      bits = q;
    } else {
      const uint64_t e = 860u + (q >> 52) % 310u;  // float underflow .. overflow
      uint64_t m = q & 0xfffffffffffffull;
      if ((i & 3) == 0) m = (m & ~0x1fffffffull) | 0x10000000ull;  // exact tie
      bits = ((r >> 63) << 63) | (e << 52) | m;
    }
    const double d = __longlong_as_double((long long)bits);
    const float x = d2f(d), y = __double2float_rn(d);
    if (!(isnan(x) && isnan(y)) && __float_as_uint(x) != __float_as_uint(y)) ++b1;
  }
  if (b0) atomicAdd(bad, b0);
  if (b1) atomicAdd(bad + 1, b1);
}

// Distance in units in the last place of b (at least the spacing of the
// smallest normal, so exact zeros compare by absolute error).
__device__ __forceinline__ double ulps(double a, double b) {
  const double fb = fabs(b);
  const double up = __longlong_as_double(__double_as_longlong(fb) + 1);  // the next double above |b|
  const double u = fmax(up - fb, 2.2250738585072014e-308);
  return fabs(a - b) / u;
}
// The table-driven ln and sincospi of the FP64 Box-Muller (philox.cuh)
// against CUDA's log and sincospi on n uniforms (k + 1/2) 2^-52: k over its
// whole range, its smallest values, and values next to 2^52; the largest
// distances in ulp (rounded up) into worst[0] (ln) and worst[1] (sin, cos).
__global__ void k_selftest_box_muller(uint64_t seed, long long n, unsigned long long* worst) {
  double w0 = 0.0, w1 = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const uint64_t r = splitmix64(seed + (uint64_t)i);
    uint64_t k = r >> 12;                                        // 52 bits
    if ((i & 15) == 1) k >>= (r & 63) % 52;                      // small k: deep tail of ln
    if ((i & 15) == 2) k = ((1ull << 52) - 1) - (k >> 30);       // u next to 1
    if ((i & 15) == 3) k = (k >> 45) << 45 | ((r & 1) ? 0 : (1ull << 45) - 1);  // next to the sin grid
    const double u = u52_bits(k);
    w0 = fmax(w0, ulps(ln_unit(u), log(u)));
    double s, c, s0, c0;
    sincospi_2u52(k, &s, &c);
    sincospi(2.0 * u, &s0, &c0);
    w1 = fmax(w1, fmax(ulps(s, s0), ulps(c, c0)));
  }
  atomicMax(worst, (unsigned long long)ceil(w0));
  atomicMax(worst + 1, (unsigned long long)ceil(w1));
}

}  // namespace

// ------------------------------------------------------------ fused batch
// The cooling kernels of a fused batch: one launch over the blocks of every
// listed chain, each block running the body of the chain's own kernel with
// the chain's geometry, buffers and rule state (see ensemble.cuh).  Cooling
// follows the step's update, which wrote the chain's Un: that is the link
// field these kernels cool (the runtime swaps U and Un after the step).
namespace {

__device__ __forceinline__ Geo ens_geo(const ChainDesc& c) {
  Geo g;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    g.L[mu] = c.L[mu];
    g.stride[mu] = c.stride[mu];
  }
  g.V = c.V;
  return g;
}
template <typename L>
__device__ __forceinline__ SweepArgs ens_sweep(const ChainDesc& c) {
  // the step's new links; fixed point: their words in the old links' buffer
  return SweepArgs{c.Un, is_fx<L>() ? c.U : c.Un, (double*)c.f, c.Om, c.Omi, (double2*)c.arec, &c.sd->pad, c.cs, c.ca};
}
template <typename L, bool FIRST>
__global__ void __launch_bounds__(CS_THREADS) k_ens_cool_grad(const ChainDesc* __restrict__ cd, const WorkItem* __restrict__ w) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  sweep_grad_body<L, FIRST, cs_wide_grad<L>()>(ens_geo(c), ens_sweep<L>(c), it.vb, true);
}
template <typename L>
__global__ void __launch_bounds__(CS_THREADS) k_ens_cool_omega(const ChainDesc* __restrict__ cd, const WorkItem* __restrict__ w) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  sweep_omega_body<L, false>(ens_geo(c), ens_sweep<L>(c), it.vb);
}
template <typename L>
__global__ void __launch_bounds__(CS_THREADS) k_ens_cool_grad_omega(const ChainDesc* __restrict__ cd,
                                                                   const WorkItem* __restrict__ w) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  sweep_grad_omega_body<L, cs_wide_omega<L>()>(ens_geo(c), ens_sweep<L>(c), it.vb);
}
// sweep: which of the call's sweeps this launch is (each chain has its own last one)
template <typename L, bool RULE>
__global__ void __launch_bounds__(CS_THREADS, CS_APPLY_BLOCKS(L)) k_ens_cool_apply(const ChainDesc* __restrict__ cd,
                                                                  const WorkItem* __restrict__ w, int sweep) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  sweep_apply<L, RULE, true>(ens_geo(c), ens_sweep<L>(c), it.vb, sweep == cs_sweeps(c.ca) - 1);
}

template <typename L>
cudaError_t launch_ens_cool_family(int fam, const ChainDesc* cd, const WorkItem* w, int nw, int arg, cudaStream_t st) {
  const unsigned n = (unsigned)nw;
  switch (fam) {
    case ENS_COOL_GRAD:
      if (arg)
        k_ens_cool_grad<L, true><<<n, CS_THREADS, 0, st>>>(cd, w);
      else
        k_ens_cool_grad<L, false><<<n, CS_THREADS, 0, st>>>(cd, w);
      break;
    case ENS_COOL_OMEGA: k_ens_cool_omega<L><<<n, CS_THREADS, 0, st>>>(cd, w); break;
    case ENS_COOL_APPLY: k_ens_cool_apply<L, false><<<n, CS_THREADS, 0, st>>>(cd, w, arg); break;
    case ENS_COOL_GRAD_OMEGA: k_ens_cool_grad_omega<L><<<n, CS_THREADS, 0, st>>>(cd, w); break;
    case ENS_COOL_APPLY_UN: k_ens_cool_apply<L, true><<<n, CS_THREADS, 0, st>>>(cd, w, arg); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ens_step_f64(int fam, const ChainDesc* cd, const WorkItem* w, int nw, cudaStream_t st);
cudaError_t launch_ens_step_f32(int fam, const ChainDesc* cd, const WorkItem* w, int nw, cudaStream_t st);

cudaError_t launch_ens(int prec, int fam, const ChainDesc* cd, const WorkItem* w, int nw, int arg, cudaStream_t st) {
  if (nw <= 0) return cudaSuccess;
  if (prec != 0 && prec != 1) return cudaErrorInvalidValue;
  if (fam < ENS_COOL_GRAD)
    return prec == 0 ? launch_ens_step_f64(fam, cd, w, nw, st) : launch_ens_step_f32(fam, cd, w, nw, st);
  return prec == 0 ? launch_ens_cool_family<double>(fam, cd, w, nw, arg, st)
                   : launch_ens_cool_family<float>(fam, cd, w, nw, arg, st);
}

cudaError_t launch_selftest_convert(uint64_t seed, long long n, unsigned long long* bad, cudaStream_t st) {
  k_selftest_convert<<<RED_MAX_BLOCKS, RED_THREADS, 0, st>>>(seed, n, bad);
  return cudaGetLastError();
}

cudaError_t launch_selftest_box_muller(uint64_t seed, long long n, unsigned long long* worst, cudaStream_t st) {
  k_selftest_box_muller<<<RED_MAX_BLOCKS, RED_THREADS, 0, st>>>(seed, n, worst);
  return cudaGetLastError();
}

// Reduction kernels loop over sites with at most RED_MAX_BLOCKS blocks, so
// the one-block rule reads few records; the split depends on V only.
// Launch with the link type of precision prec (0 FP64, 1 FP32 storage, 2 DF64).
template <typename Fn>
cudaError_t by_prec(int prec, Fn fn) {
  if (prec == 0) fn(double());
  else if (prec == 1) fn(float());
  else fn(df64());
  return cudaGetLastError();
}

int reduce_blocks(int V) {
  int b = (V + RED_THREADS - 1) / RED_THREADS;
  return b < RED_MAX_BLOCKS ? b : RED_MAX_BLOCKS;
}

cudaError_t launch_cold(int prec, const GeoH& h, void* U, cudaStream_t st) {
  Geo g = to_geo(h);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_cold<T><<<grid_sites(g.V, 4), RED_THREADS, 0, st>>>(g, (typename vec2_of<T>::type*)U);
  });
}

cudaError_t launch_hot(int prec, const GeoH& h, void* U, uint64_t seed, cudaStream_t st) {
  Geo g = to_geo(h);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_hot<T><<<grid_sites(g.V, 4), RED_THREADS, 0, st>>>(g, (typename vec2_of<T>::type*)U, seed);
  });
}

cudaError_t launch_gauge_omega(int prec, const GeoH& h, void* Om, void* Omi, uint64_t seed,
                               double sigma, cudaStream_t st) {
  Geo g = to_geo(h);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_gauge_omega<T><<<grid_sites(g.V), RED_THREADS, 0, st>>>(g, (T*)Om, (T*)Omi, seed, sigma);
  });
}

cudaError_t launch_aos_to_soa(int prec, const GeoH& h, const double* aos, void* U, int nplanes,
                              cudaStream_t st) {
  Geo g = to_geo(h);
  if (nplanes < 1 || 9 * nplanes > CONV_MAX_ROWS) return cudaErrorInvalidValue;
  const unsigned blocks = (unsigned)((g.V + CONV_SITES - 1) / CONV_SITES);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_aos_to_soa<T><<<blocks, 256, 0, st>>>(g, aos, (typename vec2_of<T>::type*)U, nplanes);
  });
}

cudaError_t launch_soa_to_aos(int prec, const GeoH& h, const void* U, double* aos, int nplanes,
                              cudaStream_t st) {
  Geo g = to_geo(h);
  if (nplanes < 1 || 9 * nplanes > CONV_MAX_ROWS) return cudaErrorInvalidValue;
  const unsigned blocks = (unsigned)((g.V + CONV_SITES - 1) / CONV_SITES);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_soa_to_aos<T><<<blocks, 256, 0, st>>>(g, (const typename vec2_of<T>::type*)U, aos, nplanes);
  });
}

cudaError_t launch_noise_sample(int prec, int site0, int n, uint64_t seed, uint32_t step, int mu, double* out,
                                cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    k_noise_sample<T><<<(n + 127) / 128, 128, 0, st>>>(site0, n, seed, step, (uint32_t)mu, out);
  });
}

namespace {
SweepArgs sweep_args(const CoolBufs& b) {
  return SweepArgs{b.U, b.Ux, (double*)b.f, b.Om, b.Omi, (double2*)b.rec, &b.sd->pad, b.cs, b.ca};
}
}  // namespace

cudaError_t launch_cool_grad(int prec, const GeoH& h, const CoolBufs& b, bool first, bool rule, cudaStream_t st) {
  Geo g = to_geo(h);
  const SweepArgs a = sweep_args(b);
  const int r = rule ? 1 : 0;
  return by_prec(prec, [&](auto t) {
    using L = decltype(t);
    constexpr int W = cs_wide_grad<L>();
    const int n = cs_grad_blocks<L>(g.V, cs_narrow(g.V) ? 1 : W);
    if (cs_narrow(g.V)) {
      if (first)
        k_cool_grad<L, true, 1><<<n, CS_THREADS, 0, st>>>(g, a, r);
      else
        k_cool_grad<L, false, 1><<<n, CS_THREADS, 0, st>>>(g, a, r);
    } else {
      if (first)
        k_cool_grad<L, true, W><<<n, CS_THREADS, 0, st>>>(g, a, r);
      else
        k_cool_grad<L, false, W><<<n, CS_THREADS, 0, st>>>(g, a, r);
    }
  });
}
cudaError_t launch_cool_omega(int prec, const GeoH& h, const CoolBufs& b, cudaStream_t st) {
  Geo g = to_geo(h);
  const SweepArgs a = sweep_args(b);
  return by_prec(prec, [&](auto t) {
    using L = decltype(t);
    const int n = cs_omega_blocks(g.V, cs_narrow(g.V));
    if (cs_narrow(g.V))
      k_cool_omega<L, true><<<n, CS_THREADS, 0, st>>>(g, a);
    else
      k_cool_omega<L, false><<<n, CS_THREADS, 0, st>>>(g, a);
  });
}
cudaError_t launch_cool_grad_omega(int prec, const GeoH& h, const CoolBufs& b, cudaStream_t st) {
  Geo g = to_geo(h);
  const SweepArgs a = sweep_args(b);
  return by_prec(prec, [&](auto t) {
    using L = decltype(t);
    if (cs_narrow(g.V))
      k_cool_grad_omega<L, 1><<<cs_grad_omega_blocks(g.V, 1), CS_THREADS, 0, st>>>(g, a);
    else
      k_cool_grad_omega<L, cs_wide_omega<L>()><<<cs_grad_omega_blocks(g.V, cs_wide_omega<L>()), CS_THREADS, 0, st>>>(g, a);
  });
}
cudaError_t launch_cool_apply(int prec, const GeoH& h, const CoolBufs& b, bool rule, bool last, cudaStream_t st) {
  Geo g = to_geo(h);
  const SweepArgs a = sweep_args(b);
  const int k = last ? 1 : 0;
  return by_prec(prec, [&](auto t) {
    using L = decltype(t);
    const bool wide = is_fx<L>() || !cs_narrow(g.V);  // fixed point: one shape
    const int n = cs_apply_blocks<L>(g.V, wide ? 4 : 1);
    if (wide) {
      if (rule)
        k_cool_apply<L, true, true><<<n, CS_THREADS, 0, st>>>(g, a, k);
      else
        k_cool_apply<L, false, true><<<n, CS_THREADS, 0, st>>>(g, a, k);
    } else if constexpr (!is_fx<L>()) {
      if (rule)
        k_cool_apply<L, true, false><<<n, CS_THREADS, 0, st>>>(g, a, k);
      else
        k_cool_apply<L, false, false><<<n, CS_THREADS, 0, st>>>(g, a, k);
    }
  });
}
cudaError_t launch_cool_load(int prec, const GeoH& h, const void* U, void* Ux, cudaStream_t st) {
  Geo g = to_geo(h);
  const int n = cs_groups(g.V);
  if (prec == 0) k_cool_load<double><<<n, CS_THREADS, 0, st>>>(g, (const double2*)U, (int4*)Ux);
  if (prec == 2) k_cool_load<df64><<<n, CS_THREADS, 0, st>>>(g, (const float4*)U, (int4*)Ux);
  return cudaGetLastError();
}
int ens_cool_blocks(int prec, int fam, int V) {
  switch (fam) {
    case ENS_COOL_GRAD:
      return prec == 0 ? cs_grad_blocks<double>(V, cs_wide_grad<double>()) : cs_grad_blocks<float>(V, cs_wide_grad<float>());
    case ENS_COOL_OMEGA: return cs_omega_blocks(V, false);
    case ENS_COOL_GRAD_OMEGA: return cs_grad_omega_blocks(V, prec == 0 ? cs_wide_omega<double>() : cs_wide_omega<float>());
    default: return prec == 0 ? cs_apply_blocks<double>(V, 4) : cs_apply_blocks<float>(V, 4);
  }
}

cudaError_t launch_obs(int prec, const GeoH& h, const void* U, const void* Ux, const void* Pq, const void* Dq,
                       const void* F, double* partials, double* q_site, StepDev* sd, cudaStream_t st) {
  Geo g = to_geo(h);
  return by_prec(prec, [&](auto t) {
    using T = decltype(t);
    typedef typename obs_word<T>::type W;
    k_obs<T><<<reduce_blocks(g.V), RED_THREADS, 0, st>>>(g, (const typename vec2_of<T>::type*)U, (const int4*)Ux,
                                                        (const W*)Pq, (const W*)Dq, (const W*)F, partials, q_site, field_top(sd));
  });
}

cudaError_t launch_obs_final(const GeoH& h, const double* partials, double beta, double th_re,
                             double th_im, ObsOut* out, cudaStream_t st) {
  Geo g = to_geo(h);
  k_obs_final<<<1, 256, 0, st>>>(g, partials, reduce_blocks(g.V), beta, th_re, th_im, out);
  return cudaGetLastError();
}

}  // namespace clgc
