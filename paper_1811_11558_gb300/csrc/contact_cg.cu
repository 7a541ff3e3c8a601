// Fused kernels of the Polonsky-Keer contact iteration (Sec. 5.1) on power-of-two surfaces with
// both sides from 16 to 1024: six kernels per iteration.
//
// An iteration is a chain of global sums (mean gap and G, tau, total load), each of which the next
// elementwise step needs, and two surface convolutions u = K*p, r = K*t.  Each elementwise step
// runs inside the row pass of the convolution next to it:
//   rowsT  g = u - h - gbar; t = g + beta t on the contact, 0 elsewhere; forward rows of t
//   cols   columns: transform, surface compliance, inverse
//   rowsR  inverse rows of r = K*t, kept in registers; sums of r, t, g t and r t over the contact
//          -> tau = <g, t> / (<r, t> - rbar <t, 1>)
//   rowsP  p <- max(p - tau t, 0), points that would penetrate re-enter; sum p -> load scale s;
//          forward rows of the unscaled p
//   cols   as above, times s (the transform is linear)
//   rowsU  inverse rows of u = K*p; p <- s p, change against the old pressure -> stop test; over
//          the contact sums of d and d^2, d = u - h - (last gbar) -> gbar, G = sum of g^2 -> beta
// (d is the gap up to the change of its mean, so G = sum d^2 - (sum d)^2 / n cancels nothing that
// the iteration does not itself lose; the first G is summed from g.)  The sums are FP64, block
// partials in block order added by the last block to finish, so results do not depend on timing.
// Every scalar, the surface and pressure pointers, the load and the tolerance live in the device
// state (PkState): one captured loop serves every call of a context.
//
// What bounds it: an FP64 instruction holds its pipe for 64 cycles per warp here (a conversion
// counts as one), so a kernel's time is its FP64 instructions per warp and the dependent chain of
// its sums.  So: four complex values per thread (more warps with less each); elementwise FP32
// updates in two-float arithmetic, rounded once as the FP64 expression is; FP64 only in the sums,
// and there only at points that carry pressure; a warp's sums of several values reduced together.
// us per iteration, fourteen kernels -> seven with eight values per thread and FP64 updates -> this:
// 32^2 FP64 100 -> 97 -> 56, 32^2 FP32 62 -> 63 -> 41, 512^2 132 -> 75 -> 56, 1024^2 206 -> 156 -> 112.
#include <algorithm>

#include "fvim_internal.cuh"

namespace {

enum { FWD_INIT = 0, FWD_P, FWD_T };
enum { INV_U0 = 0, INV_U, INV_R };

// ---- elementwise updates with FP64 scalars, rounded once to the path's precision ------------
// FP32: the scalar as a float pair, products and sums as exact pairs (to about 2^-46 of the result
// before its one rounding)
__device__ __forceinline__ float2 pair_of(double x) {
  const float h = (float)x;
  return make_float2(h, isfinite(h) ? (float)(x - (double)h) : 0.f);
}
// a + k x
__device__ __forceinline__ float axpy1(float a, double, float2 k, float x) {
  const float p = __fmul_rn(k.x, x), pl = __fmaf_rn(k.x, x, -p);
  const float s = __fadd_rn(a, p), e = two_sum_err(a, p, s);
  return __fadd_rn(s, __fadd_rn(e, __fmaf_rn(k.y, x, pl)));
}
__device__ __forceinline__ double axpy1(double a, double k, float2, double x) { return a + k * x; }
// k x
__device__ __forceinline__ float mul1(double, float2 k, float x) {
  const float p = __fmul_rn(k.x, x);
  return __fadd_rn(p, __fmaf_rn(k.y, x, __fmaf_rn(k.x, x, -p)));
}
__device__ __forceinline__ double mul1(double k, float2, double x) { return k * x; }
// u - h - c
__device__ __forceinline__ float gap1(float u, float h, double, float2 c) {
  const float d = __fsub_rn(u, h), e = two_sum_err(u, -h, d);
  const float s = __fsub_rn(d, c.x), e2 = two_sum_err(d, -c.x, s);
  return __fadd_rn(s, __fadd_rn(e2, __fsub_rn(e, c.y)));
}
__device__ __forceinline__ double gap1(double u, double h, double c, float2) { return u - h - c; }

// state of a new solve, with the scale of the initial pressure from its sum (a guess without load
// is replaced by the uniform pressure)
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_begin(PkState* S, const T* __restrict__ p, size_t n, PkState init, double* part,
                                                   unsigned* cnt) {
  double v[4] = {0, 0, 0, 0};
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) v[0] += (double)p[i];
  if (grid_sum(v, part, cnt)) {
    init.start = v[0] > 0 ? init.W / (init.dA * v[0]) : 0.0;
    *S = init;
  }
}
// surface compliance u3_hat / p_hat = (1 - nu) / (mu q) of every mode, 0 for mode 0 and the Nyquist row
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_green(T* __restrict__ green, int h1, int n2, T w1, T w2, T nu, T mu) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= h1 * n2) return;
  const int k2 = i / h1, k1 = i - k2 * h1;
  const T q1 = w1 * (T)k1;
  const T q2 = w2 * (T)(k2 < n2 / 2 ? k2 : k2 - n2);
  const T q = sqrt(q1 * q1 + q2 * q2);
  green[i] = i == 0 || k2 == n2 / 2 ? (T)0 : ((T)1 - nu) / (mu * q);
}

// Forward rows of p or t, two rows per transform, N / 4 threads per transform, blockDim.x / (N / 4)
// transforms per CTA; the half spectrum k1 < N/2 goes to surf (the Nyquist column carries no
// operator term).
template <typename T, int N, int MODE>
__global__ void __launch_bounds__(512) k_pkf_rows_fwd(PkState* S, const T* __restrict__ u, T* __restrict__ g,
                                                      T* __restrict__ t, T* __restrict__ pold,
                                                      typename Cx<T>::t* __restrict__ surf,
                                                      const typename Cx<T>::t* __restrict__ tw, int n2, double* part,
                                                      unsigned* cnt) {
  typedef typename Cx<T>::t V;
  if (MODE != FWD_INIT && S->done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, tt = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const T* h = static_cast<const T*>(S->h);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  const double start = S->start, unif = S->unif, tau = S->tau, gbar = S->gbar, beta = S->beta;
  const float2 tau2 = S->tau2, gbar2 = S->gbar2, beta2 = S->beta2;
  V v[4];
  double sum[4] = {0, 0, 0, 0};
  int nol = 0;
  auto value = [&](size_t i) -> T {
    if constexpr (MODE == FWD_INIT) {
      const T x = start > 0 ? (T)(start * (double)p[i]) : (T)unif;
      p[i] = x;
      t[i] = (T)0;
      return x;
    } else if constexpr (MODE == FWD_P) {
      const T po = p[i], ti = t[i], gi = g[i];
      T pn = (T)0;
      if (po != (T)0 || ti != (T)0) {
        const T x = axpy1(po, -tau, make_float2(-tau2.x, -tau2.y), ti);
        pn = x > (T)0 ? x : (T)0;
      }
      if (pn == (T)0 && gi < (T)0) {
        pn = mul1(-tau, make_float2(-tau2.x, -tau2.y), gi);
        ++nol;
      }
      pold[i] = po;
      p[i] = pn;
      if (pn != (T)0) sum[0] += (double)pn;
      return pn;
    } else {
      const T gi = gap1(u[i], h[i], gbar, gbar2);
      g[i] = gi;
      const T x = p[i] > (T)0 ? axpy1(gi, beta, beta2, t[i]) : (T)0;
      t[i] = x;
      return x;
    }
  };
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[m] = mk<V>(0, 0);
    if (live) {
      const size_t i = i0 + m * T4;
      v[m].x = value(i);
      v[m].y = value(i + N);
    }
  }
  SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft4_ct<V, false, N, 1>(v, tt, sm, tw);
  // separation of the two rows: Z(N - k) of k = tt + m N/4, m < 2, is in another thread's upper half
  sm.put(tt + 2 * T4, v[2]);
  sm.put(tt + 3 * T4, v[3]);
  __syncthreads();
  if (live) {
    V* o = surf + (size_t)2 * pair * H1 + tt;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      V zm = sm.get((N - tt - m * T4) & (N - 1));
      if (m == 0 && tt == 0) zm = v[0];
      const V c = cconj(zm), a = cadd(v[m], c), d = csub(v[m], c);
      o[m * T4] = cscale(a, (T)0.5);
      o[H1 + m * T4] = mk<V>((T)0.5 * d.y, (T)-0.5 * d.x);
    }
  }
  if (MODE == FWD_P) {
    sum[1] = (double)nol;
    if (grid_sum(sum, part, cnt)) {
      S->delta = sum[1] > 0 ? 0.0 : 1.0;
      if (!(sum[0] > 0) || !isfinite(sum[0])) {
        S->bad = 1;
        S->done = 1;
      } else {
        const double x = S->W / (S->dA * sum[0]);
        S->s = x;
        S->s2 = pair_of(x);
      }
    }
  }
}

// Columns: forward transform of kc k1 columns, surface compliance, times the load scale for the
// pressure, inverse transform.  Few columns per CTA (32-byte row segments): the plane stays in L2,
// and 512 points in 16-column CTAs would leave most of the chip idle.
template <typename T, int N, bool SCALE>
__global__ void __launch_bounds__(512) k_pkf_cols(const PkState* S, typename Cx<T>::t* __restrict__ plane,
                                                  const T* __restrict__ green, const typename Cx<T>::t* __restrict__ tw,
                                                  int h1, int kc) {
  typedef typename Cx<T>::t V;
  if (S->done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4;
  const int f = threadIdx.x % kc, t = threadIdx.x / kc;
  const size_t at = (size_t)blockIdx.x * kc + f;
  V* col = plane + at;
  V v[4];
  const double scl = SCALE ? S->s : 1.0;
  const float2 scl2 = S->s2;
  T f0[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[m] = col[(size_t)(t + m * T4) * h1];
    f0[m] = green[(size_t)(t + m * T4) * h1 + at];
  }
  const SurfColSm<V> sm{reinterpret_cast<V*>(smraw), kc, f};
  fft4_ct<V, false, N, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = cscale(v[m], SCALE ? mul1(scl, scl2, f0[m]) : f0[m]);
  fft4_ct<V, true, N, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 4; ++m) col[(size_t)(t + m * T4) * h1] = v[m];
}

// Inverse rows of u or r (two rows per transform) with the elementwise step and sums that follow.
template <typename T, int N, int MODE>
__global__ void __launch_bounds__(512) k_pkf_rows_inv(PkState* S, const T* __restrict__ g, const T* __restrict__ t,
                                                      const T* __restrict__ pold, T* __restrict__ u,
                                                      const typename Cx<T>::t* __restrict__ surf,
                                                      const typename Cx<T>::t* __restrict__ tw, int n2, T scale, double* part,
                                                      unsigned* cnt, cudaGraphConditionalHandle cond, int use_cond) {
  typedef typename Cx<T>::t V;
  if (S->done) {
    if (MODE == INV_U && use_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0u);
    return;
  }
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, tt = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const T* h = static_cast<const T*>(S->h);
  V v[4];
  const V* sa = surf + (size_t)(live ? 2 * pair : 0) * H1;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int k = tt + m * T4;
    const int kk = k < H1 ? k : (k > H1 ? N - k : 0);
    V A = sa[kk], B = sa[H1 + kk];
    if (k > H1) { A = cconj(A); B = cconj(B); }
    if (k == H1) A = B = mk<V>(0, 0);
    v[m] = cadd(A, cmuli(B));
  }
  const SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft4_ct<V, true, N, 1>(v, tt, sm, tw);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  const double scl = S->s, gbar = S->gbar;
  const float2 scl2 = S->s2;
  double sum[4] = {0, 0, 0, 0};
  int nc = 0;
  auto add = [&](size_t i, T x) {
    if constexpr (MODE == INV_R) {
      if (p[i] > (T)0) {
        const double xi = (double)x, ti = (double)t[i];
        sum[0] += xi;
        sum[1] += ti;
        sum[2] += (double)g[i] * ti;
        sum[3] += xi * ti;
      }
    } else {
      T pi = p[i];
      if constexpr (MODE == INV_U) {
        const T po = pold[i];
        if (pi != (T)0) {
          pi = mul1(scl, scl2, pi);
          p[i] = pi;
        }
        if (pi != po) sum[2] += fabs((double)pi - (double)po);
      }
      u[i] = x;
      if (pi > (T)0) {
        const double d = MODE == INV_U ? (double)x - (double)h[i] - gbar : (double)x - (double)h[i];
        sum[0] += d;
        if (MODE == INV_U) sum[1] += d * d;
        ++nc;
      }
    }
  };
  if (live) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      add(i0 + m * T4, v[m].x * scale);
      add(i0 + m * T4 + N, v[m].y * scale);
    }
  }
  if (MODE != INV_R) sum[3] = (double)nc;
  if (!grid_sum(sum, part, cnt)) return;
  if (MODE == INV_R) {
    // <g, t> / (<r, t> - rbar <t, 1>), rbar = sum r / nIc
    const double den = sum[3] * S->nIc - sum[0] * sum[1];
    const double tau = den != 0 ? sum[2] * S->nIc / den : 0.0;
    S->tau = tau;
    S->tau2 = pair_of(tau);
    return;
  }
  int done = 0, bad = 0;
  if (MODE == INV_U) {
    const double err = sum[2] * S->dA_W;
    S->err = err;
    S->it += 1;
    if (err < S->tol || S->it >= S->max_it) done = 1;
    if (!isfinite(err)) bad = 1;
  }
  S->nIc = sum[3];
  if (!done && (!(sum[3] > 0) || !isfinite(sum[0]))) {
    bad = 1;
  } else {
    const double mean = sum[0] / sum[3], gb = (MODE == INV_U ? gbar : 0.0) + mean;
    S->gbar = gb;
    S->gbar2 = pair_of(gb);
    if (MODE == INV_U) {
      // (a gap that vanishes to the last bit restarts the direction)
      const double G = fmax(sum[1] - sum[0] * mean, 0.0), beta = S->G_old > 0 ? S->delta * (G / S->G_old) : 0.0;
      S->beta = beta;
      S->beta2 = pair_of(beta);
      S->G_old = G;
    }
  }
  if (bad) S->bad = 1;
  S->done = done | bad;
  if (MODE == INV_U && use_cond) cudaGraphSetConditional(cond, (done | bad) ? 0u : 1u);
}

// G = sum over the contact of g^2, g = u - h - gbar, of the first iteration
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_gap(PkState* S, const T* __restrict__ u, size_t n, double* part, unsigned* cnt) {
  if (S->done) return;
  const double gbar = S->gbar;
  const T* h = static_cast<const T*>(S->h);
  const T* p = static_cast<const T*>(S->p);
  double v[4] = {0, 0, 0, 0};
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (p[i] > (T)0) {
      const double gi = (double)u[i] - (double)h[i] - gbar;
      v[0] += gi * gi;
    }
  }
  if (grid_sum(v, part, cnt)) S->G_old = v[0];
}

template <typename T, int N, int MODE> void rows_fwd(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  const SurfRowCfg r = surf_row_cfg<T, N>(a.n2);
  surf_row_smem_cap(k_pkf_rows_fwd<T, N, MODE>);
  k_pkf_rows_fwd<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(a.S, (const T*)a.u, (T*)a.g, (T*)a.t, (T*)a.pold,
                                                                   (V*)a.surf, (const V*)a.tw1, a.n2, a.part, a.cnt);
}
template <typename T, int N, int MODE> void rows_inv(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  const SurfRowCfg r = surf_row_cfg<T, N>(a.n2);
  surf_row_smem_cap(k_pkf_rows_inv<T, N, MODE>);
  k_pkf_rows_inv<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(
      a.S, (const T*)a.g, (const T*)a.t, (const T*)a.pold, (T*)a.u, (const V*)a.surf, (const V*)a.tw1, a.n2,
      (T)(1.0 / ((double)N * (double)a.n2)), a.part, a.cnt, a.cond, a.use_cond);
}
template <typename T, int N, bool SCALE> void cols(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  int kc = (int)(32 / sizeof(V));
  if (kc > a.h1) kc = a.h1;
  while (kc * (N / 4) > 512) kc >>= 1;
  smem_cap(k_pkf_cols<T, N, SCALE>);
  k_pkf_cols<T, N, SCALE><<<a.h1 / kc, kc * (N / 4), (size_t)kc * N * sizeof(V), a.stream>>>(
      a.S, (V*)a.surf, (const T*)a.green, (const V*)a.tw2, a.h1, kc);
}

#define PKF_SIZES(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)
template <typename T, int MODE> void rows_fwd_any(const PkfArgs& a) {
#define CASE(N) if (a.n1 == N) rows_fwd<T, N, MODE>(a);
  PKF_SIZES(CASE)
#undef CASE
}
template <typename T, int MODE> void rows_inv_any(const PkfArgs& a) {
#define CASE(N) if (a.n1 == N) rows_inv<T, N, MODE>(a);
  PKF_SIZES(CASE)
#undef CASE
}
template <typename T, bool SCALE> void cols_any(const PkfArgs& a) {
#define CASE(N) if (a.n2 == N) cols<T, N, SCALE>(a);
  PKF_SIZES(CASE)
#undef CASE
}
inline int flat_grid(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 256); }

}  // namespace

bool pkf_available(const fvim_ctx* c) { return !c->gen && c->n1 >= 16 && c->n2 >= 16; }

template <typename T> int pkf_begin(const PkfArgs& a, const PkState& init) {
  const size_t n = (size_t)a.n1 * a.n2;
  k_pkf_begin<T><<<flat_grid(n), 256, 0, a.stream>>>(a.S, (const T*)init.p, n, init, a.part, a.cnt);
  const double two_pi = 6.283185307179586476925;
  k_pkf_green<T><<<(a.h1 * a.n2 + 255) / 256, 256, 0, a.stream>>>((T*)a.green, a.h1, a.n2, (T)(two_pi / a.L1),
                                                                  (T)(two_pi / a.L2), (T)a.nu, (T)a.mu);
  rows_fwd_any<T, FWD_INIT>(a);
  cols_any<T, false>(a);
  rows_inv_any<T, INV_U0>(a);
  k_pkf_gap<T><<<flat_grid(n), 256, 0, a.stream>>>(a.S, (const T*)a.u, n, a.part, a.cnt);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template <typename T> int pkf_iteration(const PkfArgs& a) {
  rows_fwd_any<T, FWD_T>(a);
  cols_any<T, false>(a);
  rows_inv_any<T, INV_R>(a);
  rows_fwd_any<T, FWD_P>(a);
  cols_any<T, true>(a);
  rows_inv_any<T, INV_U>(a);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template int pkf_begin<float>(const PkfArgs&, const PkState&);
template int pkf_begin<double>(const PkfArgs&, const PkState&);
template int pkf_iteration<float>(const PkfArgs&);
template int pkf_iteration<double>(const PkfArgs&);
