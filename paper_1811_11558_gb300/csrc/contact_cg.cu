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
// the iteration does not itself lose, unless a point whose depth dominated the mean has left the
// contact: then the last block sums both again, gap_lost; the first G is summed from g.)  The sums are FP64, block
// partials in block order added by the last block to finish, so results do not depend on timing.
// Every scalar, the surface and pressure pointers, the load and the tolerance live in the device
// state (PkState): one captured loop serves every call of a context.
//
// What bounds it: an FP64 instruction holds its pipe for 64 cycles per warp here (a conversion
// counts as one), so a kernel's time is its FP64 instructions per warp and the dependent chain of
// its sums.  So: four complex values per thread (more warps with less each); elementwise FP32
// updates in words of FP32, rounded once as the FP64 expression is; FP64 only in the sums,
// and there only at points that carry pressure; a warp's sums of several values reduced together.
// us per iteration, fourteen kernels -> seven with eight values per thread and FP64 updates -> this
// (with all of a thread's points read before the first store): 256^2 83 -> 46, 512^2 132 -> 75 ->
// 53, 1024^2 206 -> 156 -> 118 (smaller squares: the cluster kernel below).
#include <cooperative_groups.h>

#include <algorithm>

#include "fvim_internal.cuh"

namespace {

enum { FWD_INIT = 0, FWD_P, FWD_T };
enum { INV_U0 = 0, INV_U, INV_R };

// ---- elementwise updates with FP64 scalars, rounded once to the path's precision ------------
// FP32: the scalar's 53 bits in three words and a power of two, products and sums error-free in two
// words, a third for what they leave.  Over 2^21 draws each, the result is the exact value's rounding
// wherever the FP64 expression's is; where a sum cancels to its last bits the FP64 expression is off in
// 3.3e-2 of the draws and this in 2.9e-5 (the scalar in two floats only: 2.1e-1).  A leading sum that is not
// finite is the result: the rounding error taken from it would be a NaN.

// x = (x + y + z) w, the words of a number in [1, 2) with x's sign; integer operations, for an FP64
// conversion holds the pipe as long as an addition
__device__ __forceinline__ float4 words_of(double x) {
  const long long u = __double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  const float one = u < 0 ? -1.f : 1.f;
  if (ex > 1023 - 126 && ex < 1023 + 127) {
    const long long m = (u & 0xfffffffffffffll) | 0x10000000000000ll;
    return make_float4(one * (float)(int)(m >> 29) * 0x1p-23f, one * (float)((int)(m >> 5) & 0xffffff) * 0x1p-47f,
                       one * (float)((int)m & 31) * 0x1p-52f, __int_as_float((ex - 1023 + 127) << 23));
  }
  if (x == 0) return make_float4(0.f, 0.f, 0.f, 1.f);
  // beyond FP32's exponents (or not finite): the nearest scale, the largest value where that is too little
  const float w = ex < 1023 ? 0x1p-126f : 0x1p127f;
  const double r = ex < 1023 ? x * 0x1p126 : x * 0x1p-127;
  float a = (float)r;
  if (isinf(a) && ex != 0x7ff) a = one * 3.402823466e+38f;
  return make_float4(a, 0.f, 0.f, w);
}
__device__ __forceinline__ float4 words_neg(float4 k) { return make_float4(-k.x, -k.y, -k.z, k.w); }
// s + (t + lo) rounded once
__device__ __forceinline__ float three_sum(float s, float t, float lo) {
  const float r = __fadd_rn(s, t), v = __fadd_rn(r, __fadd_rn(two_sum_err(s, t, r), lo));
  return isfinite(s) ? v : s;
}
// a + k x
__device__ __forceinline__ float axpy1(float a, double, float4 k, float x) {
  x = __fmul_rn(x, k.w);
  const float p = __fmul_rn(k.x, x), pl = __fmaf_rn(k.x, x, -p), q = __fmul_rn(k.y, x);
  const float r = __fmaf_rn(k.z, x, __fmaf_rn(k.y, x, -q));
  const float s = __fadd_rn(a, p), e = two_sum_err(a, p, s), t = __fadd_rn(e, pl), u = __fadd_rn(t, q);
  return three_sum(s, u, __fadd_rn(__fadd_rn(two_sum_err(e, pl, t), two_sum_err(t, q, u)), r));
}
__device__ __forceinline__ double axpy1(double a, double k, float4, double x) { return a + k * x; }
// k x
__device__ __forceinline__ float mul1(double, float4 k, float x) {
  x = __fmul_rn(x, k.w);
  const float p = __fmul_rn(k.x, x), pl = __fmaf_rn(k.x, x, -p), q = __fmul_rn(k.y, x);
  const float r = __fmaf_rn(k.z, x, __fmaf_rn(k.y, x, -q)), t = __fadd_rn(pl, q);
  return three_sum(p, t, __fadd_rn(two_sum_err(pl, q, t), r));
}
__device__ __forceinline__ double mul1(double k, float4, double x) { return k * x; }
// u - h - c
__device__ __forceinline__ float gap1(float u, float h, double, float4 c) {
  const float d = __fsub_rn(u, h), e = two_sum_err(u, -h, d), c0 = c.x * c.w, c1 = c.y * c.w, c2 = c.z * c.w;
  const float s = __fsub_rn(d, c0), e2 = two_sum_err(d, -c0, s), t = __fadd_rn(e2, e), v = __fsub_rn(t, c1);
  return three_sum(s, v, __fsub_rn(__fadd_rn(two_sum_err(e2, e, t), two_sum_err(t, -c1, v)), c2));
}
__device__ __forceinline__ double gap1(double u, double h, double c, float4) { return u - h - c; }

// Whether sums about the mean gap c have lost the new mean gb and G = sum g^2 over n points: c is far
// above everything that is left (a point whose depth dominated the mean has gone out of contact).
// Then both are summed again from the gaps themselves.
__device__ __forceinline__ bool gap_lost(double c, double gb, double G, double n) {
  return fabs(c) > 1e3 * (fabs(gb) + sqrt(G / n));
}

// state of a new solve, with the scale of the initial pressure from its sum (a guess without load
// is replaced by the uniform pressure, scale -1; one of infinite load scales to nothing, and the empty
// contact that leaves is refused)
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_begin(PkState* S, const T* __restrict__ p, size_t n, PkState init, double* part,
                                                   unsigned* cnt) {
  double v[4] = {0, 0, 0, 0};
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) v[0] += (double)p[i];
  if (grid_sum(v, part, cnt)) {
    init.start = v[0] > 0 ? init.W / (init.dA * v[0]) : -1.0;
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
  if (MODE == FWD_T && blockIdx.x == 0 && threadIdx.x == 0) S->passes += 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, tt = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const T* h = static_cast<const T*>(S->h);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  const double start = S->start, unif = S->unif, tau = S->tau, gbar = S->gbar, beta = S->beta;
  const float4 tauw = S->tauw, gbarw = S->gbarw, betaw = S->betaw;
  V v[4];
  double sum[4] = {0, 0, 0, 0};
  int nol = 0;
  // the thread's eight points (four places in two rows), read together before anything is stored: with
  // loads and stores in turn each point waited for memory by itself
  auto at = [&](int e) { return i0 + (size_t)(e >> 1) * T4 + (size_t)(e & 1) * N; };
  T a[8], b[8], c[8], d[8], x[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    a[e] = b[e] = c[e] = d[e] = x[e] = (T)0;
    if (live) {
      a[e] = p[at(e)];
      if (MODE != FWD_INIT) b[e] = t[at(e)];
      if (MODE == FWD_P) c[e] = g[at(e)];
      if (MODE == FWD_T) {
        c[e] = u[at(e)];
        d[e] = h[at(e)];
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (!live) break;
    if constexpr (MODE == FWD_INIT) {
      x[e] = start >= 0 ? (T)(start * (double)a[e]) : (T)unif;
      p[at(e)] = x[e];
      t[at(e)] = (T)0;
    } else if constexpr (MODE == FWD_P) {
      const T po = a[e], gi = c[e];
      T pn = (T)0;
      if (po != (T)0 || b[e] != (T)0) {
        const T y = axpy1(po, -tau, words_neg(tauw), b[e]);
        pn = y > (T)0 ? y : (T)0;
      }
      if (pn == (T)0 && gi < (T)0) {
        pn = mul1(-tau, words_neg(tauw), gi);
        ++nol;
      }
      pold[at(e)] = po;
      p[at(e)] = pn;
      if (pn != (T)0) sum[0] += (double)pn;
      x[e] = pn;
    } else {
      const T gi = gap1(c[e], d[e], gbar, gbarw);
      g[at(e)] = gi;
      x[e] = a[e] > (T)0 ? axpy1(gi, beta, betaw, b[e]) : (T)0;
      t[at(e)] = x[e];
    }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = mk<V>(x[2 * m], x[2 * m + 1]);
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
        S->sw = words_of(x);
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
  const float4 sclw = S->sw;
  T f0[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[m] = col[(size_t)(t + m * T4) * h1];
    f0[m] = green[(size_t)(t + m * T4) * h1 + at];
  }
  const SurfColSm<V> sm{reinterpret_cast<V*>(smraw), kc, f};
  fft4_ct<V, false, N, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = cscale(v[m], SCALE ? mul1(scl, sclw, f0[m]) : f0[m]);
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
  // the pass cap does not wait for the sums: the first block ends the loop there by itself, and the last
  // block never asks for another pass beyond it
  const bool cap = MODE == INV_U && S->passes >= S->max_it;
  if (cap && use_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0u);
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, tt = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const T* h = static_cast<const T*>(S->h);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  auto at = [&](int e) { return i0 + (size_t)(e >> 1) * T4 + (size_t)(e & 1) * N; };
  // what the elementwise step needs at the thread's eight points, in flight during the transform
  T fp[8], fa[8], fb[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    fp[e] = fa[e] = fb[e] = (T)0;
    if (live) {
      fp[e] = p[at(e)];
      fa[e] = MODE == INV_R ? t[at(e)] : h[at(e)];
      if (MODE == INV_R) fb[e] = g[at(e)];
      if (MODE == INV_U) fb[e] = pold[at(e)];
    }
  }
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
  const double scl = S->s, gbar = S->gbar;
  const float4 sclw = S->sw;
  double sum[4] = {0, 0, 0, 0};
  int nc = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (!live) break;
    const T x = ((e & 1) ? v[e >> 1].y : v[e >> 1].x) * scale;
    if constexpr (MODE == INV_R) {
      if (fp[e] > (T)0) {
        const double xi = (double)x, ti = (double)fa[e];
        sum[0] += xi;
        sum[1] += ti;
        sum[2] += (double)fb[e] * ti;
        sum[3] += xi * ti;
      }
    } else {
      T pi = fp[e];
      if constexpr (MODE == INV_U) {
        if (pi != (T)0) {
          pi = mul1(scl, sclw, pi);
          p[at(e)] = pi;
        }
        if (pi != fb[e]) sum[2] += fabs((double)pi - (double)fb[e]);
      }
      u[at(e)] = x;
      if (pi > (T)0) {
        const double d = MODE == INV_U ? (double)x - (double)fa[e] - gbar : (double)x - (double)fa[e];
        sum[0] += d;
        if (MODE == INV_U) sum[1] += d * d;
        ++nc;
      }
    }
  }
  if (MODE != INV_R) sum[3] = (double)nc;
  __shared__ int redo;
  if (MODE == INV_U && threadIdx.x == 0) redo = 0;
  if (MODE == INV_U && blockDim.x == 32) __threadfence();  // (more warps: the barriers of grid_sum before its fence)
  const bool lead = grid_sum(sum, part, cnt);
  if (MODE == INV_U) {
    if (lead) {
      const double mean = sum[0] / sum[3];
      redo = sum[3] > 0 && isfinite(sum[0]) && gap_lost(gbar, gbar + mean, fmax(sum[1] - sum[0] * mean, 0.0), sum[3]);
    }
    __syncthreads();
    if (redo) {  // the last block: every u and p of the pass is in memory
      __shared__ double wsum[32];
      __shared__ double mean;
      double G = 0;
      for (int pass = 0; pass < 2; ++pass) {
        double a = 0;
        for (size_t i = threadIdx.x; i < (size_t)N * n2; i += blockDim.x)
          if (__ldcg(p + i) > (T)0) {
            const double d = (double)__ldcg(u + i) - (double)h[i];
            a += pass == 0 ? d : (d - mean) * (d - mean);
          }
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
          a = 0;
          for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += wsum[w];
          if (pass == 0) mean = a / sum[3];
          else G = a;
        }
        __syncthreads();
      }
      if (lead) {  // as sums about the old mean whose difference is G
        sum[0] = 0;
        sum[1] = G;
        S->gbar = mean;
      }
    }
  }
  if (!lead) return;
  if (MODE == INV_R) {
    // <g, t> / (<r, t> - rbar <t, 1>), rbar = sum r / nIc
    const double den = sum[3] * S->nIc - sum[0] * sum[1];
    const double tau = den != 0 ? sum[2] * S->nIc / den : 0.0;
    S->tau = tau;
    S->tauw = words_of(tau);
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
    const double mean = sum[0] / sum[3], gb = (MODE == INV_U ? (redo ? S->gbar : gbar) : 0.0) + mean;
    S->gbar = gb;
    S->gbarw = words_of(gb);
    if (MODE == INV_U) {
      // (a gap that vanishes to the last bit restarts the direction)
      const double G = fmax(sum[1] - sum[0] * mean, 0.0), beta = S->G_old > 0 ? S->delta * (G / S->G_old) : 0.0;
      S->beta = beta;
      S->betaw = words_of(beta);
      S->G_old = G;
    }
  }
  if (bad) S->bad = 1;
  S->done = done | bad;
  if (MODE == INV_U && use_cond) cudaGraphSetConditional(cond, (done | bad) || cap ? 0u : 1u);
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
  k_pkf_rows_fwd<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(a.S, (const T*)a.u, (T*)a.g, (T*)a.t, (T*)a.pold,
                                                                   (V*)a.surf, (const V*)a.tw1, a.n2, a.part, a.cnt);
}
template <typename T, int N, int MODE> void rows_inv(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  const SurfRowCfg r = surf_row_cfg<T, N>(a.n2);
  k_pkf_rows_inv<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(
      a.S, (const T*)a.g, (const T*)a.t, (const T*)a.pold, (T*)a.u, (const V*)a.surf, (const V*)a.tw1, a.n2,
      (T)(1.0 / ((double)N * (double)a.n2)), a.part, a.cnt, a.cond, a.use_cond);
}
template <typename T, int N, bool SCALE> void cols(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  int kc = (int)(32 / sizeof(V));
  if (kc > a.h1) kc = a.h1;
  while (kc * (N / 4) > 512) kc >>= 1;
  smem_cap(k_pkf_cols<T, N, SCALE>, (size_t)kc * N * sizeof(V));
  k_pkf_cols<T, N, SCALE><<<a.h1 / kc, kc * (N / 4), (size_t)kc * N * sizeof(V), a.stream>>>(
      a.S, (V*)a.surf, (const T*)a.green, (const V*)a.tw2, a.h1, kc);
}

// ---- small square surfaces: the whole solve in one cluster of eight CTAs --------------------
// On 16^2 to 128^2 surfaces an iteration of six kernels is launches and latency (41 us at 32^2
// FP32, 56 us FP64, whatever the work).  Here eight CTAs keep the surface, the iterate and both
// spectra in shared memory: CTA r owns rows [r N/8, (r+1) N/8) and columns [r N/16, (r+1) N/16) of
// the half spectrum, row results go straight to the owners' shared memory (remote stores) and
// back, and sums are exchanged the same way, each CTA adding the eight partials in rank order (the
// same value everywhere, so every decision is the same everywhere).  Six cluster barriers per
// iteration (about 350 cycles each); the loop ends at the stop test or the iteration cap.
// us per iteration, six kernels -> this: FP64 32^2 55 -> 22, 64^2 57 -> 36, FP32 32^2 35 -> 12, 64^2 37 -> 20,
// 128^2 45 -> 31 (256^2 does not fit).
constexpr int CL = 8;

// Stockham stages of radix 2 on two values per thread (FP64: the pipes are idle but for the few
// warps of a transform, so half the work per thread is half the time)
template <typename V, bool INV, int N, int NS, class Sm>
__device__ __forceinline__ void fft2_ct(V (&v)[2], int t, bool on, const Sm& sm, const V* __restrict__ tw) {
  const int k = t & (NS - 1);
  if constexpr (NS > 1) {
    if (on) bf2(v[0], v[1], twiddle<V, INV>(tw, k * (N / (2 * NS))));
  } else {
    const V a = v[0], c = v[1];
    v[0] = cadd(a, c);
    v[1] = csub(a, c);
  }
  if constexpr (2 * NS < N) {
    const int base = (t / NS) * NS * 2 + k;
    if (on) {
      sm.put(base, v[0]);
      sm.put(base + NS, v[1]);
    }
    __syncthreads();
    if (on) {
      v[0] = sm.get(t);
      v[1] = sm.get(t + N / 2);
    }
    __syncthreads();
    fft2_ct<V, INV, N, 2 * NS>(v, t, on, sm, tw);
  }
}

template <typename T, int N> struct ClCfg {
  typedef typename Cx<T>::t V;
  static constexpr int H1 = N / 2, R = N / CL, K = H1 / CL;   // rows and columns of a CTA
  static constexpr int E = R * N;                             // points of a CTA
  static constexpr int BT = E < 64 ? 64 : (E > 512 ? 512 : E);
  static constexpr int VT = (sizeof(T) == 8 && N <= 64) ? 2 : 4;  // values per transform thread
  static constexpr int TT = N / VT;                               // threads per transform
  static constexpr int LD = N + N / 8;
  static constexpr int NT = R / 2 > K ? R / 2 : K;                // transforms at once (R / 2 == K)
  static_assert(R / 2 == K && NT * TT <= BT, "transform threads");
  static constexpr size_t bytes = (size_t)(NT * LD + K * N + R * H1 + N) * sizeof(V) + (size_t)(6 * E + K * N) * sizeof(T);
};

// transform of NT sequences of the CTA by its first NT TT threads; get(f, i) reads, put(f, i, x) takes
// the results (natural order)
template <typename T, int N, bool INV, class G, class P>
__device__ __forceinline__ void cl_fft(typename Cx<T>::t* xch, const typename Cx<T>::t* tw, G&& get, P&& put) {
  typedef typename Cx<T>::t V;
  typedef ClCfg<T, N> C;
  const int f = threadIdx.x / C::TT, t = threadIdx.x % C::TT;
  const bool on = f < C::NT;
  SurfSm<V, N> sm{xch + (size_t)(on ? f : 0) * C::LD};
  V v[C::VT];
#pragma unroll
  for (int m = 0; m < C::VT; ++m) v[m] = on ? get(f, t + m * C::TT) : mk<V>(0, 0);
  if constexpr (C::VT == 2) {
    fft2_ct<V, INV, N, 1>(v, t, on, sm, tw);
  } else {
    // (threads without a transform take part in the barriers; their exchange area is a spare copy)
    fft4_on<V, INV, N, 1>(v, t, on, sm, tw);
  }
#pragma unroll
  for (int m = 0; m < C::VT; ++m)
    if (on) put(f, t + m * C::TT, v[m]);
}

template <typename T, int N>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(ClCfg<T, N>::BT)
    k_pkf_cluster(PkState* out, PkState init, const typename Cx<T>::t* __restrict__ tw_g, T w1, T w2, T nu, T mu) {
  typedef typename Cx<T>::t V;
  typedef ClCfg<T, N> C;
  constexpr int H1 = C::H1, R = C::R, K = C::K, E = C::E;
  namespace cgx = cooperative_groups;
  cgx::cluster_group cl = cgx::this_cluster();
  const int rank = (int)cl.block_rank();
  extern __shared__ __align__(16) unsigned char smraw[];
  V* xch = reinterpret_cast<V*>(smraw);   // [NT][LD] exchange
  V* colb = xch + C::NT * C::LD;          // [K][N] columns of this CTA
  V* rowb = colb + K * N;                 // [R][H1] half spectra of its rows
  V* tw = rowb + R * H1;                  // [N]
  T* p = reinterpret_cast<T*>(tw + N);    // [R][N] each
  T* h = p + E;
  T* t = h + E;
  T* g = t + E;
  T* po = g + E;
  T* u = po + E;
  T* green = u + E;                       // [K][N] compliance of its columns
  __shared__ PkState S;
  __shared__ double red[4][CL][4];        // partial sums of every CTA: start, tau, load, gap
  __shared__ double wsum[32 * 4];
  __shared__ int redo;

  const int tid = threadIdx.x, nth = blockDim.x;
  T* pg = static_cast<T*>(init.p) + (size_t)rank * E;
  const T* hg = static_cast<const T*>(init.h) + (size_t)rank * E;
  if (tid == 0) S = init;
  for (int i = tid; i < N; i += nth) tw[i] = tw_g[i];
  for (int i = tid; i < K * N; i += nth) {
    const int k1 = rank * K + i / N, k2 = i % N;
    const T q1 = w1 * (T)k1, q2 = w2 * (T)(k2 < N / 2 ? k2 : k2 - N);
    const T q = sqrt(q1 * q1 + q2 * q2);
    green[i] = (k1 == 0 && k2 == 0) || k2 == N / 2 ? (T)0 : ((T)1 - nu) / (mu * q);
  }

  cl.sync();  // every CTA runs before its shared memory is written from outside

  // sums of this CTA to every CTA's slot `which`; totals(which) after the next cluster barrier
  auto send = [&](int which, double a, double b, double c, double d) {
    double x = warp_sum4(a, b, c, d);
    x = __shfl_sync(0xffffffffu, x, ((tid & 3) >> 1) * 16 + (tid & 1) * 8);
    x = block_sum_kind(x, wsum);
    // lanes 4 r + j of warp 0: value j to CTA r
    if (tid < 32) {
      x = __shfl_sync(0xffffffffu, x, tid & 3);
      *cl.map_shared_rank(&red[which][rank][tid & 3], tid >> 2) = x;
    }
  };
  // value j of the totals in lanes of equal tid & 3 of warp 0
  auto total = [&](int which) {
    double x = red[which][(tid & 31) >> 2][tid & 3];
    for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  };
  auto value = [&](double x, int j) { return __shfl_sync(0xffffffffu, x, j); };

  // rows of `src` forward, half spectra to the column owners
  auto rows_fwd = [&](const T* src) {
    cl_fft<T, N, false>(
        xch, tw, [&](int f, int i) { return mk<V>(src[(2 * f) * N + i], src[(2 * f + 1) * N + i]); },
        [&](int f, int i, V x) { xch[f * C::LD + i + (i >> 3)] = x; });
    __syncthreads();
    for (int i = tid; i < (R / 2) * H1; i += nth) {
      const int f = i / H1, k = i - f * H1, km = (N - k) & (N - 1);
      const V zk = xch[f * C::LD + k + (k >> 3)], zm = xch[f * C::LD + km + (km >> 3)];
      const V c = cconj(zm), a = cadd(zk, c), d = csub(zk, c);
      V* dst = cl.map_shared_rank(colb, k / K) + (k % K) * N + rank * R + 2 * f;
      dst[0] = cscale(a, (T)0.5);
      dst[1] = mk<V>((T)0.5 * d.y, (T)-0.5 * d.x);
    }
  };
  // this CTA's columns: transform, compliance (times the load scale), inverse, rows to their owners
  auto cols = [&](bool scaled) {
    const double s = scaled ? S.s : 1.0;
    const float4 sw = scaled ? S.sw : make_float4(1.f, 0.f, 0.f, 1.f);
    cl_fft<T, N, false>(
        xch, tw, [&](int f, int i) { return colb[f * N + i]; },
        [&](int f, int i, V x) { colb[f * N + i] = cscale(x, scaled ? mul1(s, sw, green[f * N + i]) : green[f * N + i]); });
    __syncthreads();
    cl_fft<T, N, true>(
        xch, tw, [&](int f, int i) { return colb[f * N + i]; },
        [&](int f, int i, V x) { cl.map_shared_rank(rowb, i / R)[(i % R) * H1 + rank * K + f] = x; });
  };
  const T scale = (T)(1.0 / ((double)N * (double)N));
  // rows of the result in u
  auto rows_inv = [&]() {
    cl_fft<T, N, true>(
        xch, tw,
        [&](int f, int k) {
          const int kk = k < H1 ? k : (k > H1 ? N - k : 0);
          V A = rowb[(2 * f) * H1 + kk], B = rowb[(2 * f + 1) * H1 + kk];
          if (k > H1) { A = cconj(A); B = cconj(B); }
          if (k == H1) A = B = mk<V>(0, 0);
          return cadd(A, cmuli(B));
        },
        [&](int f, int i, V x) {
          u[(2 * f) * N + i] = x.x * scale;
          u[(2 * f + 1) * N + i] = x.y * scale;
        });
    __syncthreads();
  };

  // start: pressure scaled to the load (uniform where the guess carries none), its displacement, mean
  // gap and G
  {
    double a = 0;
    for (int i = tid; i < E; i += nth) {
      h[i] = hg[i];
      p[i] = pg[i];
      t[i] = (T)0;
      a += (double)p[i];
    }
    send(0, a, 0, 0, 0);
    cl.sync();
    if (tid < 32) {
      const double sum = value(total(0), 0);
      if (tid == 0) S.start = sum > 0 ? S.W / (S.dA * sum) : -1.0;
    }
    __syncthreads();
    const double start = S.start, unif = S.unif;
    for (int i = tid; i < E; i += nth) p[i] = start >= 0 ? (T)(start * (double)p[i]) : (T)unif;
    __syncthreads();
    rows_fwd(p);
    cl.sync();
    cols(false);
    cl.sync();
    rows_inv();
    double s0 = 0, s1 = 0;
    for (int i = tid; i < E; i += nth)
      if (p[i] > (T)0) {
        s0 += (double)u[i] - (double)h[i];
        s1 += 1;
      }
    send(1, s0, s1, 0, 0);
    cl.sync();
    if (tid < 32) {
      const double x = total(1), sum = value(x, 0), n = value(x, 1);
      if (tid == 0) {
        S.nIc = n;
        if (!(n > 0) || !isfinite(sum)) {
          S.bad = 1;
          S.done = 1;
        } else {
          S.gbar = sum / n;
          S.gbarw = words_of(S.gbar);
        }
      }
    }
    __syncthreads();
    double G = 0;
    const double gbar = S.gbar;
    for (int i = tid; i < E; i += nth)
      if (p[i] > (T)0) {
        const double gi = (double)u[i] - (double)h[i] - gbar;
        G += gi * gi;
      }
    send(2, G, 0, 0, 0);
    cl.sync();
    if (tid < 32) {
      G = value(total(2), 0);
      if (tid == 0) S.G_old = G;
    }
    __syncthreads();
  }

  while (!S.done) {  // at most max_it passes; the same decision in every CTA
    // g, conjugate direction
    {
      const double gbar = S.gbar, beta = S.beta;
      const float4 gbarw = S.gbarw, betaw = S.betaw;
      for (int i = tid; i < E; i += nth) {
        const T gi = gap1(u[i], h[i], gbar, gbarw);
        g[i] = gi;
        t[i] = p[i] > (T)0 ? axpy1(gi, beta, betaw, t[i]) : (T)0;
      }
    }
    __syncthreads();
    rows_fwd(t);
    cl.sync();
    cols(false);
    cl.sync();
    rows_inv();
    // step length
    {
      double a = 0, b = 0, c = 0, d = 0;
      for (int i = tid; i < E; i += nth)
        if (p[i] > (T)0) {
          const double xi = (double)u[i], ti = (double)t[i];
          a += xi;
          b += ti;
          c += (double)g[i] * ti;
          d += xi * ti;
        }
      send(1, a, b, c, d);
    }
    cl.sync();
    if (tid < 32) {
      const double x = total(1), sr = value(x, 0), st = value(x, 1), sgt = value(x, 2), srt = value(x, 3);
      if (tid == 0) {
        const double den = srt * S.nIc - sr * st;
        S.tau = den != 0 ? sgt * S.nIc / den : 0.0;
        S.tauw = words_of(S.tau);
      }
    }
    __syncthreads();
    // pressure step
    {
      const double tau = S.tau;
      const float4 mt = words_neg(S.tauw);
      double a = 0;
      int nol = 0;
      for (int i = tid; i < E; i += nth) {
        const T pi = p[i], ti = t[i], gi = g[i];
        T pn = (T)0;
        if (pi != (T)0 || ti != (T)0) {
          const T x = axpy1(pi, -tau, mt, ti);
          pn = x > (T)0 ? x : (T)0;
        }
        if (pn == (T)0 && gi < (T)0) {
          pn = mul1(-tau, mt, gi);
          ++nol;
        }
        po[i] = pi;
        p[i] = pn;
        if (pn != (T)0) a += (double)pn;
      }
      send(2, a, (double)nol, 0, 0);
    }
    __syncthreads();
    rows_fwd(p);
    cl.sync();
    if (tid < 32) {
      const double x = total(2), sum = value(x, 0), nol = value(x, 1);
      if (tid == 0) {
        S.delta = nol > 0 ? 0.0 : 1.0;
        if (!(sum > 0) || !isfinite(sum)) {
          S.bad = 1;
          S.done = 1;
        } else {
          S.s = S.W / (S.dA * sum);
          S.sw = words_of(S.s);
        }
      }
    }
    __syncthreads();
    if (S.done) break;  // the same in every CTA
    cols(true);
    cl.sync();
    rows_inv();
    // load scale, change, mean gap and G
    {
      const double s = S.s, gbar = S.gbar;
      const float4 sw = S.sw;
      double a = 0, b = 0, c = 0;
      int n = 0;
      for (int i = tid; i < E; i += nth) {
        T pi = p[i];
        if (pi != (T)0) {
          pi = mul1(s, sw, pi);
          p[i] = pi;
        }
        if (pi != po[i]) c += fabs((double)pi - (double)po[i]);
        if (pi > (T)0) {
          const double d = (double)u[i] - (double)h[i] - gbar;
          a += d;
          b += d * d;
          ++n;
        }
      }
      send(3, a, b, c, (double)n);
    }
    cl.sync();
    if (tid < 32) {
      const double x = total(3), sd = value(x, 0), sdd = value(x, 1), ch = value(x, 2), n = value(x, 3);
      if (tid == 0) {
        const double err = ch * S.dA_W;
        int done = 0, bad = 0;
        S.err = err;
        S.it += 1;
        if (err < S.tol || S.it >= S.max_it) done = 1;
        if (!isfinite(err)) bad = 1;
        S.nIc = n;
        redo = 0;
        if (!done && (!(n > 0) || !isfinite(sd))) {
          bad = 1;
        } else {
          const double mean = sd / n, G = fmax(sdd - sd * mean, 0.0);
          redo = !done && gap_lost(S.gbar, S.gbar + mean, G, n);
          S.gbar += mean;
          S.gbarw = words_of(S.gbar);
          if (!redo) {
            S.beta = S.G_old > 0 ? S.delta * (G / S.G_old) : 0.0;
            S.betaw = words_of(S.beta);
            S.G_old = G;
          }
        }
        if (bad) S.bad = 1;
        S.done = done | bad;
      }
    }
    __syncthreads();
    if (redo) {  // the same in every CTA
      double a = 0;
      for (int i = tid; i < E; i += nth)
        if (p[i] > (T)0) a += (double)u[i] - (double)h[i];
      send(1, a, 0, 0, 0);
      cl.sync();
      if (tid < 32) {
        const double sum = value(total(1), 0);
        if (tid == 0) S.gbar = sum / S.nIc;
      }
      __syncthreads();
      const double gbar = S.gbar;
      a = 0;
      for (int i = tid; i < E; i += nth)
        if (p[i] > (T)0) {
          const double gi = (double)u[i] - (double)h[i] - gbar;
          a += gi * gi;
        }
      send(2, a, 0, 0, 0);
      cl.sync();
      if (tid < 32) {
        const double G = value(total(2), 0);
        if (tid == 0) {
          S.gbarw = words_of(gbar);
          S.beta = S.G_old > 0 ? S.delta * (G / S.G_old) : 0.0;
          S.betaw = words_of(S.beta);
          S.G_old = G;
        }
      }
      __syncthreads();
    }
  }
  for (int i = tid; i < E; i += nth) pg[i] = p[i];
  if (rank == 0 && tid == 0) *out = S;
  cl.sync();  // no CTA leaves while another may still write to its shared memory
}

template <typename T, int N> int cluster_solve(const PkfArgs& a, const PkState& init) {
  const double two_pi = 6.283185307179586476925;
  // static shared memory besides: a constant cap below the opt-in maximum
  static_assert(ClCfg<T, N>::bytes <= 200 * 1024, "surface in shared memory");
  auto kern = k_pkf_cluster<T, N>;
  if (FVIM_CU(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024))) return FVIM_ERR_CUDA;
  kern<<<CL, ClCfg<T, N>::BT, ClCfg<T, N>::bytes, a.stream>>>(a.S, init, (const typename Cx<T>::t*)a.tw1,
                                                            (T)(two_pi / a.L1), (T)(two_pi / a.L2), (T)a.nu, (T)a.mu);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
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

// (FP64 at 128^2: eight SMs hold too few FP64 pipes, 120 us an iteration there against 66 in six kernels)
bool pkf_small(const fvim_ctx* c) {
  return !c->gen && c->n1 == c->n2 && c->n1 >= 16 && c->n1 <= (c->prec == FVIM_FP64 ? 64 : 128);
}

template <typename T> int pkf_solve_small(const PkfArgs& a, const PkState& init) {
  if (a.n1 == 16) return cluster_solve<T, 16>(a, init);
  if (a.n1 == 32) return cluster_solve<T, 32>(a, init);
  if (a.n1 == 64) return cluster_solve<T, 64>(a, init);
  if constexpr (sizeof(T) == 4)
    if (a.n1 == 128) return cluster_solve<T, 128>(a, init);
  return FVIM_ERR_UNSUPPORTED;
}

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

template int pkf_solve_small<float>(const PkfArgs&, const PkState&);
template int pkf_solve_small<double>(const PkfArgs&, const PkState&);
template int pkf_begin<float>(const PkfArgs&, const PkState&);
template int pkf_begin<double>(const PkfArgs&, const PkState&);
template int pkf_iteration<float>(const PkfArgs&);
template int pkf_iteration<double>(const PkfArgs&);
