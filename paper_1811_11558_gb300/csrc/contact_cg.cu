// Fused kernels of the Polonsky-Keer contact iteration (Sec. 5.1) on power-of-two surfaces with
// both sides from 16 to 1024: seven kernels per iteration instead of fourteen.
//
// An iteration is a chain of global sums (mean gap, G, tau, total load, change), each of which the
// next elementwise step needs, and two surface convolutions u = K*p, r = K*t.  Each elementwise
// step runs inside the row pass of the convolution next to it:
//   gap    g = u - h - gbar on the surface; G = sum over the contact of g^2 -> beta
//   rowsT  t = g + beta t on the contact, 0 elsewhere; forward rows of t
//   cols   columns: transform, surface compliance, inverse
//   rowsR  inverse rows of r = K*t, kept in registers; sums of r, t, g t and r t over the contact
//          -> tau = <g, t> / (<r, t> - rbar <t, 1>)
//   rowsP  p <- max(p - tau t, 0), points that would penetrate re-enter; sum p -> load scale s;
//          forward rows of the unscaled p
//   cols   as above, times s (the transform is linear)
//   rowsU  inverse rows of u = K*p; p <- s p, change against the old pressure, mean gap over the
//          contact -> gbar, stop test
// The sums are FP64, block partials in block order added by the last block to finish, so results
// do not depend on timing.  Every scalar, the surface and pressure pointers, the load and the
// tolerance live in the device state (PkState): one captured loop serves every call of a context.
//
// Why: each kernel is a few microseconds of launch, latency and dependent global reads, and the
// surface FFTs ran on a generic runtime-length kernel: 132 -> 75 us per iteration at 512^2 FP32, 206
// -> 156 at 1024^2.
#include <algorithm>

#include "fvim_internal.cuh"

namespace {

enum { FWD_INIT = 0, FWD_P, FWD_T };
enum { INV_U0 = 0, INV_U, INV_R };

// sums of NV doubles over the block (any whole number of warps) into part[blockIdx.x * NV + j]
template <int NV> __device__ __forceinline__ void block_sum(double (&v)[NV], double* part) {
  __shared__ double sh[NV][32];
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    double x = v[j];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) sh[j][w] = x;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0;
    for (int k = 0; k < nw; ++k) s += sh[threadIdx.x][k];
    part[blockIdx.x * NV + threadIdx.x] = s;
  }
}
// true in the last block of the grid to arrive; its first warp then adds the partials in a fixed
// order and every lane gets the sums
template <int NV> __device__ __forceinline__ bool grid_sum(double (&v)[NV], double* part, unsigned* cnt) {
  __shared__ bool last;
  block_sum<NV>(v, part);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last || threadIdx.x >= 32) return false;
  __threadfence();
  const int n = gridDim.x;
#pragma unroll
  for (int j = 0; j < NV; ++j) v[j] = 0;
  for (int b = threadIdx.x; b < n; b += 32)
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] += __ldcg(part + b * NV + j);
#pragma unroll
  for (int j = 0; j < NV; ++j)
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  if (threadIdx.x == 0) *cnt = 0u;
  return threadIdx.x == 0;
}

// state of a new solve, with the scale of the initial pressure from its sum (a guess without load
// is replaced by the uniform pressure)
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_begin(PkState* S, const T* __restrict__ p, size_t n, PkState init, double* part,
                                                   unsigned* cnt) {
  double v[1] = {0};
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) v[0] += (double)p[i];
  if (grid_sum<1>(v, part, cnt)) {
    init.start = v[0] > 0 ? init.W / (init.dA * v[0]) : 0.0;
    *S = init;
  }
}

// index of entry p of a transform in the exchange area: contiguous rows, swizzled (8-byte entries,
// 128 points and more) or with a pad slot every 8 entries, conflict-free for the radix-8 stages
template <typename V, int N> struct SurfSm {
  static constexpr bool swz = sizeof(V) == 8 && N >= 128;
  static constexpr int LD = swz ? N : N + N / 8;
  V* buf;
  static __device__ __forceinline__ int idx(int p) { return swz ? (p ^ ((p >> 3) & 15)) : p + (p >> 3); }
  __device__ __forceinline__ void put(int, int p, V x) const { buf[idx(p)] = x; }
  __device__ __forceinline__ V get(int, int p) const { return buf[idx(p)]; }
};

// Forward rows of p or t, two rows per transform, N / 8 threads per transform, blockDim.x / (N / 8)
// transforms per CTA; the half spectrum k1 < N/2 goes to surf (the Nyquist column carries no
// operator term).
template <typename T, int N, int MODE>
__global__ void __launch_bounds__(512) k_pkf_rows_fwd(PkState* S, const T* __restrict__ g, T* __restrict__ t,
                                                      T* __restrict__ pold, typename Cx<T>::t* __restrict__ surf,
                                                      const typename Cx<T>::t* __restrict__ tw, int n2, double* part,
                                                      unsigned* cnt) {
  typedef typename Cx<T>::t V;
  if (MODE != FWD_INIT && S->done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T8, tt = threadIdx.x % T8;
  const int pair = blockIdx.x * (blockDim.x / T8) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  const double beta = S->beta, tau = S->tau, start = S->start, unif = S->unif;
  V v[1][8];
  double sum[2] = {0, 0};
  auto value = [&](size_t i) -> T {
    if (MODE == FWD_INIT) {
      const T x = start > 0 ? (T)(start * (double)p[i]) : (T)unif;
      p[i] = x;
      t[i] = (T)0;
      return x;
    } else if (MODE == FWD_P) {
      const T po = p[i], gi = g[i];
      T pn = (T)fmax((double)po - tau * (double)t[i], 0.0);
      const bool ol = (pn == (T)0) && (gi < (T)0);
      if (ol) pn = (T)(-tau * (double)gi);
      pold[i] = po;
      p[i] = pn;
      sum[0] += (double)pn;
      sum[1] += ol ? 1.0 : 0.0;
      return pn;
    } else {
      const T x = p[i] > (T)0 ? (T)((double)g[i] + beta * (double)t[i]) : (T)0;
      t[i] = x;
      return x;
    }
  };
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    v[0][m] = mk<V>(0, 0);
    if (live) {
      const size_t i = i0 + m * T8;
      v[0][m].x = value(i);
      v[0][m].y = value(i + N);
    }
  }
  SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft_ct<V, false, N, 1, 1>(v, tt, sm, tw);
  // separation of the two rows: Z(N - k) of k = tt + m N/8, m < 4, is in another thread's upper half
#pragma unroll
  for (int m = 4; m < 8; ++m) sm.put(0, tt + m * T8, v[0][m]);
  __syncthreads();
  if (live) {
    V* o = surf + (size_t)2 * pair * H1 + tt;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      V zm = sm.get(0, (N - tt - m * T8) & (N - 1));
      if (m == 0 && tt == 0) zm = v[0][0];
      const V c = cconj(zm), a = cadd(v[0][m], c), d = csub(v[0][m], c);
      o[m * T8] = cscale(a, (T)0.5);
      o[H1 + m * T8] = mk<V>((T)0.5 * d.y, (T)-0.5 * d.x);
    }
  }
  if (MODE == FWD_P && grid_sum<2>(sum, part, cnt)) {
    S->delta = sum[1] > 0 ? 0.0 : 1.0;
    if (!(sum[0] > 0) || !isfinite(sum[0])) {
      S->bad = 1;
      S->done = 1;
    } else {
      S->s = S->W / (S->dA * sum[0]);
    }
  }
}

// Columns: forward transform of kc k1 columns, surface compliance u3_hat = (1 - nu) / (mu q) p_hat
// (zero on mode 0 and on the Nyquist row), times the load scale for the pressure, inverse
// transform.  Few columns per CTA (32-byte row segments): the plane stays in L2, and 512 points
// in 16-column CTAs would leave most of the chip idle.
template <typename T, int N, bool SCALE>
__global__ void __launch_bounds__(512) k_pkf_cols(const PkState* S, typename Cx<T>::t* __restrict__ plane,
                                                  const typename Cx<T>::t* __restrict__ tw, int h1, int kc, T w1, T w2, T nu,
                                                  T mu) {
  typedef typename Cx<T>::t V;
  if (S->done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8;
  const int f = threadIdx.x % kc, t = threadIdx.x / kc;
  const int k1 = blockIdx.x * kc + f;
  const double s = SCALE ? S->s : 1.0;
  V* col = plane + k1;
  V v[1][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[0][m] = col[(size_t)(t + m * T8) * h1];
  struct Sm {
    V* buf;
    int kc, f;
    __device__ __forceinline__ void put(int, int p, V x) const { buf[p * kc + f] = x; }
    __device__ __forceinline__ V get(int, int p) const { return buf[p * kc + f]; }
  } sm{reinterpret_cast<V*>(smraw), kc, f};
  fft_ct<V, false, N, 1, 1>(v, t, sm, tw);
  const T q1 = w1 * (T)k1;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k2 = t + m * T8;
    const T q2 = w2 * (T)(k2 < N / 2 ? k2 : k2 - N);
    const T q = sqrt(q1 * q1 + q2 * q2);
    const bool none = (k1 == 0 && k2 == 0) || k2 == N / 2;
    T f0 = none ? (T)0 : ((T)1 - nu) / (mu * q);
    if (SCALE) f0 = (T)(s * (double)f0);
    v[0][m] = cscale(v[0][m], f0);
  }
  __syncthreads();  // the exchange area is reused by the inverse transform
  fft_ct<V, true, N, 1, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 8; ++m) col[(size_t)(t + m * T8) * h1] = v[0][m];
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
  constexpr int T8 = N / 8, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T8, tt = threadIdx.x % T8;
  const int pair = blockIdx.x * (blockDim.x / T8) + r;
  const bool live = pair < n2 / 2;
  T* p = static_cast<T*>(S->p);
  const T* h = static_cast<const T*>(S->h);
  V v[1][8];
  const V* sa = surf + (size_t)(live ? 2 * pair : 0) * H1;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k = tt + m * T8;
    const int kk = k < H1 ? k : (k > H1 ? N - k : 0);
    V A = sa[kk], B = sa[H1 + kk];
    if (k > H1) { A = cconj(A); B = cconj(B); }
    if (k == H1) A = B = mk<V>(0, 0);
    v[0][m] = cadd(A, cmuli(B));
  }
  SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft_ct<V, true, N, 1, 1>(v, tt, sm, tw);
  const size_t i0 = (size_t)(live ? 2 * pair : 0) * N + tt;
  if (MODE == INV_R) {
    double sum[4] = {0, 0, 0, 0};
    auto add = [&](size_t i, T x) {
      if (p[i] > (T)0) {
        const double ti = (double)t[i];
        sum[0] += (double)x;
        sum[1] += ti;
        sum[2] += (double)g[i] * ti;
        sum[3] += (double)x * ti;
      }
    };
    if (live) {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        add(i0 + m * T8, v[0][m].x * scale);
        add(i0 + m * T8 + N, v[0][m].y * scale);
      }
    }
    if (grid_sum<4>(sum, part, cnt)) {
      const double den = sum[3] - sum[0] / S->nIc * sum[1];
      S->tau = den != 0 ? sum[2] / den : 0.0;
    }
  } else {
    const double s = S->s;
    double sum[3] = {0, 0, 0};
    auto add = [&](size_t i, T x) {
      T pi = p[i];
      if (MODE == INV_U) {
        pi = (T)(s * (double)pi);
        p[i] = pi;
        sum[2] += fabs((double)pi - (double)pold[i]);
      }
      u[i] = x;
      if (pi > (T)0) {
        sum[0] += (double)x - (double)h[i];
        sum[1] += 1;
      }
    };
    if (live) {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        add(i0 + m * T8, v[0][m].x * scale);
        add(i0 + m * T8 + N, v[0][m].y * scale);
      }
    }
    if (grid_sum<3>(sum, part, cnt)) {
      int done = 0, bad = 0;
      if (MODE == INV_U) {
        S->err = S->dA * sum[2] / S->W;
        S->it += 1;
        if (S->err < S->tol || S->it >= S->max_it) done = 1;
        if (!isfinite(S->err)) bad = 1;
      }
      S->nIc = sum[1];
      if (!done && (!(sum[1] > 0) || !isfinite(sum[0]))) bad = 1;
      else S->gbar = sum[0] / sum[1];
      if (bad) S->bad = 1;
      S->done = done | bad;
      if (MODE == INV_U && use_cond) cudaGraphSetConditional(cond, (done | bad) ? 0u : 1u);
    }
  }
}

// g = u - h - gbar; sum over the contact of g^2 -> beta
template <typename T>
__global__ void __launch_bounds__(256) k_pkf_gap(PkState* S, const T* __restrict__ u, T* __restrict__ g, size_t n,
                                                 double* part, unsigned* cnt) {
  if (S->done) return;
  const double gbar = S->gbar;
  const T* h = static_cast<const T*>(S->h);
  const T* p = static_cast<const T*>(S->p);
  double v[1] = {0};
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const T gi = (T)((double)u[i] - (double)h[i] - gbar);
    g[i] = gi;
    if (p[i] > (T)0) v[0] += (double)gi * (double)gi;
  }
  if (grid_sum<1>(v, part, cnt)) {
    S->beta = S->delta * (v[0] / S->G_old);
    S->G_old = v[0];
  }
}

// CTA of a row pass: about one transform pair per CTA and SM, whole warps
struct RowCfg {
  int grid, threads;
  size_t smem;
};
template <typename T, int N> RowCfg row_cfg(int n2) {
  typedef typename Cx<T>::t V;
  const int pairs = n2 / 2, T8 = N / 8;
  int slots = 1;
  while (slots * 2 * 128 <= pairs && slots * 2 * T8 <= 512) slots *= 2;
  const int threads = std::max(32, slots * T8);
  slots = threads / T8;
  return RowCfg{(pairs + slots - 1) / slots, threads, (size_t)slots * SurfSm<V, N>::LD * sizeof(V)};
}

// dynamic shared memory cap of the row kernels (at most four FP64 transforms of 1024 points; they
// hold static shared memory too, so not the whole opt-in maximum); the same value on every call
template <typename K> void row_smem_cap(K kern) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
}

template <typename T, int N, int MODE> void rows_fwd(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  const RowCfg r = row_cfg<T, N>(a.n2);
  row_smem_cap(k_pkf_rows_fwd<T, N, MODE>);
  k_pkf_rows_fwd<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(a.S, (const T*)a.g, (T*)a.t, (T*)a.pold, (V*)a.surf,
                                                                   (const V*)a.tw1, a.n2, a.part, a.cnt);
}
template <typename T, int N, int MODE> void rows_inv(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  const RowCfg r = row_cfg<T, N>(a.n2);
  row_smem_cap(k_pkf_rows_inv<T, N, MODE>);
  k_pkf_rows_inv<T, N, MODE><<<r.grid, r.threads, r.smem, a.stream>>>(
      a.S, (const T*)a.g, (const T*)a.t, (const T*)a.pold, (T*)a.u, (const V*)a.surf, (const V*)a.tw1, a.n2,
      (T)(1.0 / ((double)N * (double)a.n2)), a.part, a.cnt, a.cond, a.use_cond);
}
template <typename T, int N, bool SCALE> void cols(const PkfArgs& a) {
  typedef typename Cx<T>::t V;
  int kc = (int)(32 / sizeof(V));
  if (kc > a.h1) kc = a.h1;
  const double two_pi = 6.283185307179586476925;
  smem_cap(k_pkf_cols<T, N, SCALE>);
  k_pkf_cols<T, N, SCALE><<<a.h1 / kc, kc * (N / 8), (size_t)kc * N * sizeof(V), a.stream>>>(
      a.S, (V*)a.surf, (const V*)a.tw2, a.h1, kc, (T)(two_pi / a.L1), (T)(two_pi / a.L2), (T)a.nu, (T)a.mu);
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
inline int flat_grid(size_t n) { return (int)std::min<size_t>(std::max<size_t>((n + 1023) / 1024, 1), 152); }

}  // namespace

bool pkf_available(const fvim_ctx* c) { return !c->gen && c->n1 >= 16 && c->n2 >= 16; }

template <typename T> int pkf_begin(const PkfArgs& a, const PkState& init) {
  const size_t n = (size_t)a.n1 * a.n2;
  k_pkf_begin<T><<<flat_grid(n), 256, 0, a.stream>>>(a.S, (const T*)init.p, n, init, a.part, a.cnt);
  rows_fwd_any<T, FWD_INIT>(a);
  cols_any<T, false>(a);
  rows_inv_any<T, INV_U0>(a);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template <typename T> int pkf_iteration(const PkfArgs& a) {
  const size_t n = (size_t)a.n1 * a.n2;
  k_pkf_gap<T><<<flat_grid(n), 256, 0, a.stream>>>(a.S, (const T*)a.u, (T*)a.g, n, a.part, a.cnt);
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
