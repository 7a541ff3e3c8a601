// Surface transforms (one plane) and the Boussinesq volume field.
//
// A plane of 512 x 512 is 1 MB: its transforms are latency bound, so the kernels hold four values per
// thread and few rows or columns per CTA (the plane stays in L2).  Rows of a real field go two per
// complex transform; the half spectrum k1 < N1/2 is kept (the Nyquist column carries no operator
// term).  512 x 512 FP32, us (event-bracketed): rows 13.6 -> 7.4, columns 8.2 -> 7.5.
#include "fvim_internal.cuh"

namespace {

template <typename T, int N>
__global__ void __launch_bounds__(512) k_surf_rows_fwd(const T* __restrict__ f, typename Cx<T>::t* __restrict__ surf,
                                                       const typename Cx<T>::t* __restrict__ tw, int n2) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, t = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  const T* src = f + (size_t)(live ? 2 * pair : 0) * N + t;
  V v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = mk<V>(src[m * T4], src[N + m * T4]);
  SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft4_ct<V, false, N, 1>(v, t, sm, tw);
  // separation of the two rows: Z(N - k) of k = t + m N/4, m < 2, is in another thread's upper half
  sm.put(t + 2 * T4, v[2]);
  sm.put(t + 3 * T4, v[3]);
  __syncthreads();
  if (!live) return;
  V* o = surf + (size_t)2 * pair * H1 + t;
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    V zm = sm.get((N - t - m * T4) & (N - 1));
    if (m == 0 && t == 0) zm = v[0];
    const V c = cconj(zm), a = cadd(v[m], c), d = csub(v[m], c);
    o[m * T4] = cscale(a, (T)0.5);
    o[H1 + m * T4] = mk<V>((T)0.5 * d.y, (T)-0.5 * d.x);
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(512) k_surf_rows_inv(const typename Cx<T>::t* __restrict__ surf, T* __restrict__ f,
                                                       const typename Cx<T>::t* __restrict__ tw, int n2, T scale) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4, H1 = N / 2, LD = SurfSm<V, N>::LD;
  const int r = threadIdx.x / T4, t = threadIdx.x % T4;
  const int pair = blockIdx.x * (blockDim.x / T4) + r;
  const bool live = pair < n2 / 2;
  const V* sa = surf + (size_t)(live ? 2 * pair : 0) * H1;
  V v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int k = t + m * T4;
    const int kk = k < H1 ? k : (k > H1 ? N - k : 0);
    V A = sa[kk], B = sa[H1 + kk];
    if (k > H1) { A = cconj(A); B = cconj(B); }
    if (k == H1) A = B = mk<V>(0, 0);
    v[m] = cadd(A, cmuli(B));
  }
  const SurfSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * LD};
  fft4_ct<V, true, N, 1>(v, t, sm, tw);
  if (!live) return;
  T* o = f + (size_t)2 * pair * N + t;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    o[m * T4] = v[m].x * scale;
    o[N + m * T4] = v[m].y * scale;
  }
}

template <typename T, int N, bool INV>
__global__ void __launch_bounds__(512) k_surf_cols(typename Cx<T>::t* __restrict__ plane,
                                                   const typename Cx<T>::t* __restrict__ tw, int h1, int kc) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T4 = N / 4;
  const int f = threadIdx.x % kc, t = threadIdx.x / kc;
  V* col = plane + (size_t)blockIdx.x * kc + f;
  V v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = col[(size_t)(t + m * T4) * h1];
  const SurfColSm<V> sm{reinterpret_cast<V*>(smraw), kc, f};
  fft4_ct<V, INV, N, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 4; ++m) col[(size_t)(t + m * T4) * h1] = v[m];
}

// Inverse column pass of the Boussinesq field of a normal pressure (Eq. B:fourier): every value of
// the field's spectrum is a closed form of p_hat, so it is evaluated as the column's input instead
// of being written and read back (one pass over the volume less).  With f = p_hat e^{-qz}, a = qz,
// the rotated strain times 2 mu is qq: (2 nu - 1 + a) f, 33: (2 nu - 1 - a) f, q3: i a f; in the
// stress the normal components gain -2 nu f.  A thread owns two adjacent columns (16-byte
// accesses), CW columns per CTA, one (layer, component) plane per blockIdx.y.  Bound by instruction
// issue (the exponential and the wavenumber are evaluated per plane).  512 x 512 x 32: 105 us for the
// separate evaluation and column pass -> 83.
template <int CW> struct PairSm {
  float2* buf;
  int f2;  // column pair
  __device__ __forceinline__ void put(int g, int p, float2 x) const { buf[p * CW + 2 * f2 + g] = x; }
  __device__ __forceinline__ float2 get(int g, int p) const { return buf[p * CW + 2 * f2 + g]; }
};
template <int COMP, int N>
__device__ __forceinline__ void bous_values(float2 (&v)[2][8], const float4* __restrict__ src, size_t rs, int kc, int t,
                                            float w1, float w2, float zi, float nu, float sc, int stress) {
  const float al = 2.f * nu - 1.f, off = stress ? -2.f * nu : 0.f;
  const float q1[2] = {w1 * (float)kc, w1 * (float)(kc + 1)};
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const float4 p4 = src[(size_t)(t + m * (N / 8)) * rs];
    v[0][m] = make_float2(p4.x, p4.y);
    v[1][m] = make_float2(p4.z, p4.w);
  }
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k2 = t + m * (N / 8);
    const float q2 = w2 * (float)(m < 4 ? k2 : k2 - N);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float2 p = v[j][m];
      const float qq = q1[j] * q1[j] + q2 * q2;
      // 1 / q with one Newton step, q = q^2 / q with its residual (e^{-qz} magnifies the rounding of
      // q); mode 0 is set apart by the caller
      float iq = rsqrtf(qq);
      iq = iq * (1.5f - 0.5f * qq * iq * iq);
      const float qh = qq * iq;
      const float a = fmaf(fmaf(-qh, qh, qq) * 0.5f, iq, qh) * zi, ex = expf(-a) * sc;
      const float c = q1[j] * iq, s = q2 * iq, l = al + a;
      float r;
      if (COMP == 0) r = c * c * l + off;
      else if (COMP == 1) r = s * s * l + off;
      else if (COMP == 2) r = al - a + off;
      else if (COMP == 3) r = s * a;
      else if (COMP == 4) r = c * a;
      else r = c * s * l;
      r *= ex;
      v[j][m] = (COMP == 3 || COMP == 4) ? make_float2(-r * p.y, r * p.x) : cscale(p, r);
    }
  }
}
template <int N, int CW>
__global__ void __launch_bounds__(N / 16 * CW, 1024 / (N / 16 * CW) > 0 ? 1024 / (N / 16 * CW) : 1)
    k_bous_cols(const float2* __restrict__ surf, float2* __restrict__ spec, const float2* __restrict__ tw,
                const float* __restrict__ zn, int h1, float w1, float w2, float nu, float sc, float zero33, float zero11,
                int stress) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8, NP = CW / 2;
  const int f2 = threadIdx.x % NP, t = threadIdx.x / NP;
  const int z = blockIdx.y / 6, comp = blockIdx.y - 6 * z;
  const int kc = blockIdx.x * CW + 2 * f2;  // first of the thread's two columns
  const float4* src = reinterpret_cast<const float4*>(surf + kc);
  const size_t rs = (size_t)h1 / 2;  // row stride in float4
  const float zi = zn[z];
  float2 v[2][8];
  switch (comp) {
    case 0: bous_values<0, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
    case 1: bous_values<1, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
    case 2: bous_values<2, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
    case 3: bous_values<3, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
    case 4: bous_values<4, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
    default: bous_values<5, N>(v, src, rs, kc, t, w1, w2, zi, nu, sc, stress); break;
  }
  if (t == 0) {
    v[0][4] = v[1][4] = make_float2(0.f, 0.f);  // k2 = N/2 is not in Z^2_N
    if (kc == 0) {                              // mode 0: laminate
      const float4 p4 = src[0];
      const float r = comp == 2 ? zero33 : (comp < 2 ? zero11 : 0.f);
      v[0][0] = make_float2(r * p4.x, r * p4.y);
    }
  }
  const PairSm<CW> x{reinterpret_cast<float2*>(smraw), f2};
  fft_ct<float2, true, N, 2, 1>(v, t, x, tw);
  float4* o = reinterpret_cast<float4*>(spec + (size_t)blockIdx.y * N * h1 + kc);
#pragma unroll
  for (int m = 0; m < 8; ++m) o[(size_t)(t + m * T8) * rs] = make_float4(v[0][m].x, v[0][m].y, v[1][m].x, v[1][m].y);
}

template <int N, int CW> void bous_cols(const fvim_ctx* c, int out_kind) {
  const double two_pi = 6.283185307179586476925;
  const bool st = out_kind == FVIM_STRESS;
  const double e33 = -1.0 / (c->lam + 2.0 * c->mu);  // uniform pressure: the strain below it
  smem_cap(k_bous_cols<N, CW>, (size_t)N * CW * sizeof(float2));
  launch_chain(c, k_bous_cols<N, CW>, dim3(c->h1 / CW, c->nz * 6), N / 16 * CW, (size_t)N * CW * sizeof(float2), 
      (const float2*)c->surf, (float2*)c->spec, (const float2*)c->tw2, (const float*)c->z_dev, c->h1,
      (float)(two_pi / c->L1), (float)(two_pi / c->L2), (float)c->nu, st ? 1.f : (float)(0.5 / c->mu),
      st ? -1.f : (float)e33, st ? (float)(c->lam * e33) : 0.f, st ? 1 : 0);
}

}  // namespace

#define SURF_SIZES(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)

template <typename T> bool launch_surf_rows_fwd(const fvim_ctx* c, const T* f) {
  typedef typename Cx<T>::t V;
  if (c->gen) return false;
#define CASE(N)                                                                                                 \
  if (c->n1 == N) {                                                                                             \
    const SurfRowCfg r = surf_row_cfg<T, N>(c->n2);                                                             \
    launch_chain(c, k_surf_rows_fwd<T, N>, r.grid, r.threads, r.smem, f, (V*)c->surf, (const V*)c->tw1, c->n2);   \
    return true;                                                                                                \
  }
  SURF_SIZES(CASE)
#undef CASE
  return false;
}
template <typename T> bool launch_surf_rows_inv(const fvim_ctx* c, T* f, T scale) {
  typedef typename Cx<T>::t V;
  if (c->gen) return false;
#define CASE(N)                                                                                                       \
  if (c->n1 == N) {                                                                                                   \
    const SurfRowCfg r = surf_row_cfg<T, N>(c->n2);                                                                   \
    launch_chain(c, k_surf_rows_inv<T, N>, r.grid, r.threads, r.smem, (const V*)c->surf, f, (const V*)c->tw1, c->n2, scale); \
    return true;                                                                                                      \
  }
  SURF_SIZES(CASE)
#undef CASE
  return false;
}
template <typename T> bool launch_surf_cols(const fvim_ctx* c, bool inverse) {
  typedef typename Cx<T>::t V;
  if (c->gen) return false;
  // 32-byte row segments, at most 512 threads
  int kc = (int)(32 / sizeof(V));
  if (kc > c->h1) kc = c->h1;
  while (kc > 1 && kc * (c->n2 / 4) > 512) kc >>= 1;
  const size_t smem = (size_t)kc * c->n2 * sizeof(V);
#define CASE(N)                                                                                             \
  if (c->n2 == N) {                                                                                         \
    if (inverse) {                                                                                          \
      smem_cap(k_surf_cols<T, N, true>, smem);                                                                    \
      launch_chain(c, k_surf_cols<T, N, true>, c->h1 / kc, kc * (N / 4), smem, (V*)c->surf, (const V*)c->tw2, c->h1, kc);  \
    } else {                                                                                                \
      smem_cap(k_surf_cols<T, N, false>, smem);                                                                   \
      launch_chain(c, k_surf_cols<T, N, false>, c->h1 / kc, kc * (N / 4), smem, (V*)c->surf, (const V*)c->tw2, c->h1, kc); \
    }                                                                                                       \
    return true;                                                                                            \
  }
  SURF_SIZES(CASE)
#undef CASE
  return false;
}

bool launch_bous_cols(const fvim_ctx* c, int out_kind) {
  if (c->gen || c->prec != FVIM_FP32 || c->h1 % 16) return false;
#define CASE(N, CW)              \
  if (c->n2 == N) {              \
    bous_cols<N, CW>(c, out_kind); \
    return true;                 \
  }
  CASE(64, 16) CASE(128, 16) CASE(256, 16) CASE(512, 16) CASE(1024, 8)
#undef CASE
  return false;
}

template bool launch_surf_rows_fwd<float>(const fvim_ctx*, const float*);
template bool launch_surf_rows_fwd<double>(const fvim_ctx*, const double*);
template bool launch_surf_rows_inv<float>(const fvim_ctx*, float*, float);
template bool launch_surf_rows_inv<double>(const fvim_ctx*, double*, double);
template bool launch_surf_cols<float>(const fvim_ctx*, bool);
template bool launch_surf_cols<double>(const fvim_ctx*, bool);
