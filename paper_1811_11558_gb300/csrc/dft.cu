// In-plane discrete Fourier transforms of grids whose sides are not both powers of two (odd
// sides such as 81 = 3^4, the discretisation of the paper's elastic-perfectly-plastic Hertz
// comparison, App. C).  Direct evaluation of the Sec. 3.1 DFT,
//   X(k) = sum_n x(n) exp(-2 pi i k n / N),
// O(N) per output value, with the exact twiddle table exp(-2 pi i j / N), j = (k n) mod N.
//
// Layout (fvim_ctx::gen): the half spectrum of a real row keeps k1 = 0 .. floor(N1/2) (hs
// columns; for an even N1 the last one is the Nyquist column, which the depth kernel treats
// as outside Z^2_N), stored with a row stride ldh = hs rounded up to 16 columns; the padding
// columns are written as zeros.  There is no side array: every coefficient is in the
// spectrum.  The full spectrum of a real row follows from X(N1 - k) = conj X(k).
//
// Direct evaluation in folded form: with a(n) + a(N - n) and a(n) - a(N - n), n = 1 .. (N-1)/2,
//   X(k), X(N - k) = a(0) + C(k) -+ i S(k),  C = sum (a(n) + a(N - n)) cos,  S = sum (a(n) - a(N - n)) sin
// (plus (-1)^k a(N/2) on an even side), and likewise for the inverse rows: half the terms, and two
// outputs from each column sum.  The inner loops keep one twiddle for several rows or columns per
// thread (FP32: eight rows, four complex columns), read as broadcast vectors: what bounded the plain form
// was two shared-memory reads per multiply-add.  81 x 81 x 32 FP32, us: rows 39 -> 14, columns 33 ->
// 18, inverse rows 37 -> 16 (event-bracketed launches); apply 143 -> 64.
#include "fvim_internal.cuh"

namespace {

// Rows per thread RT (row kernels, four times as many per CTA), columns per CTA and thread CT, CC (column
// kernel).  FP32: several per thread, which share a twiddle.  FP64 sums are bound by the FP64 pipe, one per
// scheduler, whatever they read, so there one each, for the most warps: eight rows and four columns per
// thread left 8 CTAs for the rows of 256 x 5 x 8.  Applies with u3, us, plain sums -> several -> one: 256 x
// 5 x 8 418 -> 938 -> 155, 255 x 64 x 8 2026 -> 994 -> 613, 81 x 81 x 32 2377 -> 674 -> 563.
template <typename T> struct Dft {
  static constexpr int RT = sizeof(T) == 4 ? 8 : 1, RB = 4 * RT, CT = sizeof(T) == 4 ? 16 : 2, CC = sizeof(T) == 4 ? 4 : 1;
  static constexpr int LD = RB + 16 / (int)sizeof(T);  // row stride of the folded tables (the fill walks them along n)
};

// RT consecutive values of T at a 16-byte boundary
template <typename T, int RT> __device__ __forceinline__ void ld_rows(T (&v)[RT], const T* p) {
  if constexpr (RT == 1) {
    v[0] = p[0];
  } else if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int q = 0; q < RT; q += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + q);
      v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < RT; q += 2) {
      const double2 a = *reinterpret_cast<const double2*>(p + q);
      v[q] = a.x; v[q + 1] = a.y;
    }
  }
}
// CC complex columns at a 16-byte boundary
template <typename V, int CC> __device__ __forceinline__ void ld_cols(V (&v)[CC], const V* p) {
  if constexpr (sizeof(V) == 8 && CC % 2 == 0) {
#pragma unroll
    for (int q = 0; q < CC; q += 2) {
      const float4 a = *reinterpret_cast<const float4*>(p + q);
      v[q] = mk<V>(a.x, a.y);
      v[q + 1] = mk<V>(a.z, a.w);
    }
  } else {
#pragma unroll
    for (int q = 0; q < CC; ++q) v[q] = p[q];
  }
}

// forward row DFTs of real rows: src [rows][n1] -> dst [rows][ldh] (k1 < hs, zeros above)
template <typename T>
__global__ void __launch_bounds__(256) k_dft_rows_fwd(const T* __restrict__ src, typename Cx<T>::t* __restrict__ dst,
                                                      const typename Cx<T>::t* __restrict__ tw, int n1, int hs,
                                                      int ldh, size_t rows) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int LD = Dft<T>::LD, RT = Dft<T>::RT, RB = Dft<T>::RB;
  const int H = n1 / 2, J = (n1 - 1) / 2;             // folded terms n = 1 .. J
  T* P = reinterpret_cast<T*>(smraw);                 // [H + 1][LD] sums; row 0: a(0), row H of an even side: a(N/2)
  T* Q = P + (size_t)(H + 1) * LD;                    // [H + 1][LD] differences
  V* w = reinterpret_cast<V*>(Q + (size_t)(H + 1) * LD);  // [n1] twiddles
  const size_t r0 = (size_t)blockIdx.x * RB;
  const int nr = (int)((rows - r0) < (size_t)RB ? rows - r0 : RB);
  for (int i = threadIdx.x; i < n1; i += blockDim.x) w[i] = tw[i];
  for (int i = threadIdx.x; i < RB * (H + 1); i += blockDim.x) {
    const int r = i / (H + 1), n = i - r * (H + 1);
    T a = 0, b = 0;
    if (r < nr) {
      a = src[(r0 + r) * n1 + n];
      if (n > 0 && n <= J) b = src[(r0 + r) * n1 + n1 - n];
    }
    P[n * LD + r] = a + b;
    Q[n * LD + r] = a - b;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (RB / RT) * ldh; i += blockDim.x) {
    const int g = i / ldh, k = i - g * ldh;
    T c[RT], s[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) c[q] = s[q] = (T)0;
    if (k < hs) {
      ld_rows(c, P + g * RT);
      const T* pp = P + g * RT + LD;
      const T* qq = Q + g * RT + LD;
      int j = 0;  // (k n) mod n1
      for (int n = 1; n <= J; ++n, pp += LD, qq += LD) {
        j += k;
        if (j >= n1) j -= n1;
        const V e = w[j];
        T a[RT], b[RT];
        ld_rows(a, pp);
        ld_rows(b, qq);
#pragma unroll
        for (int q = 0; q < RT; ++q) {
          c[q] += e.x * a[q];
          s[q] += e.y * b[q];
        }
      }
      if (J < H) {
        T a[RT];
        ld_rows(a, pp);
#pragma unroll
        for (int q = 0; q < RT; ++q) c[q] += (k & 1) ? -a[q] : a[q];
      }
    }
#pragma unroll
    for (int q = 0; q < RT; ++q)
      if (g * RT + q < nr) dst[(r0 + g * RT + q) * ldh + k] = mk<V>(c[q], s[q]);
  }
}

// column DFTs along x2, in place: planes [nplanes][n2][ldh], CT columns per CTA
template <typename T, bool INV>
__global__ void __launch_bounds__(256) k_dft_cols(typename Cx<T>::t* __restrict__ spec,
                                                  const typename Cx<T>::t* __restrict__ tw, int n2, int ldh) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int CT = Dft<T>::CT, CC = Dft<T>::CC;
  const int H = n2 / 2, J = (n2 - 1) / 2;
  V* P = reinterpret_cast<V*>(smraw);       // [H + 1][CT] sums; row 0: a(0), row H of an even side: a(N/2)
  V* Q = P + (size_t)(H + 1) * CT;          // [H + 1][CT] differences
  V* w = Q + (size_t)(H + 1) * CT;          // [n2] twiddles
  V* A = spec + (size_t)blockIdx.y * n2 * ldh + (size_t)blockIdx.x * CT;
  for (int i = threadIdx.x; i < n2; i += blockDim.x) {
    V t = tw[i];
    if (INV) t.y = -t.y;
    w[i] = t;
  }
  for (int i = threadIdx.x; i < (H + 1) * CT; i += blockDim.x) {
    const int n = i / CT, c = i - n * CT;
    const V a = A[(size_t)n * ldh + c];
    V b = mk<V>(0, 0);
    if (n > 0 && n <= J) b = A[(size_t)(n2 - n) * ldh + c];
    P[i] = cadd(a, b);
    Q[i] = csub(a, b);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (CT / CC) * (H + 1); i += blockDim.x) {
    const int g = i / (H + 1), k = i - g * (H + 1);
    V c[CC], s[CC];
#pragma unroll
    for (int q = 0; q < CC; ++q) {
      c[q] = P[g * CC + q];
      s[q] = mk<V>(0, 0);
    }
    const V* pp = P + g * CC + CT;
    const V* qq = Q + g * CC + CT;
    int j = 0;  // (k n) mod n2
    for (int n = 1; n <= J; ++n, pp += CT, qq += CT) {
      j += k;
      if (j >= n2) j -= n2;
      const V e = w[j];
      V a[CC], b[CC];
      ld_cols(a, pp);
      ld_cols(b, qq);
#pragma unroll
      for (int q = 0; q < CC; ++q) {
        c[q] = caxpy(c[q], e.x, a[q]);
        s[q] = caxpy(s[q], e.y, b[q]);
      }
    }
    if (J < H) {
#pragma unroll
      for (int q = 0; q < CC; ++q) c[q] = (k & 1) ? csub(c[q], pp[q]) : cadd(c[q], pp[q]);
    }
    V* o = A + (size_t)k * ldh + g * CC;
    V* om = A + (size_t)(n2 - k) * ldh + g * CC;
    const bool mirror = k > 0 && 2 * k != n2;
#pragma unroll
    for (int q = 0; q < CC; ++q) {
      o[q] = mk<V>(c[q].x - s[q].y, c[q].y + s[q].x);                 // c + i s, e = cos -+ i sin
      if (mirror) om[q] = mk<V>(c[q].x + s[q].y, c[q].y - s[q].x);    // c - i s
    }
  }
}

// inverse row DFTs to real rows: src [rows][ldh] (k1 < hs) -> dst [rows][n1], times scale;
// x(n), x(N - n) = X(0) + 2 sum_{0 < k < n1/2} (Re X(k) cos -+ Im X(k) sin) + (n1 even) X(n1/2) (-1)^n
template <typename T>
__global__ void __launch_bounds__(256) k_dft_rows_inv(const typename Cx<T>::t* __restrict__ src, T* __restrict__ dst,
                                                      const typename Cx<T>::t* __restrict__ tw, int n1, int hs,
                                                      int ldh, size_t rows, T scale) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int LD = Dft<T>::LD, RT = Dft<T>::RT, RB = Dft<T>::RB;
  const int H = n1 / 2, J = (n1 - 1) / 2;
  T* P = reinterpret_cast<T*>(smraw);                 // [H + 1][LD] real parts (H = hs - 1)
  T* Q = P + (size_t)(H + 1) * LD;                    // [H + 1][LD] imaginary parts
  V* w = reinterpret_cast<V*>(Q + (size_t)(H + 1) * LD);  // [n1]
  const size_t r0 = (size_t)blockIdx.x * RB;
  const int nr = (int)((rows - r0) < (size_t)RB ? rows - r0 : RB);
  for (int i = threadIdx.x; i < n1; i += blockDim.x) w[i] = tw[i];
  for (int i = threadIdx.x; i < RB * hs; i += blockDim.x) {
    const int r = i / hs, k = i - r * hs;
    V x = mk<V>(0, 0);
    if (r < nr) x = src[(r0 + r) * ldh + k];
    P[k * LD + r] = x.x;
    Q[k * LD + r] = x.y;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (RB / RT) * (H + 1); i += blockDim.x) {
    const int g = i / (H + 1), n = i - g * (H + 1);
    T c[RT], s[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) c[q] = s[q] = (T)0;
    const T* pp = P + g * RT + LD;
    const T* qq = Q + g * RT + LD;
    int j = 0;  // (k n) mod n1
    for (int k = 1; k <= J; ++k, pp += LD, qq += LD) {
      j += n;
      if (j >= n1) j -= n1;
      const V e = w[j];  // cos - i sin
      T a[RT], b[RT];
      ld_rows(a, pp);
      ld_rows(b, qq);
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        c[q] += e.x * a[q];
        s[q] += e.y * b[q];
      }
    }
    T x0[RT], xn[RT];
    ld_rows(x0, P + g * RT);
    if (J < H) {
      ld_rows(xn, pp);
#pragma unroll
      for (int q = 0; q < RT; ++q) x0[q] += (n & 1) ? -xn[q] : xn[q];
    }
    const bool mirror = n > 0 && 2 * n != n1;
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      if (g * RT + q >= nr) continue;
      T* o = dst + (r0 + g * RT + q) * n1;
      o[n] = (x0[q] + 2 * (c[q] + s[q])) * scale;
      if (mirror) o[n1 - n] = (x0[q] + 2 * (c[q] - s[q])) * scale;
    }
  }
}

// threads of a CTA with `items` work items: whole warps, at most 256, the passes evenly filled
inline int dft_threads(int items) {
  const int passes = (items + 255) / 256;
  return ((items + passes - 1) / passes + 31) / 32 * 32;
}

}  // namespace

template <typename T> int launch_dft_rows_fwd(const fvim_ctx* c, const T* src, void* dst, size_t rows) {
  typedef typename Cx<T>::t V;
  const size_t smem = (size_t)c->n1 * sizeof(V) + (size_t)2 * (c->n1 / 2 + 1) * Dft<T>::LD * sizeof(T);
  smem_cap(k_dft_rows_fwd<T>, smem);
  launch_chain(c, k_dft_rows_fwd<T>, (unsigned)((rows + Dft<T>::RB - 1) / Dft<T>::RB), dft_threads(4 * c->h1), smem, src, (V*)dst, (const V*)c->tw1, c->n1,
                                                                                c->hs, c->h1, rows);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template <typename T> int launch_dft_cols(const fvim_ctx* c, bool inverse, void* planes, int nplanes) {
  typedef typename Cx<T>::t V;
  constexpr int CT = Dft<T>::CT, CC = Dft<T>::CC;
  const size_t smem = (size_t)c->n2 * sizeof(V) + (size_t)2 * (c->n2 / 2 + 1) * CT * sizeof(V);
  const int threads = dft_threads(CT / CC * (c->n2 / 2 + 1));
  dim3 grid(c->h1 / CT, nplanes);
  if (inverse) {
    smem_cap(k_dft_cols<T, true>, smem);
    launch_chain(c, k_dft_cols<T, true>, grid, threads, smem, (V*)planes, (const V*)c->tw2, c->n2, c->h1);
  } else {
    smem_cap(k_dft_cols<T, false>, smem);
    launch_chain(c, k_dft_cols<T, false>, grid, threads, smem, (V*)planes, (const V*)c->tw2, c->n2, c->h1);
  }
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template <typename T> int launch_dft_rows_inv(const fvim_ctx* c, const void* src, T* dst, size_t rows, T scale) {
  typedef typename Cx<T>::t V;
  const size_t smem = (size_t)c->n1 * sizeof(V) + (size_t)2 * (c->n1 / 2 + 1) * Dft<T>::LD * sizeof(T);
  smem_cap(k_dft_rows_inv<T>, smem);
  launch_chain(c, k_dft_rows_inv<T>, (unsigned)((rows + Dft<T>::RB - 1) / Dft<T>::RB), dft_threads(4 * (c->n1 / 2 + 1)), smem, (const V*)src, dst, (const V*)c->tw1,
                                                                                c->n1, c->hs, c->h1, rows, scale);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template int launch_dft_rows_fwd<float>(const fvim_ctx*, const float*, void*, size_t);
template int launch_dft_rows_fwd<double>(const fvim_ctx*, const double*, void*, size_t);
template int launch_dft_cols<float>(const fvim_ctx*, bool, void*, int);
template int launch_dft_cols<double>(const fvim_ctx*, bool, void*, int);
template int launch_dft_rows_inv<float>(const fvim_ctx*, const void*, float*, size_t, float);
template int launch_dft_rows_inv<double>(const fvim_ctx*, const void*, double*, size_t, double);
