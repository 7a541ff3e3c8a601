// Compile-time-length variants of the register-resident in-plane FFT kernels (fft.cu has
// the runtime-length ones).  Same data layouts, same arithmetic, same results up to the
// order of operations inside the butterflies; chosen by the launchers for 16 <= N <= 1024.
#include <algorithm>

#include "fvim_internal.cuh"

namespace {

template <typename T>
__device__ __forceinline__ void hooke6_ct(const T* e, T* w, T lam, T mu) {
  const T tr = e[0] + e[1] + e[2];
  w[0] = lam * tr + 2 * mu * e[0];
  w[1] = lam * tr + 2 * mu * e[1];
  w[2] = lam * tr + 2 * mu * e[2];
  w[3] = 2 * mu * e[3];
  w[4] = 2 * mu * e[4];
  w[5] = 2 * mu * e[5];
}

// interleaved columns: entry p of column f at buf[p * KC + f]
template <typename V> struct ColSm {
  V* buf;
  int kc, f;
  __device__ __forceinline__ void put(int, int p, V x) const { buf[p * kc + f] = x; }
  __device__ __forceinline__ V get(int, int p) const { return buf[p * kc + f]; }
};
// Row exchange layout: transform g of a row at buf[g * LD + idx(p)].  8-byte entries on rows
// of 128 or more: no padding, entry p at p ^ ((p >> 3) & 15) (a permutation inside each
// aligned block of 16), so that a half-warp's accesses of the radix-8 stage writes (stride 8)
// and of the contiguous reads both fall on 16 distinct bank pairs; otherwise one pad slot
// every 8 entries (p + p / 8), which leaves the contiguous 8-byte reads two-way conflicted
// but suits 16-byte entries and rows shorter than a half-warp.
template <typename V, int N> struct RowLayout {
  static constexpr bool swz = sizeof(V) == 8 && N >= 128;
  static constexpr int LD = swz ? N : N + N / 8;
  static __device__ __forceinline__ int idx(int p) { return swz ? (p ^ ((p >> 3) & 15)) : p + (p >> 3); }
};
template <typename V, int N> struct RowSm {
  V* buf;
  __device__ __forceinline__ void put(int g, int p, V x) const {
    buf[g * RowLayout<V, N>::LD + RowLayout<V, N>::idx(p)] = x;
  }
  __device__ __forceinline__ V get(int g, int p) const { return buf[g * RowLayout<V, N>::LD + RowLayout<V, N>::idx(p)]; }
};

// Order of the passes: a pass ends with its last planes in L2, so the next one over whole planes
// starts with those and runs backwards (forward rows up, forward columns down; inverse columns up,
// inverse rows down, whose output goes past with streaming stores: an apply does not read it again,
// and the solvers' residual pass, which does, takes as long after plain ones: 128 x 128 x 16 and 256 x 256
// x 16 plastic solves 1124 and 2412 us against 1124 and 2410, 512 x 512 x 64 applies 651 against 652).
// Fields below the size of L2 do not care; 512 x 512 x 64: columns 126 -> 123 us, inverse rows 150
// -> 142; inverse rows of the Boussinesq field at 512 x 512 x 32 80 -> 71.
template <bool DOWN> __device__ __forceinline__ int order_y() { return DOWN ? gridDim.y - 1 - blockIdx.y : blockIdx.y; }
template <bool DOWN> __device__ __forceinline__ int order_x() { return DOWN ? gridDim.x - 1 - blockIdx.x : blockIdx.x; }

template <typename T, bool INV, int N>
__global__ void __launch_bounds__(512) k_cols_ct(typename Cx<T>::t* __restrict__ planes,
                                                 const typename Cx<T>::t* __restrict__ tw, int h1, int kc,
                                                 const int* __restrict__ zr) {
  chain_begin();
  typedef typename Cx<T>::t V;
  const int plane = order_y<!INV>();
  if (zr && (plane / 6 < zr[0] || plane / 6 >= zr[1])) return;  // layer without input
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8;
  const int f = threadIdx.x % kc, t = threadIdx.x / kc;
  V* col = planes + (size_t)plane * N * h1 + (size_t)blockIdx.x * kc + f;
  V v[1][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[0][m] = col[(size_t)(t + m * T8) * h1];
  ColSm<V> sm{reinterpret_cast<V*>(smraw), kc, f};
  fft_ct<V, INV, N, 1, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 8; ++m) col[(size_t)(t + m * T8) * h1] = v[0][m];
}

// FP32 column FFTs with 16-byte global accesses: a thread owns two adjacent columns (one
// float4 per row holds both), so every load and store moves 16 bytes; CW columns per CTA
// (CW = 16: every row access of a CTA is one whole 128-byte line).
// Interleaved exchange: entry p of column c at buf[p * CW + c].
template <int CW> struct ColPairSm {
  float2* buf;
  int f2;  // column pair
  __device__ __forceinline__ void put(int g, int p, float2 x) const { buf[p * CW + 2 * f2 + g] = x; }
  __device__ __forceinline__ float2 get(int g, int p) const { return buf[p * CW + 2 * f2 + g]; }
};

}  // namespace
// 1024-point columns, 8 per CTA: fewer table reads than the products apart; apply at 1024 x 1024 x 32
// 1591 -> 1547 us
template <> struct UseBf2<float2, 1024, ColPairSm<8>> {
  static constexpr bool v = true;
};
namespace {

// 16-byte load that asks L2 for the whole 128-byte line: the other half of a 64-byte row segment is
// the neighbouring CTA's
__device__ __forceinline__ float4 ld_line(const float4* p) {
  float4 v;
  asm volatile("ld.global.L2::128B.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

template <int N, int CW> struct ColsV {
  static constexpr int threads = N / 16 * CW;
  static constexpr int min_blocks = CW == 16 ? 1024 / threads : (N >= 1024 ? 2 : 1);  // 64 registers
};

// one CW-column block of one plane: tid in [0, N / 16 * CW), sm the block's [N][CW] exchange
// area; a group that has no block (live false) takes part in the exchange barriers only
template <bool INV, int N, int CW>
__device__ __forceinline__ void cols_v_body(float2* __restrict__ planes, const float2* __restrict__ tw, int h1,
                                            size_t plane, int cblk, int tid, float2* sm, bool live) {
  constexpr int T8 = N / 8, NP = CW / 2;
  const int f2 = tid % NP, t = tid / NP;
  float4* col = reinterpret_cast<float4*>(planes + plane * N * h1 + (size_t)cblk * CW + 2 * f2);
  const size_t rs = (size_t)h1 / 2;  // row stride in float4
  float2 v[2][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const float4* src = col + (size_t)(t + m * T8) * rs;
    const float4 a = live ? (CW < 16 ? ld_line(src) : *src) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[0][m] = make_float2(a.x, a.y);
    v[1][m] = make_float2(a.z, a.w);
  }
  ColPairSm<CW> x{sm, f2};
  fft_ct<float2, INV, N, 2, 1>(v, t, x, tw);
  if (live) {
#pragma unroll
    for (int m = 0; m < 8; ++m)
      col[(size_t)(t + m * T8) * rs] = make_float4(v[0][m].x, v[0][m].y, v[1][m].x, v[1][m].y);
  }
}

template <bool INV, int N, int CW>
__global__ void __launch_bounds__(ColsV<N, CW>::threads, ColsV<N, CW>::min_blocks)
    k_cols_v(float2* __restrict__ planes, const float2* __restrict__ tw, int h1, const int* __restrict__ zr) {
  chain_begin();
  const int plane = order_y<!INV>();
  if (zr && (plane / 6 < zr[0] || plane / 6 >= zr[1])) return;  // layer without input
  extern __shared__ __align__(16) unsigned char smraw[];
  cols_v_body<INV, N, CW>(planes, tw, h1, plane, blockIdx.x, threadIdx.x, reinterpret_cast<float2*>(smraw), true);
}

// Surface displacement of a pressure, column pass fused: forward FFT along x2 of kc k1
// columns, multiplication by the surface compliance u3_hat = (1 - nu) / (mu q) p_hat (zero on
// mode 0 and on the Nyquist row k2 = N2/2, as the Boussinesq kernel), inverse FFT, in one
// kernel (a column is whole inside the CTA).  The row passes stay separate.
template <typename T, int N>
__global__ void __launch_bounds__(512) k_cols_conv(typename Cx<T>::t* __restrict__ plane,
                                                   const typename Cx<T>::t* __restrict__ tw, int h1, int kc, T w1,
                                                   T w2, T nu, T mu) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8;
  const int f = threadIdx.x % kc, t = threadIdx.x / kc;
  const int k1 = blockIdx.x * kc + f;
  V* col = plane + k1;
  V v[1][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[0][m] = col[(size_t)(t + m * T8) * h1];
  ColSm<V> sm{reinterpret_cast<V*>(smraw), kc, f};
  fft_ct<V, false, N, 1, 1>(v, t, sm, tw);
  const T q1 = w1 * (T)k1;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k2 = t + m * T8;
    const int k2s = k2 < N / 2 ? k2 : k2 - N;
    const T q2 = w2 * (T)k2s;
    const T q = sqrt(q1 * q1 + q2 * q2);
    const bool none = (k1 == 0 && k2 == 0) || k2 == N / 2;
    v[0][m] = none ? mk<V>(0, 0) : cscale(v[0][m], ((T)1 - nu) / (mu * q));
  }
  __syncthreads();  // the exchange area is reused by the inverse transform
  fft_ct<V, true, N, 1, 1>(v, t, sm, tw);
#pragma unroll
  for (int m = 0; m < 8; ++m) col[(size_t)(t + m * T8) * h1] = v[0][m];
}

template <typename V>
__device__ __forceinline__ void split_pair_ct(V zk, V zmk, V& A, V& B) {
  typedef decltype(V::x) T;
  const V c = cconj(zmk);
  const V s = cadd(zk, c), d = csub(zk, c);
  A = cscale(s, (T)0.5);
  B = mk<V>((T)0.5 * d.y, (T)-0.5 * d.x);
}

// Forward rows straight from global memory (FP64, and FP32 rows of 16 and 32 points): the Hooke
// constants come halved (hlam = lam / 2, hmu2 = mu), which is the 1/2 of the separation.  NF = 3:
// a thread runs the row's three pair transforms; NF = 1: one of them (blockIdx.z), for grids whose
// rows would leave most of the FP64 pipes idle (an FP64 instruction holds its pipe for 64 cycles
// however few warps there are).  The mirrored half of a spectrum comes from another thread's upper
// slots through shared memory.
template <typename T, int N, int NF>
__global__ void __launch_bounds__(256) k_rows_fwd6_ct(const T* __restrict__ eps_p, typename Cx<T>::t* __restrict__ spec,
                                                      T* __restrict__ nq, const typename Cx<T>::t* __restrict__ tw,
                                                      int n2, int rb, int z0, T hlam, T hmu2, const int* __restrict__ zr) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8, LD = RowLayout<V, N>::LD, H1 = N / 2;
  const int r = threadIdx.x / T8, t = threadIdx.x % T8;
  const int z = z0 + blockIdx.y;
  if (zr && (z < zr[0] || z >= zr[1])) return;  // layer without input
  const int x2 = blockIdx.x * rb + r;
  const int g0 = NF == 3 ? 0 : blockIdx.z;
  V v[NF][8];
  const T* src = eps_p + ((size_t)z * 6 * n2 + x2) * N + t;
  const size_t cs = (size_t)n2 * N;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const T* e = src + m * T8;
    if (NF == 3) {
      const T e0 = e[0], e1 = e[cs], e2 = e[2 * cs];
      const T ltr = hlam * (e0 + e1 + e2);
      v[0][m] = mk<V>(ltr + hmu2 * e0, ltr + hmu2 * e1);
      v[NF / 3][m] = mk<V>(ltr + hmu2 * e2, hmu2 * e[3 * cs]);
      v[2 * (NF / 3)][m] = mk<V>(hmu2 * e[4 * cs], hmu2 * e[5 * cs]);
    } else if (g0 == 2) {
      v[0][m] = mk<V>(hmu2 * e[4 * cs], hmu2 * e[5 * cs]);
    } else {
      const T e0 = e[0], e1 = e[cs], e2 = e[2 * cs];
      const T ltr = hlam * (e0 + e1 + e2);
      v[0][m] = g0 == 0 ? mk<V>(ltr + hmu2 * e0, ltr + hmu2 * e1) : mk<V>(ltr + hmu2 * e2, hmu2 * e[3 * cs]);
    }
  }
  RowSm<V, N> sm{reinterpret_cast<V*>(smraw) + (size_t)r * NF * LD};
  fft_ct<V, false, N, NF, 1>(v, t, sm, tw);
#pragma unroll
  for (int g = 0; g < NF; ++g)
#pragma unroll
    for (int m = 4; m < 8; ++m) sm.put(g, t + m * T8, v[g][m]);
  __syncthreads();
  const size_t ps = (size_t)n2 * H1;
#pragma unroll
  for (int g = 0; g < NF; ++g) {
    V* o = spec + ((size_t)(z * 6 + 2 * (g0 + g)) * n2 + x2) * H1 + t;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      V zm = sm.get(g, (N - t - m * T8) & (N - 1));
      if (m == 0 && t == 0) zm = v[g][0];
      // A = Z + conj Zm, B = (Z - conj Zm) / i
      o[m * T8] = mk<V>(v[g][m].x + zm.x, v[g][m].y - zm.y);
      o[ps + m * T8] = mk<V>(v[g][m].y + zm.y, zm.x - v[g][m].x);
    }
    if (t == 0) {  // k1 = N1/2: Z there is (A + i B) / 2 with real A, B
      T* q = nq + (size_t)(z * 6 + 2 * (g0 + g)) * n2 + x2;
      q[0] = (T)2 * v[g][4].x;
      q[n2] = (T)2 * v[g][4].y;
    }
  }
}

// inverse row FFTs of row x2 of layer z (thread t of the row's N / 8; sm the row's exchange
// area [NF][LD]): the pair transforms g0 .. g0 + NF - 1 of the row's three
template <typename T, int N, int NF = 3>
__device__ __forceinline__ void rows_inv6_body(const typename Cx<T>::t* __restrict__ spec, const T* __restrict__ nq,
                                               T* __restrict__ out, const typename Cx<T>::t* __restrict__ tw, int n2,
                                               int z, int x2, int t, typename Cx<T>::t* smrow, T nq_scale, T scale, int g0 = 0) {
  typedef typename Cx<T>::t V;
  constexpr int T8 = N / 8, H1 = N / 2;
  V v[NF][8];
#pragma unroll
  for (int g = 0; g < NF; ++g) {
    const int ca = 2 * (g0 + g), cb = ca + 1;
    const V* sa = spec + (((size_t)z * 6 + ca) * n2 + x2) * H1;
    const V* sb = spec + (((size_t)z * 6 + cb) * n2 + x2) * H1;
    V ra[8], rbv[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int k = t + m * T8;
      const int kk = k < H1 ? k : (k > H1 ? N - k : 0);
      ra[m] = sa[kk];
      rbv[m] = sb[kk];
    }
    const T na = nq_scale == (T)0 ? (T)0 : nq_scale * nq[((size_t)z * 6 + ca) * n2 + x2];
    const T nb = nq_scale == (T)0 ? (T)0 : nq_scale * nq[((size_t)z * 6 + cb) * n2 + x2];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int k = t + m * T8;
      V A = ra[m], B = rbv[m];
      if (k > H1) { A = cconj(A); B = cconj(B); }
      if (k == H1) { A = mk<V>(na, 0); B = mk<V>(nb, 0); }
      v[g][m] = cadd(A, cmuli(B));
    }
  }
  RowSm<V, N> sm{smrow};
  fft_ct<V, true, N, NF, 1>(v, t, sm, tw);
#pragma unroll
  for (int g = 0; g < NF; ++g)
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int x1 = t + m * T8;
      __stcs(out + (((size_t)z * 6 + 2 * (g0 + g)) * n2 + x2) * N + x1, v[g][m].x * scale);
      __stcs(out + (((size_t)z * 6 + 2 * (g0 + g) + 1) * n2 + x2) * N + x1, v[g][m].y * scale);
    }
}

template <typename T, int N, int NF>
__global__ void __launch_bounds__(256) k_rows_inv6_ct(const typename Cx<T>::t* __restrict__ spec,
                                                      const T* __restrict__ nq, T* __restrict__ out,
                                                      const typename Cx<T>::t* __restrict__ tw, int n2, int rb, int z0,
                                                      T nq_scale, T scale) {
  chain_begin();
  typedef typename Cx<T>::t V;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int T8 = N / 8, LD = RowLayout<V, N>::LD;
  const int r = threadIdx.x / T8, t = threadIdx.x % T8;
  rows_inv6_body<T, N, NF>(spec, nq, out, tw, n2, z0 + order_y<true>(), blockIdx.x * rb + r, t,
                           reinterpret_cast<V*>(smraw) + (size_t)r * NF * LD, nq_scale, scale, NF == 3 ? 0 : blockIdx.z);
}

// FP32 forward row pass: the CTA's six eps_p rows are staged in shared memory with 16-byte
// cp.async copies (two per thread and component) and read from there in the FFT's strided order;
// the staging area then serves as the FFT exchange area.  The two real rows of a transform are
// separated in registers: thread t holds Z(t + m N/8), m < 8, and fetches only the mirrored
// Z(N - k) of its four k < N/2 through the exchange area.  Bound by instruction issue: index
// arithmetic and the round trip of the whole spectrum through shared memory before the
// separation were a third of the instructions.  512 x 512 x 64: 171 -> 135 us (1024 x 1024 x
// 32: 367 -> 305).
// row stride (floats) of the forward rows' staging area: rows of 64 or 128 points put two or
// four rows in one warp, which would read the same banks; N / 8 extra floats shift each row
// by a warp's span of one row
template <int N> struct StageLd {
  static constexpr int v = N <= 128 ? N + N / 8 : N;
};

// forward row FFTs of rows x2b .. x2b + rb - 1 of layer z by the CTA's rb * N / 8 threads;
// smraw the CTA's staging and exchange area
template <int N>
__device__ __forceinline__ void rows_fwd6_v_body(const float* __restrict__ eps_p, float2* __restrict__ spec,
                                                 float* __restrict__ nq, const float2* __restrict__ tw, int n2, int rb,
                                                 int z, int x2b, float lam, float mu, unsigned char* smraw) {
  constexpr int T8 = N / 8, LD = RowLayout<float2, N>::LD, H1 = N / 2;
  constexpr int SLD = StageLd<N>::v;
  const int r = threadIdx.x / T8, t = threadIdx.x % T8;
  const int x2 = x2b + r;
  float* stg = reinterpret_cast<float*>(smraw);  // [6][rb][SLD]
  {
    // the rb rows of a component are contiguous: rb N / 4 = 2 blockDim float4
    const int j = 4 * threadIdx.x, half = 4 * blockDim.x;
    const float* src = eps_p + ((size_t)z * 6 * n2 + x2b) * N + j;
    float* d0 = stg + j + (j / N) * (SLD - N);
    float* d1 = stg + (j + half) + ((j + half) / N) * (SLD - N);
    const size_t cs = (size_t)n2 * N;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      cp_async_16(d0 + c * rb * SLD, src + c * cs);
      cp_async_16(d1 + c * rb * SLD, src + c * cs + half);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  float2 v[3][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int x1 = t + m * T8;
    float e[6], w[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = stg[((size_t)c * rb + r) * SLD + x1];
    hooke6_ct(e, w, lam, mu);
    v[0][m] = make_float2(w[0], w[1]);
    v[1][m] = make_float2(w[2], w[3]);
    v[2][m] = make_float2(w[4], w[5]);
  }
  __syncthreads();  // staging is dead: the exchange area takes its place
  RowSm<float2, N> sm{reinterpret_cast<float2*>(smraw) + (size_t)r * 3 * LD};
  fft_ct<float2, false, N, 3, 1>(v, t, sm, tw);
  // mirrored halves: Z(N - k) of k = t + m N/8, m < 4, is in the upper half, slots 4..7 of another
  // thread (Z(0) is its own mirror)
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int m = 4; m < 8; ++m) sm.put(g, t + m * T8, v[g][m]);
  __syncthreads();
  float2* o = spec + ((size_t)z * 6 * n2 + x2) * H1 + t;
  const size_t cs = (size_t)n2 * H1;
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float2 zm = sm.get(g, (N - t - m * T8) & (N - 1));
      if (m == 0 && t == 0) zm = v[g][0];
      float2 A, B;
      split_pair_ct(v[g][m], zm, A, B);
      o[2 * g * cs + m * T8] = A;
      o[(2 * g + 1) * cs + m * T8] = B;
    }
  if (t == 0) {
    // k1 = N1/2: Z there is A + i B with real A, B
    float* q = nq + (size_t)z * 6 * n2 + x2;
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      q[(size_t)(2 * g) * n2] = v[g][4].x;
      q[(size_t)(2 * g + 1) * n2] = v[g][4].y;
    }
  }
}

template <int N>
__global__ void __launch_bounds__(256) k_rows_fwd6_v(const float* __restrict__ eps_p, float2* __restrict__ spec,
                                                     float* __restrict__ nq, const float2* __restrict__ tw, int n2,
                                                     int rb, int z0, float lam, float mu, const int* __restrict__ zr) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int z = z0 + blockIdx.y;
  if (zr && (z < zr[0] || z >= zr[1])) return;  // layer without input
  rows_fwd6_v_body<N>(eps_p, spec, nq, tw, n2, rb, z, blockIdx.x * rb, lam, mu, smraw);
}

template <typename K> void smem_attr(K kern, size_t smem) {
  smem_cap(kern, smem);
}

inline int ct_rows(int n1, int n2) {
  int rb = 256 / (n1 >> 3);
  if (rb > 8) rb = 8;
  while (rb > n2) rb >>= 1;
  return rb;
}

template <int N, int CW> void cols_v_launch(const fvim_ctx* c, bool inverse, void* planes, int nplanes, const int* zr) {
  dim3 grid(c->h1 / CW, nplanes);
  const size_t sm = (size_t)N * CW * sizeof(float2);
  if (inverse) {
    smem_attr(k_cols_v<true, N, CW>, sm);
    launch_chain(c, k_cols_v<true, N, CW>, grid, ColsV<N, CW>::threads, sm, (float2*)planes, (const float2*)c->tw2,
                                                                          c->h1, zr);
  } else {
    smem_attr(k_cols_v<false, N, CW>, sm);
    launch_chain(c, k_cols_v<false, N, CW>, grid, ColsV<N, CW>::threads, sm, (float2*)planes, (const float2*)c->tw2,
                                                                           c->h1, zr);
  }
}

template <typename T, int N> void cols_n(const fvim_ctx* c, bool inverse, void* planes, int nplanes, const int* zr) {
  typedef typename Cx<T>::t V;
  if constexpr (sizeof(T) == 4 && N >= 64) {
    // 16 columns per CTA (whole 128-byte rows, N threads); at N = 1024 that is one CTA per SM, whose
    // load, transform and store phases do not overlap: 8 columns, two CTAs
    // (1024 x 1024 x 32: 420 -> 361 us per direction).
    if constexpr (N <= 512) {
      if (c->h1 % 16 == 0) {
        cols_v_launch<N, 16>(c, inverse, planes, nplanes, zr);
        return;
      }
    }
    if (c->h1 % 8 == 0) {
      cols_v_launch<N, 8>(c, inverse, planes, nplanes, zr);
      return;
    }
  }
  int kc = (int)(128 / sizeof(V));  // 128-byte rows
  while (kc > 1 && kc * (N / 8) > 512) kc >>= 1;
  if (kc > c->h1) kc = c->h1;
  const int threads = kc * (N / 8);
  const size_t smem = (size_t)kc * N * sizeof(V);
  dim3 grid(c->h1 / kc, nplanes);
  if (inverse) {
    smem_attr(k_cols_ct<T, true, N>, smem);
    launch_chain(c, k_cols_ct<T, true, N>, grid, threads, smem, (V*)planes, (const V*)c->tw2, c->h1, kc, zr);
  } else {
    smem_attr(k_cols_ct<T, false, N>, smem);
    launch_chain(c, k_cols_ct<T, false, N>, grid, threads, smem, (V*)planes, (const V*)c->tw2, c->h1, kc, zr);
  }
}

// The three pair transforms of a row in separate CTAs: FP64 grids with fewer warps than FP64 pipes
// (four per SM) when one thread runs all three.  With the FP64 stages of
// stage_bf2 and the halved constants the 32 x 32 x 16 FP64 Hertz solve went from 301 to 266 ms.
template <typename T, int N> bool rows_apart(const fvim_ctx* c, int nzs) {
  return sizeof(T) == 8 && (size_t)nzs * c->n2 * (N / 8) / 32 < (size_t)4 * sm_count();
}

template <typename T, int N> void rows_fwd_n(const fvim_ctx* c, const T* eps_p, int z0, int nzs, const int* zr) {
  typedef typename Cx<T>::t V;
  const int rb = ct_rows(N, c->n2);
  if constexpr (sizeof(T) == 4 && N >= 64) {
    const size_t sm = std::max((size_t)rb * 3 * RowLayout<V, N>::LD * sizeof(V), (size_t)6 * rb * StageLd<N>::v * sizeof(T));
    dim3 grid(c->n2 / rb, nzs);
    smem_attr(k_rows_fwd6_v<N>, sm);
    launch_chain(c, k_rows_fwd6_v<N>, grid, rb * (N / 8), sm, (const float*)eps_p, (float2*)c->spec, (float*)c->nq,
                                                            (const float2*)c->tw1, c->n2, rb, z0, (float)c->lam,
                                                            (float)c->mu, zr);
    return;
  }
  auto go = [&](auto kern, int nf) {
    const size_t smem = (size_t)rb * nf * RowLayout<V, N>::LD * sizeof(V);
    smem_attr(kern, smem);
    launch_chain(c, kern, dim3(c->n2 / rb, nzs, 3 / nf), rb * (N / 8), smem, eps_p, (V*)c->spec, (T*)c->nq, (const V*)c->tw1,
                                                                         c->n2, rb, z0, (T)(0.5 * c->lam), (T)c->mu, zr);
  };
  if constexpr (sizeof(T) == 8) {
    if (rows_apart<T, N>(c, nzs)) {
      go(k_rows_fwd6_ct<T, N, 1>, 1);
      return;
    }
  }
  go(k_rows_fwd6_ct<T, N, 3>, 3);
}

template <typename T, int N> void rows_inv_n(const fvim_ctx* c, T* out, T nq_scale, int z0, int nzs) {
  typedef typename Cx<T>::t V;
  int rb = ct_rows(N, c->n2);
  // smaller CTAs in FP32 (128 threads at N = 512 and 1024): 5 instead of 2 per SM at ~100 registers
  if (sizeof(T) == 4 && (rb >= 4 || N >= 1024)) rb = std::max(1, rb / 2);
  const T scale = (T)(1.0 / ((double)N * (double)c->n2));
  auto go = [&](auto kern, int nf) {
    const size_t smem = (size_t)rb * nf * RowLayout<V, N>::LD * sizeof(V);
    smem_attr(kern, smem);
    launch_chain(c, kern, dim3(c->n2 / rb, nzs, 3 / nf), rb * (N / 8), smem, (const V*)c->spec, (const T*)c->nq, out,
                                                                         (const V*)c->tw1, c->n2, rb, z0, nq_scale, scale);
  };
  if constexpr (sizeof(T) == 8) {
    if (rows_apart<T, N>(c, nzs)) {
      go(k_rows_inv6_ct<T, N, 1>, 1);
      return;
    }
  }
  go(k_rows_inv6_ct<T, N, 3>, 3);
}

// ---- grouped launches: every problem of a GrpTable in one launch per pass ---------------
// A CTA finds its problem by the table's CTA offsets and runs the same body as the
// single-problem kernels, so each problem's results are those of its own launch sequence.
// Shapes are chosen so that every N in 64..512 fills the same CTA: forward rows 2048 / N1 rows
// per CTA (256 threads), inverse rows 1024 / N1 rows (128 threads), columns 512 / N2 blocks of
// 16 columns (512 threads, N2 threads per block).
constexpr int kGrpRowsFwdSmem = 2048 * 3 * 9 / 8 * 8;    // = 6 * 2048 * 9 / 8 * 4 bytes of staging
constexpr int kGrpRowsInvSmem = 1024 * 3 * 9 / 8 * 8;
constexpr int kGrpColsSmem = 512 * 16 * 8;

template <int N> __device__ __forceinline__ void grp_rows_fwd_case(const GrpProb& P, int local, unsigned char* sm) {
  const int rb = 2048 / N, nrb = P.n2 / rb;
  const int z = local / nrb, x2b = (local - z * nrb) * rb;
  rows_fwd6_v_body<N>(P.eps, P.spec, P.nq, P.tw1, P.n2, rb, z, x2b, P.lam, P.mu, sm);
}

__global__ void __launch_bounds__(256) k_grp_rows_fwd(const __grid_constant__ GrpTable tab) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int pi = grp_find(tab, blockIdx.x);
  const GrpProb& P = tab.p[pi];
  const int local = (int)blockIdx.x - tab.start[pi];
  switch (P.n1) {
    case 64: grp_rows_fwd_case<64>(P, local, smraw); break;
    case 128: grp_rows_fwd_case<128>(P, local, smraw); break;
    case 256: grp_rows_fwd_case<256>(P, local, smraw); break;
    case 512: grp_rows_fwd_case<512>(P, local, smraw); break;
    default: break;
  }
}

template <int N> __device__ __forceinline__ void grp_rows_inv_case(const GrpProb& P, int local, unsigned char* sm) {
  constexpr int T8 = N / 8, LD = RowLayout<float2, N>::LD;
  const int rb = 1024 / N, nrb = P.n2 / rb;
  const int z = local / nrb, r = threadIdx.x / T8, t = threadIdx.x % T8;
  const int x2 = (local - z * nrb) * rb + r;
  rows_inv6_body<float, N>(P.spec, P.nq, P.out, P.tw1, P.n2, z, x2, t,
                           reinterpret_cast<float2*>(sm) + (size_t)r * 3 * LD, P.nq_scale, P.scale);
}

__global__ void __launch_bounds__(128) k_grp_rows_inv(const __grid_constant__ GrpTable tab) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cta = order_x<true>();
  const int pi = grp_find(tab, cta);
  const GrpProb& P = tab.p[pi];
  const int local = cta - tab.start[pi];
  switch (P.n1) {
    case 64: grp_rows_inv_case<64>(P, local, smraw); break;
    case 128: grp_rows_inv_case<128>(P, local, smraw); break;
    case 256: grp_rows_inv_case<256>(P, local, smraw); break;
    case 512: grp_rows_inv_case<512>(P, local, smraw); break;
    default: break;
  }
}

template <bool INV, int N>
__device__ __forceinline__ void grp_cols_case(const GrpProb& P, int local, unsigned char* sm) {
  constexpr int G = 512 / N;  // column blocks per CTA, N threads each
  const int g = threadIdx.x / N, tid = threadIdx.x - g * N;
  const int ncb = P.h1 / 16, items = P.nz * 6 * ncb;
  const int item = local * G + g;
  const bool live = item < items;
  const int plane = live ? item / ncb : 0, cblk = live ? item - plane * ncb : 0;
  cols_v_body<INV, N, 16>(P.spec, P.tw2, P.h1, (size_t)plane, cblk, tid,
                          reinterpret_cast<float2*>(sm) + (size_t)g * N * 16, live);
}

template <bool INV> __global__ void __launch_bounds__(512, 2) k_grp_cols(const __grid_constant__ GrpTable tab) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cta = order_x<!INV>();
  const int pi = grp_find(tab, cta);
  const GrpProb& P = tab.p[pi];
  const int local = cta - tab.start[pi];
  switch (P.n2) {
    case 64: grp_cols_case<INV, 64>(P, local, smraw); break;
    case 128: grp_cols_case<INV, 128>(P, local, smraw); break;
    case 256: grp_cols_case<INV, 256>(P, local, smraw); break;
    case 512: grp_cols_case<INV, 512>(P, local, smraw); break;
    default: break;
  }
}

}  // namespace

#define FVIM_CT_SIZES(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)

template <typename T> bool launch_cols_ct(const fvim_ctx* c, bool inverse, void* planes, int nplanes, const int* zr) {
#define CASE(N)                                 \
  if (c->n2 == N) {                             \
    cols_n<T, N>(c, inverse, planes, nplanes, zr); \
    return true;                                \
  }
  FVIM_CT_SIZES(CASE)
#undef CASE
  return false;
}

template <typename T, int N> void cols_conv_n(const fvim_ctx* c) {
  typedef typename Cx<T>::t V;
  int kc = (int)(128 / sizeof(V));  // 128-byte rows
  while (kc > 1 && kc * (N / 8) > 512) kc >>= 1;
  if (kc > c->h1) kc = c->h1;
  const size_t smem = (size_t)kc * N * sizeof(V);
  smem_attr(k_cols_conv<T, N>, smem);
  const double two_pi = 6.283185307179586476925;
  launch_chain(c, k_cols_conv<T, N>, c->h1 / kc, kc * (N / 8), smem, 
      (V*)c->surf, (const V*)c->tw2, c->h1, kc, (T)(two_pi / c->L1), (T)(two_pi / c->L2), (T)c->nu, (T)c->mu);
}

template <typename T> bool launch_cols_conv_ct(const fvim_ctx* c) {
#define CASE(N)              \
  if (c->n2 == N) {          \
    cols_conv_n<T, N>(c);    \
    return true;             \
  }
  FVIM_CT_SIZES(CASE)
#undef CASE
  return false;
}

template <typename T> bool launch_rows_fwd6_ct(const fvim_ctx* c, const T* eps_p, int z0, int nzs, const int* zr) {
#define CASE(N)                              \
  if (c->n1 == N) {                          \
    rows_fwd_n<T, N>(c, eps_p, z0, nzs, zr); \
    return true;                             \
  }
  FVIM_CT_SIZES(CASE)
#undef CASE
  return false;
}

template <typename T> bool launch_rows_inv6_ct(const fvim_ctx* c, T* out, T nq_scale, int z0, int nzs) {
#define CASE(N)                                     \
  if (c->n1 == N) {                                 \
    rows_inv_n<T, N>(c, out, nq_scale, z0, nzs);    \
    return true;                                    \
  }
  FVIM_CT_SIZES(CASE)
#undef CASE
  return false;
}

template bool launch_cols_ct<float>(const fvim_ctx*, bool, void*, int, const int*);
template bool launch_cols_conv_ct<float>(const fvim_ctx*);
template bool launch_cols_conv_ct<double>(const fvim_ctx*);
template bool launch_cols_ct<double>(const fvim_ctx*, bool, void*, int, const int*);
template bool launch_rows_fwd6_ct<float>(const fvim_ctx*, const float*, int, int, const int*);
template bool launch_rows_fwd6_ct<double>(const fvim_ctx*, const double*, int, int, const int*);
template bool launch_rows_inv6_ct<float>(const fvim_ctx*, float*, float, int, int);
template bool launch_rows_inv6_ct<double>(const fvim_ctx*, double*, double, int, int);

int launch_grp_rows_fwd(GrpTable& t, cudaStream_t s) {
  int b = 0;
  for (int i = 0; i < t.n; ++i) {
    t.start[i] = b;
    b += t.p[i].nz * (t.p[i].n2 / (2048 / t.p[i].n1));
  }
  t.start[t.n] = b;
  if (b == 0) return FVIM_OK;
  smem_attr(k_grp_rows_fwd, kGrpRowsFwdSmem);
  launch_chain_on(s, true, k_grp_rows_fwd, b, 256, kGrpRowsFwdSmem, t);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

int launch_grp_rows_inv(GrpTable& t, cudaStream_t s) {
  int b = 0;
  for (int i = 0; i < t.n; ++i) {
    t.start[i] = b;
    b += t.p[i].nz * (t.p[i].n2 / (1024 / t.p[i].n1));
  }
  t.start[t.n] = b;
  if (b == 0) return FVIM_OK;
  smem_attr(k_grp_rows_inv, kGrpRowsInvSmem);
  launch_chain_on(s, true, k_grp_rows_inv, b, 128, kGrpRowsInvSmem, t);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

int launch_grp_cols(GrpTable& t, bool inverse, cudaStream_t s) {
  int b = 0;
  for (int i = 0; i < t.n; ++i) {
    t.start[i] = b;
    const int items = t.p[i].nz * 6 * (t.p[i].h1 / 16), per = 512 / t.p[i].n2;
    b += (items + per - 1) / per;
  }
  t.start[t.n] = b;
  if (b == 0) return FVIM_OK;
  if (inverse) {
    smem_attr(k_grp_cols<true>, kGrpColsSmem);
    launch_chain_on(s, true, k_grp_cols<true>, b, 512, kGrpColsSmem, t);
  } else {
    smem_attr(k_grp_cols<false>, kGrpColsSmem);
    launch_chain_on(s, true, k_grp_cols<false>, b, 512, kGrpColsSmem, t);
  }
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}
