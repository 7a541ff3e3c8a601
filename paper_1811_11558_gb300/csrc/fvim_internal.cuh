// Internal definitions shared by the CUDA translation units of libfvim.
// Not part of the public ABI (see include/fvim.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <utility>

#include "fvim.h"

// ---------------------------------------------------------------------------
// complex helpers (float2 / double2)
// ---------------------------------------------------------------------------
template <typename T> struct Cx;
template <> struct Cx<float> { typedef float2 t; };
template <> struct Cx<double> { typedef double2 t; };

template <typename V> __host__ __device__ __forceinline__ V mk(decltype(V::x) a, decltype(V::x) b) {
  V r; r.x = a; r.y = b; return r;
}
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  return mk<V>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename V> __device__ __forceinline__ V cconj(V a) { return mk<V>(a.x, -a.y); }
template <typename V> __device__ __forceinline__ V cscale(V a, decltype(V::x) s) { return mk<V>(a.x * s, a.y * s); }
// multiply by i
template <typename V> __device__ __forceinline__ V cmuli(V a) { return mk<V>(-a.y, a.x); }
// a + s*b (s real)
template <typename V> __device__ __forceinline__ V caxpy(V a, decltype(V::x) s, V b) {
  return mk<V>(a.x + s * b.x, a.y + s * b.y);
}
// a + s*i*b (s real): two scalar multiply-adds, the swap and the sign folded into them
template <typename V> __device__ __forceinline__ V caxpy_i(V a, decltype(V::x) s, V b) {
  return mk<V>(a.x - s * b.y, a.y + s * b.x);
}

#if defined(__CUDA_ARCH__) && (__CUDA_ARCH__ >= 1000) && !defined(FVIM_NO_F32X2)
// Blackwell packed FP32 pairs (add/sub/mul/fma .f32x2): one instruction per FP32 complex
// add, subtract, real scale or real axpy, each lane rounded as its scalar counterpart.
__device__ __forceinline__ unsigned long long f2pack(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 f2unpack(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pack(a)), "l"(f2pack(b)));
  return f2unpack(d);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pack(a)), "l"(f2pack(b)));
  return f2unpack(d);
}
__device__ __forceinline__ float2 cscale(float2 a, float s) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pack(a)), "l"(f2pack(make_float2(s, s))));
  return f2unpack(d);
}
__device__ __forceinline__ float2 caxpy(float2 a, float s, float2 b) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2pack(make_float2(s, s))), "l"(f2pack(b)), "l"(f2pack(a)));
  return f2unpack(d);
}
#endif

// ---------------------------------------------------------------------------
// Shared-memory FFT: batched, in place, Stockham autosort with radix 8/4/2
// stages.  Every thread of the block takes part; at most MAXI work items (one
// radix-R butterfly each) per thread and stage, so the caller must launch at
// least ceil(nfft * n / rmin(n) / MAXI) threads.  tw[k] = exp(-2 pi i k / n).
// ---------------------------------------------------------------------------
__host__ __device__ inline int fft_radix(int m) {
  // radix of the next stage for a remaining length m (plans 8..8 then 4/4 or 4 or 2)
  if (m == 2) return 2;
  if (m == 4) return 4;
  if (m == 16) return 4;           // 16 = 4 x 4 instead of 8 x 2
  if (m % 8 == 0) return 8;
  return 4;
}
__host__ __device__ inline int fft_rmin(int n) {
  int rmin = 8, m = n;
  while (m > 1) { int r = fft_radix(m); if (r < rmin) rmin = r; m /= r; }
  return rmin;
}

template <typename V, bool INV>
__device__ __forceinline__ V twiddle(const V* tw, int idx) {
  V w = tw[idx];
  if (INV) w.y = -w.y;
  return w;
}

template <typename V, bool INV>
__device__ __forceinline__ void dft2(V& a, V& b) { V t = a; a = cadd(t, b); b = csub(t, b); }

template <typename V, bool INV>
__device__ __forceinline__ void dft4(V* v) {
  V a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
  V b0 = cadd(v[1], v[3]), b1 = csub(v[1], v[3]);
  v[0] = cadd(a0, b0);
  v[2] = csub(a0, b0);
  // a1 -/+ i b1 (forward W4 = -i, inverse +i), the swap folded into the adds
  if (INV) {
    v[1] = mk<V>(a1.x - b1.y, a1.y + b1.x);
    v[3] = mk<V>(a1.x + b1.y, a1.y - b1.x);
  } else {
    v[1] = mk<V>(a1.x + b1.y, a1.y - b1.x);
    v[3] = mk<V>(a1.x - b1.y, a1.y + b1.x);
  }
}

template <typename V, bool INV>
__device__ __forceinline__ void dft8(V* v) {
  typedef decltype(V::x) T;
  const T r = (T)0.70710678118654752440;
  V e[4] = {v[0], v[2], v[4], v[6]};
  V o[4] = {v[1], v[3], v[5], v[7]};
  dft4<V, INV>(e);
  dft4<V, INV>(o);
  // last level v[m] = e[m] + W8^m o[m], v[m + 4] = e[m] - W8^m o[m]: W8 = r (1 -/+ i) and W8^3 =
  // r (-1 -/+ i) as a sum and a multiply-add per component
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  const V x2 = INV ? mk<V>(-o[2].y, o[2].x) : mk<V>(o[2].y, -o[2].x);
  v[2] = cadd(e[2], x2);
  v[6] = csub(e[2], x2);
  const V x1 = INV ? mk<V>(o[1].x - o[1].y, o[1].x + o[1].y) : mk<V>(o[1].x + o[1].y, o[1].y - o[1].x);
  v[1] = caxpy(e[1], r, x1);
  v[5] = caxpy(e[1], -r, x1);
  const V x3 = INV ? mk<V>(-(o[3].x + o[3].y), o[3].x - o[3].y) : mk<V>(o[3].y - o[3].x, -(o[3].x + o[3].y));
  v[3] = caxpy(e[3], r, x3);
  v[7] = caxpy(e[3], -r, x3);
}

template <typename V, bool INV, int R, int MAXI>
__device__ __forceinline__ void fft_stage(V* buf, int n, int nfft, int fstride, int Ns, const V* tw) {
  const int per = n / R;
  const int items = nfft * per;
  V v[MAXI][R];
#pragma unroll
  for (int it = 0; it < MAXI; ++it) {
    const int w = threadIdx.x + it * blockDim.x;
    if (w < items) {
      const int f = w / per, j = w - f * per;
      const V* b = buf + (size_t)f * fstride;
#pragma unroll
      for (int r = 0; r < R; ++r) v[it][r] = b[j + r * per];
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < MAXI; ++it) {
    const int w = threadIdx.x + it * blockDim.x;
    if (w < items) {
      const int f = w / per, j = w - f * per;
      const int k = j % Ns;
      const int step = n / (Ns * R);
#pragma unroll
      for (int r = 1; r < R; ++r) v[it][r] = cmul(v[it][r], twiddle<V, INV>(tw, (r * k * step) & (n - 1)));
      if (R == 8) dft8<V, INV>(v[it]);
      else if (R == 4) dft4<V, INV>(v[it]);
      else dft2<V, INV>(v[it][0], v[it][1]);
      V* b = buf + (size_t)f * fstride;
      const int base = (j / Ns) * Ns * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) b[base + r * Ns] = v[it][r];
    }
  }
  __syncthreads();
}

// nfft transforms of length n (power of two >= 2) in shared memory, FFT f at
// buf + f * fstride.  Unnormalised; INV uses exp(+2 pi i k/n).
template <typename V, bool INV, int MAXI>
__device__ void block_fft(V* buf, int n, int nfft, int fstride, const V* tw) {
  int Ns = 1;
  int m = n;
  while (m > 1) {
    const int R = fft_radix(m);
    if (R == 8) fft_stage<V, INV, 8, MAXI>(buf, n, nfft, fstride, Ns, tw);
    else if (R == 4) fft_stage<V, INV, 4, MAXI>(buf, n, nfft, fstride, Ns, tw);
    else fft_stage<V, INV, 2, MAXI>(buf, n, nfft, fstride, Ns, tw);
    Ns *= R;
    m /= R;
  }
}

// ---------------------------------------------------------------------------
// Register-resident Stockham FFT (n >= 8): thread t of an FFT holds the 8 strided
// elements x[t + m n/8], m = 0..7, for the whole transform.  A stage of radix R
// (8, 4 or 2; plan of fft_radix) runs 1, 2 or 4 butterflies per thread on those
// registers and reports, for every register slot, the natural index its result
// belongs to; between stages the values go through shared memory.  After the last
// stage slot m holds the output at index t + m n/8 (natural order).
// ---------------------------------------------------------------------------
template <typename V, bool INV>
__device__ __forceinline__ void reg_stage(V (&v)[8], int (&pos)[8], int t, int n, int R, int Ns, const V* tw) {
  const int T8 = n >> 3;
  if (R == 8) {
    const int k = t & (Ns - 1);
    const int step = n / (Ns * 8);
#pragma unroll
    for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], twiddle<V, INV>(tw, (r * k * step) & (n - 1)));
    dft8<V, INV>(v);
    const int base = (t / Ns) * Ns * 8 + k;
#pragma unroll
    for (int r = 0; r < 8; ++r) pos[r] = base + r * Ns;
  } else if (R == 4) {
    const int step = n / (Ns * 4);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int b = t + g * T8;
      const int k = b & (Ns - 1);
      V u[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) u[r] = v[2 * r + g];
#pragma unroll
      for (int r = 1; r < 4; ++r) u[r] = cmul(u[r], twiddle<V, INV>(tw, (r * k * step) & (n - 1)));
      dft4<V, INV>(u);
      const int base = (b / Ns) * Ns * 4 + k;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        v[2 * r + g] = u[r];
        pos[2 * r + g] = base + r * Ns;
      }
    }
  } else {
    const int step = n / (Ns * 2);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int b = t + m * T8;
      const int k = b & (Ns - 1);
      V a = v[m], c = cmul(v[m + 4], twiddle<V, INV>(tw, (k * step) & (n - 1)));
      v[m] = cadd(a, c);
      v[m + 4] = csub(a, c);
      const int base = (b / Ns) * Ns * 2 + k;
      pos[m] = base;
      pos[m + 4] = base + Ns;
    }
  }
}

// ---------------------------------------------------------------------------
// The same register-resident Stockham FFT with the length N known at compile time:
// the stage list is unrolled, the first stage has no twiddles, and every index is a
// shift or a mask.  NF transforms per thread share each shared-memory exchange; the
// exchange layout is the caller's (Sm::put / Sm::get).  After the call slot m of
// transform f holds the output at index t + m N/8.
// ---------------------------------------------------------------------------
template <int REM> struct StageRadix {
  static constexpr int v = (REM == 2) ? 2 : ((REM == 4 || REM == 16) ? 4 : ((REM % 8 == 0) ? 8 : 4));
};

// twiddles w^1..w^7 of a radix-8 butterfly (w = tw[idx]) from three table reads: w, w^2, w^4
// are read, w^3 = w w^2, w^5 = w^4 w, w^6 = w^4 w^2, w^7 = w^4 w^3 (three table reads instead of
// seven: the reads of one stage are scattered, a table read per product was the costly part)
template <typename V, bool INV>
__device__ __forceinline__ void twiddles8(const V* __restrict__ tw, int idx, V (&w)[8]) {
  w[1] = twiddle<V, INV>(tw, idx);
  w[2] = twiddle<V, INV>(tw, 2 * idx);
  w[4] = twiddle<V, INV>(tw, 4 * idx);
  w[3] = cmul(w[1], w[2]);
  w[5] = cmul(w[4], w[1]);
  w[6] = cmul(w[4], w[2]);
  w[7] = cmul(w[4], w[3]);
}

template <typename V, bool INV, int N, int R, int NS>
__device__ __forceinline__ void stage_prod(V (&v)[8], int (&pos)[8], int t, const V* __restrict__ tw) {
  constexpr int T8 = N / 8;
  if constexpr (R == 8) {
    const int k = t & (NS - 1);
    if constexpr (NS > 1) {
      constexpr int step = N / (NS * 8);
      V w[8];
      twiddles8<V, INV>(tw, k * step, w);
#pragma unroll
      for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], w[r]);
    }
    dft8<V, INV>(v);
    const int base = (t / NS) * NS * 8 + k;
#pragma unroll
    for (int r = 0; r < 8; ++r) pos[r] = base + r * NS;
  } else if constexpr (R == 4) {
    constexpr int step = N / (NS * 4);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int b = t + g * T8;
      const int k = b & (NS - 1);
      V u[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) u[r] = v[2 * r + g];
      if constexpr (NS > 1) {
        // w, w^2 read, w^3 = w w^2
        const V w1 = twiddle<V, INV>(tw, k * step), w2 = twiddle<V, INV>(tw, 2 * k * step);
        u[1] = cmul(u[1], w1);
        u[2] = cmul(u[2], w2);
        u[3] = cmul(u[3], cmul(w1, w2));
      }
      dft4<V, INV>(u);
      const int base = (b / NS) * NS * 4 + k;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        v[2 * r + g] = u[r];
        pos[2 * r + g] = base + r * NS;
      }
    }
  } else {
    constexpr int step = N / (NS * 2);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int b = t + m * T8;
      const int k = b & (NS - 1);
      V c = v[m + 4];
      if constexpr (NS > 1) c = cmul(c, twiddle<V, INV>(tw, k * step));
      const V a = v[m];
      v[m] = cadd(a, c);
      v[m + 4] = csub(a, c);
      const int base = (b / NS) * NS * 2 + k;
      pos[m] = base;
      pos[m + 4] = base + NS;
    }
  }
}

// Radix-2 butterfly with the twiddle inside: t = a + w b, s = a - w b as multiply-adds.  FP64: s = 2 a -
// t, six of them (a separate complex product and two complex sums are eight operations).  s then carries
// the rounding of t, which shows in FP32, so there s takes its own two multiply-adds per component:
// rms error of a 1024-point transform of noise 1.20e-7 -> 1.11e-7 (products apart: 1.17e-7).  In FP64 the
// whole operator stays below its error with the products apart (128 x 128 x 8: 6.6e-16 -> 6.4e-16), and
// direct differences cost 10 % of it (128 x 128 x 126: 1323 -> 1461 us).
template <typename V> __device__ __forceinline__ void bf2(V& a, V& b, V w) {
  typedef decltype(V::x) T;
  V t;
  t.x = fma(w.x, b.x, fma(-w.y, b.y, a.x));
  t.y = fma(w.x, b.y, fma(w.y, b.x, a.y));
  if constexpr (sizeof(T) == 4) {
    const V c = b;
    b.x = fma(-w.x, c.x, fma(w.y, c.y, a.x));
    b.y = fma(-w.x, c.y, fma(-w.y, c.x, a.y));
  } else {
    b.x = fma((T)2, a.x, -t.x);
    b.y = fma((T)2, a.y, -t.y);
  }
  a = t;
}
// w times -i (forward) or i (inverse)
template <typename V, bool INV> __device__ __forceinline__ V quarter(V w) {
  return INV ? mk<V>(-w.y, w.x) : mk<V>(w.y, -w.x);
}

// One stage of a radix-8, 4 or 2 transform on the eight values of a thread, twiddled stages run
// as radix-2 levels of bf2 (72, 24 and 6 multiply-adds for 8, 4 and 2 values, against 84, 28 and 8
// with the products apart), from four, two or one table reads: w, w^2, w^4 and w W_8.
// FP64 is bound by its pipe (one instruction per warp and 64 cycles), so the fewest operations win:
// 128 x 128 x 126 rows 353 -> 319, columns 261 -> 212, inverse rows 317 -> 278 us.  In FP32 the
// levels' longer dependency chains cost more than the operations save (512 x 512 x 64 columns 126
// -> 151 us at 64 registers), so it keeps stage_prod, but for the 8-column CTAs of 1024 points.
template <typename V, bool INV, int N, int R, int NS>
__device__ __forceinline__ void stage_bf2(V (&v)[8], int (&pos)[8], int t, const V* __restrict__ tw) {
  constexpr int T8 = N / 8;
  if constexpr (R == 8) {
    const int k = t & (NS - 1);
    if constexpr (NS > 1) {
      const int idx = k * (N / (NS * 8));
      const V w1 = twiddle<V, INV>(tw, idx), w2 = twiddle<V, INV>(tw, 2 * idx), w4 = twiddle<V, INV>(tw, 4 * idx);
      const V w1e = twiddle<V, INV>(tw, idx + N / 8);
#pragma unroll
      for (int r = 0; r < 4; ++r) bf2(v[r], v[r + 4], w4);
      const V w2q = quarter<V, INV>(w2);
      bf2(v[0], v[2], w2);
      bf2(v[1], v[3], w2);
      bf2(v[4], v[6], w2q);
      bf2(v[5], v[7], w2q);
      bf2(v[0], v[1], w1);
      bf2(v[4], v[5], w1e);
      bf2(v[2], v[3], quarter<V, INV>(w1));
      bf2(v[6], v[7], quarter<V, INV>(w1e));
      // bit-reversed slots hold outputs 0, 4, 2, 6, 1, 5, 3, 7
      const int base = (t / NS) * NS * 8 + k;
      constexpr int out[8] = {0, 4, 2, 6, 1, 5, 3, 7};
      V u[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) u[out[r]] = v[r];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        v[r] = u[r];
        pos[r] = base + r * NS;
      }
    } else {
      dft8<V, INV>(v);
      const int base = t * 8;
#pragma unroll
      for (int r = 0; r < 8; ++r) pos[r] = base + r;
    }
  } else if constexpr (R == 4) {
    constexpr int step = N / (NS * 4);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int b = t + g * T8;
      const int k = b & (NS - 1);
      V u[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) u[r] = v[2 * r + g];
      if constexpr (NS > 1) {
        const V w1 = twiddle<V, INV>(tw, k * step), w2 = twiddle<V, INV>(tw, 2 * k * step);
        bf2(u[0], u[2], w2);
        bf2(u[1], u[3], w2);
        bf2(u[0], u[1], w1);
        bf2(u[2], u[3], quarter<V, INV>(w1));
        const V x = u[1];  // slots hold outputs 0, 2, 1, 3
        u[1] = u[2];
        u[2] = x;
      } else {
        dft4<V, INV>(u);
      }
      const int base = (b / NS) * NS * 4 + k;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        v[2 * r + g] = u[r];
        pos[2 * r + g] = base + r * NS;
      }
    }
  } else {
    constexpr int step = N / (NS * 2);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int b = t + m * T8;
      const int k = b & (NS - 1);
      if constexpr (NS > 1) {
        bf2(v[m], v[m + 4], twiddle<V, INV>(tw, k * step));
      } else {
        const V a = v[m], c = v[m + 4];
        v[m] = cadd(a, c);
        v[m + 4] = csub(a, c);
      }
      const int base = (b / NS) * NS * 2 + k;
      pos[m] = base;
      pos[m + 4] = base + NS;
    }
  }
}

// barrier over the whole CTA (the default exchange synchronisation of fft_ct)
struct CtaSync {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
// barrier over a group of NG threads (a multiple of 32, whole warps): the warp itself, or a
// named barrier id (1..15) shared by the group's warps only
template <int NG> struct GroupSync {
  int id;
  __device__ __forceinline__ void operator()() const {
    if constexpr (NG == 32) {
      __syncwarp();
    } else {
      asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(NG) : "memory");
    }
  }
};

// whether the stages of a transform run as bf2 levels (stage_bf2) or with the products apart
template <typename V, int N, class Sm> struct UseBf2 {
  static constexpr bool v = sizeof(V) == 16;
};

template <typename V, bool INV, int N, int NF, int NS, class Sm, class Sync = CtaSync>
__device__ __forceinline__ void fft_ct(V (&v)[NF][8], int t, const Sm& sm, const V* __restrict__ tw,
                                       const Sync& sync = Sync()) {
  constexpr int R = StageRadix<N / NS>::v;
  int pos[8];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if constexpr (UseBf2<V, N, Sm>::v) stage_bf2<V, INV, N, R, NS>(v[f], pos, t, tw);
    else stage_prod<V, INV, N, R, NS>(v[f], pos, t, tw);
    if constexpr (NS * R < N) {
#pragma unroll
      for (int m = 0; m < 8; ++m) sm.put(f, pos[m], v[f][m]);
    }
  }
  if constexpr (NS * R < N) {
    sync();
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int m = 0; m < 8; ++m) v[f][m] = sm.get(f, t + m * (N / 8));
    sync();
    fft_ct<V, INV, N, NF, NS * R>(v, t, sm, tw, sync);
  }
}

// ---------------------------------------------------------------------------
// Transforms of four values per thread (surface kernels: more threads with less work each)
// ---------------------------------------------------------------------------
// Stockham stages of radix 4, the first of radix 2 where log2 N is odd; thread t of N / 4 holds the
// values t + m N / 4 before and after.  Exchange layout by the caller (Sm), CTA barriers.
template <int N> struct OddLog2 {
  static constexpr bool v = (N & 0x55555555) == 0;
};
// on: threads without a transform (false) take part in the barriers only.
template <typename V, bool INV, int N, int NS, class Sm>
__device__ __forceinline__ void fft4_on(V (&v)[4], int t, bool on, const Sm& sm, const V* __restrict__ tw) {
  constexpr int T4 = N / 4, R = (NS == 1 && OddLog2<N>::v) ? 2 : 4;
  int pos[4];
  if constexpr (R == 2) {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const V a = v[m], c = v[m + 2];
      v[m] = cadd(a, c);
      v[m + 2] = csub(a, c);
      pos[m] = 2 * (t + m * T4);
      pos[m + 2] = pos[m] + 1;
    }
  } else {
    const int k = t & (NS - 1);
    if constexpr (NS > 1) {
      constexpr int step = N / (NS * 4);
      const V w1 = twiddle<V, INV>(tw, k * step), w2 = twiddle<V, INV>(tw, 2 * k * step);
      if constexpr (sizeof(V) == 16) {
        bf2(v[0], v[2], w2);
        bf2(v[1], v[3], w2);
        bf2(v[0], v[1], w1);
        bf2(v[2], v[3], quarter<V, INV>(w1));
        const V x = v[1];
        v[1] = v[2];
        v[2] = x;
      } else {
        // products apart: a difference as 2 a - t carries the rounding of t, which shows in FP32
        v[1] = cmul(v[1], w1);
        v[2] = cmul(v[2], w2);
        v[3] = cmul(v[3], twiddle<V, INV>(tw, 3 * k * step));
        dft4<V, INV>(v);
      }
    } else {
      dft4<V, INV>(v);
    }
    const int base = (t / NS) * NS * 4 + k;
#pragma unroll
    for (int r = 0; r < 4; ++r) pos[r] = base + r * NS;
  }
  if constexpr (NS * R < N) {
    if (on) {
#pragma unroll
      for (int m = 0; m < 4; ++m) sm.put(pos[m], v[m]);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = sm.get(t + m * T4);
    __syncthreads();
    fft4_on<V, INV, N, NS * R>(v, t, on, sm, tw);
  }
}
template <typename V, bool INV, int N, int NS, class Sm>
__device__ __forceinline__ void fft4_ct(V (&v)[4], int t, const Sm& sm, const V* __restrict__ tw) {
  fft4_on<V, INV, N, NS>(v, t, true, sm, tw);
}
// rows: one pad slot every 8 entries
template <typename V, int N> struct SurfSm {
  static constexpr int LD = N + N / 8;
  V* buf;
  __device__ __forceinline__ void put(int p, V x) const { buf[p + (p >> 3)] = x; }
  __device__ __forceinline__ V get(int p) const { return buf[p + (p >> 3)]; }
};
template <typename V> struct SurfColSm {
  V* buf;
  int kc, f;
  __device__ __forceinline__ void put(int p, V x) const { buf[p * kc + f] = x; }
  __device__ __forceinline__ V get(int p) const { return buf[p * kc + f]; }
};

// CTA of a row pass: about one transform pair per CTA and SM, whole warps.  At most 512 threads, each
// with four values and their padding: 36 KB of dynamic shared memory in FP64, below the 48 KB that need
// a raised limit, also beside the static arrays of the contact kernels.
struct SurfRowCfg {
  int grid, threads;
  size_t smem;
};
template <typename T, int N> inline SurfRowCfg surf_row_cfg(int n2) {
  typedef typename Cx<T>::t V;
  const int pairs = n2 / 2, T4 = N / 4;
  int slots = 1;
  while (slots * 2 * 128 <= pairs && slots * 2 * T4 <= 512) slots *= 2;
  const int threads = slots * T4 > 32 ? slots * T4 : 32;
  slots = threads / T4;
  static_assert((size_t)512 / T4 * SurfSm<V, N>::LD * sizeof(V) <= 36 * 1024, "row CTAs need no shared-memory opt-in");
  return SurfRowCfg{(pairs + slots - 1) / slots, threads, (size_t)slots * SurfSm<V, N>::LD * sizeof(V)};
}

// ---------------------------------------------------------------------------
// FP64 sums over a grid in a fixed order.  An FP64 instruction holds its pipe for 64 cycles per
// warp on this chip, so the chain of additions is what they cost.
// ---------------------------------------------------------------------------
// Sums of up to four values over a warp, reduced together: six additions instead of five per value.
// Lane l ends with the sum of value ((l >> 4) & 1) 2 + ((l >> 3) & 1).
__device__ __forceinline__ double warp_sum4(double v0, double v1, double v2, double v3) {
  const unsigned all = 0xffffffffu;
  const bool h16 = threadIdx.x & 16, h8 = threadIdx.x & 8;
  double a = (h16 ? v2 : v0) + __shfl_xor_sync(all, h16 ? v0 : v2, 16);
  const double b = (h16 ? v3 : v1) + __shfl_xor_sync(all, h16 ? v1 : v3, 16);
  a = (h8 ? b : a) + __shfl_xor_sync(all, h8 ? a : b, 8);
  for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(all, a, o);
  return a;
}
// over the block's whole warps of per-thread values x of kind j = threadIdx.x & 3 that are already
// summed over the lanes of equal j: lanes 0..3 of warp 0 end with the sums
__device__ __forceinline__ double block_sum_kind(double x, double* sh) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (nw == 1) return x;
  if (l < 4) sh[w * 4 + l] = x;
  __syncthreads();
  if (w > 0) return 0;
  x = 0;
  for (int k = l >> 2; k < nw; k += 8) x += sh[k * 4 + (l & 3)];
  for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// sums of v over the grid: true in thread 0 of the last block to arrive, which then holds them
__device__ __forceinline__ bool grid_sum(double (&v)[4], double* part, unsigned* cnt) {
  __shared__ double sh[32 * 4];
  __shared__ bool last;
  const int l = threadIdx.x & 31;
  double x = warp_sum4(v[0], v[1], v[2], v[3]);
  // value j from the lane group that holds it
  x = __shfl_sync(0xffffffffu, x, ((l & 3) >> 1) * 16 + (l & 1) * 8);
  x = block_sum_kind(x, sh);
  if (threadIdx.x < 4) {
    part[blockIdx.x * 4 + threadIdx.x] = x;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  x = 0;
  for (int b = threadIdx.x >> 2; b < (int)gridDim.x; b += blockDim.x >> 2) x += __ldcg(part + b * 4 + (threadIdx.x & 3));
  for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  x = block_sum_kind(x, sh);
  if (threadIdx.x >= 32) return false;
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = __shfl_sync(0xffffffffu, x, j);
  if (threadIdx.x == 0) *cnt = 0u;
  return threadIdx.x == 0;
}

__device__ __forceinline__ float two_sum_err(float a, float b, float s) {  // a + b - s
  const float bb = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// Running sum of FP32 values in three words: the rounding of each word goes to the next, only the
// last word's is lost (below 2^-70 of the sum; an FP64 sum loses 2^-53 at every addition).
struct Sum3 {
  float a, b, c;
};
__device__ __forceinline__ void sum3_add(Sum3& s, float x) {
  const float a = __fadd_rn(s.a, x), e = two_sum_err(s.a, x, a);
  const float b = __fadd_rn(s.b, e);
  s.c = __fadd_rn(s.c, two_sum_err(s.b, e, b));
  s.a = a;
  s.b = b;
}
// Three such sums in FP64, by a whole warp.  The third words, zero up to two values per sum, are added
// only where a lane has one, and by a call: FP64 instructions under a predicate hold the pipe all the same.
static __device__ __noinline__ double sum3_third(double v, float c) { return v + (double)c; }
__device__ __forceinline__ void sum3_values(const Sum3& x, const Sum3& y, const Sum3& z, double& vx, double& vy, double& vz) {
  vx = (double)x.b;
  vy = (double)y.b;
  vz = (double)z.b;
  if (__any_sync(0xffffffffu, x.c != 0.f || y.c != 0.f || z.c != 0.f)) {
    vx = sum3_third(vx, x.c);
    vy = sum3_third(vy, y.c);
    vz = sum3_third(vz, z.c);
  }
  vx += (double)x.a;
  vy += (double)y.a;
  vz += (double)z.a;
}

// ---------------------------------------------------------------------------
// asynchronous global -> shared copies (cp.async), all in flight before one wait
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_async_8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
template <typename V> __device__ __forceinline__ void cp_async_cx(V* smem, const V* gmem) {
  if (sizeof(V) == 16) cp_async_16(smem, gmem);
  else cp_async_8(smem, gmem);
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's committed copy groups are still in flight
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Raises a kernel's dynamic shared-memory cap to the device's opt-in maximum.  The value is
// the same on every call: contexts used from several host threads launch one kernel with
// different sizes, and a cap set to the exact size of one launch could be lowered under
// another thread's launch of the same kernel.
inline int smem_optin_max() {
  static const int v = [] {
    int dev = 0, m = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return m > 0 ? m : 48 * 1024;
  }();
  return v;
}
// multiprocessors of the current device
inline int sm_count() {
  static const int v = [] {
    int dev = 0, m = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev);
    return m > 0 ? m : 1;
  }();
  return v;
}
// Launches of at most 48 KB need no cap (a runtime call less on the host path of small grids).
template <typename K> inline void smem_cap(K kern, size_t smem) {
  if (smem <= 48 * 1024) return;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin_max());
}

// ---------------------------------------------------------------------------
// context
// ---------------------------------------------------------------------------
#define FVIM_NSOLVER_BUFS 26

// fixed parts of the solver workspace, bytes
constexpr int kDfsBlocks = 4096;  // blocks of the DF-SANE residual pass (at least one per plane, 3072 planes)
constexpr size_t kPartBytes = (size_t)kDfsBlocks * 4 * sizeof(double);  // block partials, up to four values each
constexpr size_t kScalarBlock = 256;  // scalars of the solver loops (V_PKS)
constexpr size_t kDfsBytes = 1024;    // device DF-SANE state (V_DFS)
constexpr size_t kPkfBytes = 512;     // fused contact iteration (V_PKF): PkState, arrival counter at byte 256

struct fvim_ctx {
  int no_pdl;  // launches without the programmatic-serialisation attribute (solver graph capture)
  // h1: row stride of the half spectrum (complex); power-of-two grids: N1/2 columns (the
  // k1 = N1/2 coefficient kept apart in nq); gen: floor(N1/2) + 1 columns rounded up to 16
  int n1, n2, nz, h1;
  int gen;  // a side is not a power of two: direct DFTs (dft.cu), every coefficient in spec
  int hs;   // stored k1 columns (k1 < hs); == h1 for power-of-two grids
  int prec;  // FVIM_FP32 / FVIM_FP64
  double L1, L2;
  double E, nu, sigma_y, E_h, lam, mu;
  cudaStream_t stream;
  int device;
  int uniform;   // depth nodes equally spaced
  double hz;     // spacing when uniform
  double* z_host;
  void* z_dev;   // T[nz]
  void* tw1;     // complex T[n1]
  void* tw2;     // complex T[n2]
  void* spec;    // complex T[nz][6][n2][h1]
  void* nq;      // T[nz][6][n2] row-Nyquist coefficients
  void* surf;    // complex T[n2][h1]
  void* surf_nq; // T[n2]
  void* st_eps_p; // T[nz][6][n2][n1]
  void* st_ep;    // T[nz][n2][n1]
  void* st_sig;   // T[nz][6][n2][n1]
  void* st_T;     // T[n2][n1] contact pressure of the last converged increment
  int last_kernels;
  void* prof;  // ProfState* (capi.cu) or NULL
  // solver workspace (solvers.cu), allocated on first use
  void* sv[FVIM_NSOLVER_BUFS];
  double* h_part;  // host copy of reduction partials
  long n_applies;  // Mindlin applies issued by the solvers
  int fft2_cl;     // whole-plane cluster FFTs usable: -1 not yet known, 0 no, 1 yes
  void* srt;       // solver runtime (solvers.cu): own stream, events, captured CUDA graphs
  int depth_chunk; // depth nodes per chunk thread of the depth kernel; 0: depth_chunk_default
  int plan_tuned;  // depth_chunk came from a timing run (fvim_autotune) in this process
  int depth_ctas;  // CTAs per SM of the FP32 register depth kernel: 0 or 2 (128 registers), 3 (80)
  float depth_cut; // chunk-scan cutoff eps_co of the FP32 register depth kernel (0: exact scan)
  void* tmap;      // CUtensorMap (host, 64-byte aligned) over the spectrum for the depth tile, or NULL
  int tma_rows;    // rows (z, component) per tensor-copy box of the depth tile; 0: no tensor copies
  int* dev_status; // device status word: bit 0 set by a bounded device wait that expired
  int tma_test_extra;  // bytes added to the depth tile's expected copy count (tests of the
                       // expired-wait path only; FVIM_TEST_TMA_EXTRA at creation, else 0)
  int fft2_fused;  // one-pass 2-D FFTs through L2: -1 not yet known, 0 not used, 1 used
  int fft_path;    // in-plane FFT path chosen by the tuner or fvim_set_plan (FVIM_FFT_*), -1: none
                   // (the row / column kernels unless an environment variable selects another)
};

// ---------------------------------------------------------------------------
// Chained launches.  The kernels of an apply depend on one another in stream order, and from one
// stream launch to the next a dependent kernel starts about 4.5 us later, which is all the time there
// is on small grids.  They are launched with programmatic stream serialisation: a kernel may be
// placed on the device when the CTAs of the one before have left it, and chain_begin() - the first
// statement of every such kernel, before any global access and any return - waits until that one is
// complete and its writes are visible (so completion of a kernel implies completion of everything
// before it).  There is no earlier trigger: placed from the start of the kernel before, the next
// kernel's CTAs crowd the SMs that drain first (81 x 81 x 32 73 us against 53, a captured 64 x 64 x 8
// apply 15.1 us against 11.1).  Applies, us, plain launches -> chained: 64 x 64 x 8 22.5 -> 13.6,
// 128 x 128 x 32 with u3 48.1 -> 33.2, 81 x 81 x 32 64 -> 53, 256 x 128 x 57 94 -> 80, 512 x 512 x 64
// 672 -> 661, grouped 823 -> 805.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline void launch_chain_on(cudaStream_t stream, bool chained, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                            A&&... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at;
  memset(&at, 0, sizeof(at));
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline void launch_chain(const fvim_ctx* c, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, A&&... args) {
  launch_chain_on(c->stream, !c->no_pdl, kern, grid, block, smem, std::forward<A>(args)...);
}

// tile plan of the depth kernel (depth.cu): default chunk length, and whether a chunk length
// gives a launchable configuration on this context's grid and precision
int depth_chunk_default(int nz);
// ctas: CTAs per SM the FP32 register variant is compiled for (2 default, 3 with 80 registers)
bool depth_chunk_ok(const fvim_ctx* c, int chunk, int ctas = 2);
// CTAs per SM the depth kernel is launched for with a chunk length and register budget, and under the
// context's plan (0: shared-memory variant; a budget of 3 whose tile does not fit three times gives 2)
int depth_shape_ctas(const fvim_ctx* c, int chunk, int ctas);
int depth_launch_ctas(const fvim_ctx* c);
// process-wide plan table (tune.cu): the tuned chunk length of a grid, or 0; its tuned FFT
// path, or -1
int plan_lookup(const fvim_ctx* c);
int plan_lookup_fft(const fvim_ctx* c);
int plan_lookup_ctas(const fvim_ctx* c);
// whether an in-plane FFT path is built for the context's grid and precision (capi.cu)
bool fft_path_available(const fvim_ctx* c, int path);

// material constants of the depth operator for one kind of output, evaluated on the host in FP64
template <typename T> struct DepthMat {
  T lam, mu, iu;      // iu = 1 / (2 mu)
  T ms, la;           // 2 nu - 1; factor of w_33 in the local terms
  T kap, hq, p, w, t; // factors of the moments in the output (depth.cu, node_out)
  int stress;
};
template <typename T> inline DepthMat<T> depth_mat(double lam, double mu, double nu, int out_kind) {
  const bool st = out_kind == FVIM_STRESS;
  const double sc = st ? 1.0 : 1.0 / (2.0 * mu);
  DepthMat<T> m;
  m.lam = (T)lam;
  m.mu = (T)mu;
  m.iu = (T)(1.0 / (2.0 * mu));
  m.ms = (T)(2.0 * nu - 1.0);
  m.la = (T)(st ? nu / (1.0 - nu) : 1.0 / (lam + 2.0 * mu));
  m.kap = (T)(sc / (4.0 * (1.0 - nu)));
  m.hq = (T)(0.5 * sc);
  m.p = (T)(st ? -2.0 * nu : 0.0);
  m.w = (T)(st ? 2.0 : 2.0 - 2.0 * nu);
  m.t = (T)(st ? 0.0 : 2.0 * nu);
  m.stress = st ? 1 : 0;
  return m;
}

// kernel kinds for fvim_profile_read
enum ProfSlot {
  PROF_ROWS_FWD6 = 0, PROF_COLS_FWD, PROF_MINDLIN_DEPTH, PROF_COLS_INV, PROF_ROWS_INV6,
  PROF_ROWS_FWD1, PROF_ROWS_INV1, PROF_BOUSSINESQ, PROF_RETURN_MAP, PROF_COMMIT, PROF_FFT2_FWD,
  PROF_FFT2_INV, PROF_NSLOTS
};

// material constants handed to kernels
template <typename T> struct Mat {
  T lam, mu, nu, sigma_y, E_h;
};

// launchers (defined in the .cu files, instantiated for float and double)
// zr (device, two ints) or NULL: only layers zr[0] <= z < zr[1] hold non-zero input; the forward
// passes skip the others and the depth kernel reads them as zero
template <typename T> int launch_rows_fwd6(const fvim_ctx* c, const T* eps_p, int z0, int nzs, const int* zr = nullptr);
template <typename T> int launch_rows_fwd1(const fvim_ctx* c, const T* f);
template <typename T> int launch_cols(const fvim_ctx* c, bool inverse, void* planes, int nplanes, const int* zr = nullptr);
template <typename T> int launch_rows_inv6(const fvim_ctx* c, T* out, T nq_scale, int z0, int nzs);
template <typename T> int launch_rows_inv1(const fvim_ctx* c, T* f);
// eps_in: the spectrum holds eps_p (Hooke's law applied per mode) instead of w = C:eps_p
template <typename T>
int launch_mindlin_depth(const fvim_ctx* c, int out_kind, bool want_u3, bool eps_in = false, const int* zr = nullptr);
template <typename T> int launch_boussinesq(const fvim_ctx* c, int out_kind, bool want_vol, bool want_u3);
template <typename T> int launch_return_map(const fvim_ctx* c, const T* d_eps, T* d_eps_p, T* d_ep);
template <typename T> int launch_commit(const fvim_ctx* c, const T* d_eps, const T* d_eps_p, const T* d_ep);
// surface transforms with compile-time sides of 16 to 1024 (surface.cu); false when a side has no
// variant: rows of a real field to and from c->surf, columns of c->surf in place
template <typename T> bool launch_surf_rows_fwd(const fvim_ctx* c, const T* f);
template <typename T> bool launch_surf_rows_inv(const fvim_ctx* c, T* f, T scale);
template <typename T> bool launch_surf_cols(const fvim_ctx* c, bool inverse);
// strain or stress of the Boussinesq field evaluated in the inverse column pass (FP32): c->surf
// (p_hat) to the half row spectra in c->spec; false when the grid has no variant
bool launch_bous_cols(const fvim_ctx* c, int out_kind);

// solver runtime (solvers.cu): release, and drop captured graphs after a material change
void solver_release(fvim_ctx* c);
void solver_drop_graphs(fvim_ctx* c);

// whole-plane cluster FFTs (fft2d_cluster.cu), FP32 and a few plane sizes only
bool fft2_cluster_available(const fvim_ctx* c);
int launch_fft2_fwd_cluster(const fvim_ctx* c, const float* src);
int launch_fft2_inv_cluster(const fvim_ctx* c, float* out, int nq_mode, float nq_scale);

// one-pass 2-D FFTs with the row spectra exchanged through L2 (fft2d_l2.cu), FP32; zr as for
// launch_rows_fwd6 (planes of layers outside the range are skipped)
bool fft2_fused_available(const fvim_ctx* c);
int launch_fft2_fwd_fused(const fvim_ctx* c, const float* src, const int* zr = nullptr);
int launch_fft2_inv_fused(const fvim_ctx* c, float* out, int nq_mode, float nq_scale);

// direct DFTs of grids with a side that is not a power of two (dft.cu, fvim_ctx::gen):
// rows real -> half spectrum [rows][h1], columns in place, half spectrum -> real rows x scale
template <typename T> int launch_dft_rows_fwd(const fvim_ctx* c, const T* src, void* dst, size_t rows);
template <typename T> int launch_dft_cols(const fvim_ctx* c, bool inverse, void* planes, int nplanes);
template <typename T> int launch_dft_rows_inv(const fvim_ctx* c, const void* src, T* dst, size_t rows, T scale);
// grid sides the library takes: a power of two (4..1024 for N1, 2..1024 for N2, the FFT path)
// or an odd number 3..255 (with the other side odd or a power of two up to 256: direct DFTs)
bool grid_ok(int n1, int n2);
bool grid_gen(int n1, int n2);
int spec_stride(int n1, int n2);

// compile-time-length FFT kernels (fft_ct.cu); false when the length has no variant
template <typename T> bool launch_cols_ct(const fvim_ctx* c, bool inverse, void* planes, int nplanes, const int* zr = nullptr);
// surface compliance applied in the column pass (fft_ct.cu); false when N2 has no variant
template <typename T> bool launch_cols_conv_ct(const fvim_ctx* c);
template <typename T> bool launch_rows_fwd6_ct(const fvim_ctx* c, const T* eps_p, int z0, int nzs, const int* zr = nullptr);
template <typename T> bool launch_rows_inv6_ct(const fvim_ctx* c, T* out, T nq_scale, int z0, int nzs);

// ---- fused Polonsky-Keer iteration (contact_cg.cu) ---------------------------------------
// device state of one contact solve
struct PkState {
  double nIc, gbar, G_old, beta, delta, tau, s, err;  // scalars of the iteration
  double start, unif;                                  // scale of the initial pressure (negative: uniform), uniform pressure
  double W, dA, dA_W, tol;                             // dA_W = dA / W
  float4 gbarw, betaw, tauw, sw;                       // the scalars of the elementwise steps in words of FP32
  const void* h;
  void* p;
  int done, it, bad, max_it;
  int passes;  // iterations begun, counted apart from the sums: the loop ends at max_it whatever they do
};
static_assert(sizeof(PkState) <= 256, "pinned copy of the contact state");
struct PkfArgs {
  int n1, n2, h1;
  double L1, L2, nu, mu;
  cudaStream_t stream;
  PkState* S;
  void *u, *g, *t, *pold;  // surface work arrays [n2][n1]
  void* green;             // surface compliance [n2][h1]
  void* surf;              // half spectrum [n2][h1]
  const void *tw1, *tw2;
  double* part;            // block partials of the sums
  unsigned* cnt;           // arrival counter, zero between kernels
  cudaGraphConditionalHandle cond;
  int use_cond;            // the last kernel of an iteration sets the loop condition
};
bool pkf_available(const fvim_ctx* c);
// whole solve in one kernel (small square surfaces)
bool pkf_small(const fvim_ctx* c);
template <typename T> int pkf_solve_small(const PkfArgs& a, const PkState& init);
// state, initial pressure scaled to the load, its displacement and mean gap
template <typename T> int pkf_begin(const PkfArgs& a, const PkState& init);
// one iteration; does nothing once the state's done flag is set
template <typename T> int pkf_iteration(const PkfArgs& a);

// ---- J2 radial return with linear isotropic hardening (Sec. 4.1) at one voxel -----------
// de: strain increment, sig: stress of the last converged increment, ep: cumulated plastic
// strain there.  Returns the increment of cumulated plastic strain and writes the plastic
// strain increment (Voigt order 11, 22, 33, 23, 13, 12; shear entries are tensor components).
// Shared by the return-map kernel and the fused DF-SANE trial kernel (the same arithmetic).
template <typename T>
__device__ __forceinline__ T rmap_voxel(const T (&de)[6], const T (&sig)[6], T ep, T lam, T mu, T sy, T Eh,
                                        T (&dp)[6]) {
  T st[6];
  const T tr = de[0] + de[1] + de[2];
#pragma unroll
  for (int c = 0; c < 6; ++c) st[c] = sig[c] + 2 * mu * de[c];
  st[0] += lam * tr;
  st[1] += lam * tr;
  st[2] += lam * tr;
  const T m = (st[0] + st[1] + st[2]) / (T)3;
  const T s[6] = {st[0] - m, st[1] - m, st[2] - m, st[3], st[4], st[5]};
  const T nrm2 = s[0] * s[0] + s[1] * s[1] + s[2] * s[2] + 2 * (s[3] * s[3] + s[4] * s[4] + s[5] * s[5]);
  const T fy = sqrt((T)1.5 * nrm2);
  const T f = fy - (sy + Eh * ep);
  T dEp = 0, k = 0;
  if (f > 0) {
    dEp = f / ((T)3 * mu + Eh);
    k = (T)1.5 * dEp / fy;
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) dp[c] = k * s[c];
  return dEp;
}

// layer range of the flowing voxels (elsewhere the plastic increment is exactly zero): one
// pair of atomics per warp, over the lanes that flow
__device__ __forceinline__ void flow_range_note(int* zr, int z) {
  const unsigned am = __activemask();
  const int lo = __reduce_min_sync(am, z), hi = __reduce_max_sync(am, z);
  if ((int)(threadIdx.x & 31) == __ffs(am) - 1) {
    atomicMin(zr, lo);
    atomicMax(zr + 1, hi + 1);
  }
}

// ---- grouped Mindlin apply: FP32 problems of uneven size, one launch per phase ----------
// One problem of a group: its context's buffers and the constants its kernels need.
constexpr int kGrpMax = 64;  // problems per group (the table travels as a kernel parameter)
struct GrpProb {
  const float* eps;      // eps_p [nz][6][n2][n1]
  float* out;            // stress or strain [nz][6][n2][n1]
  float2* spec;          // half spectrum [nz][6][n2][h1]
  float* nq;             // k1 = N1/2 coefficients [nz][6][n2]
  const float2* tw1;     // twiddles of N1
  const float2* tw2;     // twiddles of N2
  const float* zn;       // depth nodes [nz]
  int n1, n2, nz, h1, hs;
  int nch, nchp;         // depth chunks of 4 nodes, and that count rounded up to a power of two
  int uniform;
  float w1, w2, lam, mu, hz, cut;
  DepthMat<float> dm;
  float nq_scale, scale; // inverse rows: Nyquist factor and 1 / (N1 N2)
};
struct GrpTable {
  int n;                     // problems
  int start[kGrpMax + 1];    // first CTA of each problem in the launch; start[n] = CTAs
  GrpProb p[kGrpMax];
};
static_assert(sizeof(GrpTable) < 16 * 1024, "the group table is a kernel parameter");
// the problem of CTA b: the last i with start[i] <= b
__device__ __forceinline__ int grp_find(const GrpTable& t, int b) {
  int lo = 0, hi = t.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (t.start[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
// the four kinds of grouped launch (fft_ct.cu, depth.cu); each fills t.start for its own CTA
// counts.  Problems: FP32, 64 <= N1, N2 <= 512 powers of two, Nz <= 64.
int launch_grp_rows_fwd(GrpTable& t, cudaStream_t s);
int launch_grp_cols(GrpTable& t, bool inverse, cudaStream_t s);
int launch_grp_depth(GrpTable& t, cudaStream_t s);
int launch_grp_rows_inv(GrpTable& t, cudaStream_t s);

// launch sequences of the entry points (capi.cu), used by the solvers
// zr: see launch_rows_fwd6; honoured for FVIM_STRAIN output only
template <typename T> int apply_mindlin_t(fvim_ctx* c, const T* eps_p, T* out, int kind, T* u3, const int* zr = nullptr);
template <typename T> int apply_boussinesq_t(fvim_ctx* c, const T* p, T* u3, T* vol, int kind);
// zr (device, two ints) or NULL: receives the layer range [zr[0], zr[1]) of the voxels that
// flow (reset by the caller to {INT_MAX-ish, 0} first).
template <typename T> int return_map_t(fvim_ctx* c, const T* d_eps, T* d_eps_p, T* d_ep, int* zr = nullptr);
template <typename T> int commit_t(fvim_ctx* c, const T* d_eps, const T* d_eps_p, const T* d_ep);

// true when e is an error; the error and the source line that saw it are kept as this host
// thread's last CUDA error (fvim_last_cuda_error)
bool fvim_cuda_failed(cudaError_t e, const char* file = nullptr, int line = 0);
#define FVIM_CU(call) fvim_cuda_failed((call), __FILE__, __LINE__)
#define FVIM_CUDA_CHECK_LAUNCH()                                                        \
  do {                                                                                  \
    if (fvim_cuda_failed(cudaGetLastError(), __FILE__, __LINE__)) return FVIM_ERR_CUDA; \
  } while (0)
