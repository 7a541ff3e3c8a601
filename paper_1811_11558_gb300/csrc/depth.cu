// Per-wavevector depth operators of the discretised Mindlin and Boussinesq operators.
//
// For one in-plane mode q = 2 pi (k1/L1, k2/L2) the Mindlin displacement gradient at the
// depth node x3^i is (Eq. 2gradient, Eq. jump, Eq. mindlin_B_U, Thm 1)
//   grad N[w](q, x3^i) = - int grad^2 U_inf(-q, y3 - x3^i) : w_h(q, y3) dy3
//                        - ([[grad U_inf]] : w(q, x3^i)) x e3  +  image term,
// with w_h the piecewise-linear interpolant of the nodal coefficients (Sec. 3.2).
//
// GB300 formulation (the paper's element integrals, evaluated exactly, reorganised):
// * Frame: the tensors are rotated so that q lies along x1; with Delta(-q) = (-i, 0, 0) every
//   kernel coefficient of Table 1 becomes a constant.  In that frame the contraction of the
//   kernels with w has rank three per branch: with the nodal sources
//     n = w_33 - w_qq -+ 2i w_q3,   m = (2 nu - 1)(w_qq + w_33),   a = w_qp +- i w_p3
//   (upper sign: the branch A of the elements above the node, lower: P, below), every strain
//   and stress component is a fixed combination of three moments per branch,
//     n = int g0 n,   a = int g0 a,   v = int g0 m -+ int g1 n.
//   (The generic form carries five rotated components and one contraction per branch, and
//   evaluates the image field per node: 457 warp instructions per warp of nodes, measured on
//   512 x 512 x 64 FP32, against 236 here.  Depth kernel, ms, generic form -> this one: 512 x
//   512 x 64 FP32 0.204 -> 0.146, 1024 x 1024 x 32 (C = 2) 0.642 -> 0.336, 256 x 128 x 57
//   refined 0.043 -> 0.028, 128 x 128 x 126 FP64 1.163 -> 0.355.)
// * Depth integral: the g0/g1 kernels are exponentials exp(-q|y3 - x3|) times polynomials, so
//   the moments follow from those of the neighbouring node by exact one-element steps,
//     v <- e^{-qh}(v - qh n) + ...,  n <- e^{-qh} n + ...,  a <- e^{-qh} a + ...,
//   with the linear-element integrals of Eq. (int_g0)/(int_g1) in closed form.  This replaces
//   the cutoff of Sec. 3.2 (no approximation) and costs O(Nz) per mode.
// * Image term: the Boussinesq field that cancels the surface traction of the full-space field
//   has the form of the A branch of a source at the surface, so it is the starting value of
//   the A recursion there: A(0) = (n_P + 2 v_P, -v_P, a_P) with P = P(0) the complete moments
//   of the branch below.  The surface displacement is u3(0) = v_P / (2 mu).
// * In the stress the local terms of the 33, 23 and 13 components cancel exactly (the
//   traction is continuous across the layer), and those of the others are w_33 nu / (1 - nu) - w.
// * Parallelism: a CTA holds KT consecutive k1 columns (one k2) for all depth nodes; the depth
//   range is cut into chunks of C nodes, one thread per (chunk, k1).  Each chunk computes its
//   own moments at every node and the carry it hands to its neighbours (both recursions from
//   zero); 4 KT threads then run the chunk recurrences of the carries (two branches, the
//   coupled pair (n, v) and a apart), in chunk order: a log-depth scan by all threads cost more
//   instructions than everything else at C = 2; then every thread adds the propagated carries.
// * q = 0 (mode k = 0): laminate solution (sigma_i3 = 0, eps_ab = 0).  k2 = N2/2
//   (not in Z^2_N): no operator term, so sigma_hat = -w_hat (stress) or 0 (strain).
#include <string.h>

#include <algorithm>

#include "fvim_internal.cuh"

namespace {

constexpr int KT_MAX = 16;  // k1 columns per CTA (128-byte rows in FP32)
constexpr double kTwoPi = 6.283185307179586476925;

template <typename T> __device__ __forceinline__ T dexp(T x);
template <> __device__ __forceinline__ float dexp<float>(float x) { return expf(x); }
template <> __device__ __forceinline__ double dexp<double>(double x) { return exp(x); }

// wait for phase 0 of the mbarrier at shared address bar, at most limit_ns nanoseconds of the
// global timer and at most 2^24 polls (should the timer not advance); true when the phase
// completed
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned long long limit_ns) {
  unsigned long long t0 = 0;
  for (int it = 0; it < (1 << 24); ++it) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(bar)
                 : "memory");
    if (ok) return true;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (it == 0) t0 = t;
    if (t - t0 > limit_ns) return false;
  }
  return false;
}


// ---- moments and element coefficients ------------------------------------------------
// One branch of the depth integral at a node (rank-three form, see the head of the file).
template <typename V> struct Br {
  V n, v, a;
};
template <typename V> __device__ __forceinline__ Br<V> br_zero() {
  Br<V> s;
  s.n = s.v = s.a = mk<V>(0, 0);
  return s;
}

// One element: with a = q h and I_n(a) = int_0^1 s^n exp(-a s) ds (Eq. (int_g0)/(int_g1)),
// E = e^{-a}; b0, d0 weight the source of the node the step arrives at (h (I0 - I1), a h (I1 - I2)),
// b1, d1 that of the node it leaves (h I1, a h I2).
template <typename T> struct El {
  T E, a, b0, b1, d0, d1;
};
constexpr int EL_N = 6;

// closed form for a above a threshold, Taylor series below it (no cancellation)
template <typename T> __device__ __forceinline__ El<T> elem_coef(T q, T h) {
  El<T> c;
  const T a = q * h;
  const T E = dexp<T>(-a);
  T I0, I1, I2;
  const T thr = sizeof(T) == 4 ? (T)1.0 : (T)0.5;
  if (a < thr) {
    // I_2(a) = sum_m (-a)^m / (m! (m + 3)) by Horner's rule (constant coefficients), then upwards by
    // parts, I_{n-1} = (a I_n + E) / n, which loses nothing
    constexpr int M = sizeof(T) == 4 ? 12 : 18;
    double f = 1;  // 1 / m!, folded at compile time
    T cm[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
      cm[m] = (T)(f / (m + 3));
      f /= m + 1;
    }
    I2 = cm[M - 1];
#pragma unroll
    for (int m = M - 2; m >= 0; --m) I2 = fma(-a, I2, cm[m]);
    I1 = (T)0.5 * fma(a, I2, E);
    I0 = fma(a, I1, E);
  } else {
    const T ia = (T)1 / a;
    I0 = ((T)1 - E) * ia;
    I1 = ((T)1 - E * ((T)1 + a)) * ia * ia;
    I2 = ((T)2 - E * (a * a + (T)2 * a + (T)2)) * ia * ia * ia;
  }
  c.E = E;
  c.a = a;
  c.b0 = h * (I0 - I1);
  c.b1 = h * I1;
  c.d0 = a * h * (I1 - I2);
  c.d1 = a * h * I2;
  return c;
}
// the coefficients of one element and column in shared memory: p[j * KT], j < EL_N
template <typename T, int KT> __device__ __forceinline__ void el_put(T* p, const El<T>& c) {
  p[0] = c.E; p[KT] = c.a; p[2 * KT] = c.b0; p[3 * KT] = c.b1; p[4 * KT] = c.d0; p[5 * KT] = c.d1;
}
template <typename T, int KT> __device__ __forceinline__ El<T> el_get(const T* p) {
  El<T> c;
  c.E = p[0]; c.a = p[KT]; c.b0 = p[2 * KT]; c.b1 = p[3 * KT]; c.d0 = p[4 * KT]; c.d1 = p[5 * KT];
  return c;
}

// one step of a branch: arriving at a node (its source weighted b0, d0), and leaving it across
// the next element (propagation, its source weighted b1, d1)
template <typename T, typename V>
__device__ __forceinline__ void br_arrive(Br<V>& s, const El<T>& c, V n, V m, V a) {
  s.n = caxpy(s.n, c.b0, n);
  s.v = caxpy(caxpy(s.v, c.b0, m), -c.d0, n);
  s.a = caxpy(s.a, c.b0, a);
}
template <typename T, typename V>
__device__ __forceinline__ void br_leave(Br<V>& s, const El<T>& c, V n, V m, V a) {
  V v = cscale(caxpy(s.v, -c.a, s.n), c.E);
  s.v = caxpy(caxpy(v, c.b1, m), -c.d1, n);
  s.n = caxpy(cscale(s.n, c.E), c.b1, n);
  s.a = caxpy(cscale(s.a, c.E), c.b1, a);
}
// d += c propagated over a distance with E = e^{-x}, xE = x e^{-x}, x = q times the distance
template <typename T, typename V>
__device__ __forceinline__ void br_add_prop(Br<V>& d, const Br<V>& c, T E, T xE) {
  d.n = caxpy(d.n, E, c.n);
  d.v = caxpy(caxpy(d.v, E, c.v), -xE, c.n);
  d.a = caxpy(d.a, E, c.a);
}

template <typename T> struct ModeGeom {
  T q, c, s;
  bool zero, nyq;
};

// wavevector of the mode (k1, k2) in the arithmetic of the path: w1 = 2 pi / L1, w2 = 2 pi / L2.
// k2 is signed (k2 - N2 above N2/2); modes outside Z^2_N (k1 = N1/2 or k2 = N2/2 on even
// sides) and the padding columns k1 >= hs carry no operator term (flag nyq).
template <typename T>
__device__ __forceinline__ ModeGeom<T> mode_geom(int k1, int k2, int n1, int n2, int hs, T w1, T w2) {
  ModeGeom<T> g;
  const int k2s = 2 * k2 < n2 ? k2 : k2 - n2;
  g.nyq = (2 * k2 == n2) || (2 * k1 == n1) || k1 >= hs;
  g.zero = (k1 == 0 && k2 == 0);
  const T q1 = w1 * (T)k1;
  const T q2 = w2 * (T)k2s;
  const T q = sqrt(q1 * q1 + q2 * q2);
  const T iq = q > (T)0 ? (T)1 / q : (T)0;
  g.q = q;
  g.c = q > (T)0 ? q1 * iq : (T)1;
  g.s = q2 * iq;
  return g;
}

// Constants of a column (one mode), evaluated once per column while the tile is in flight and read
// from shared memory by the column's chunk threads: evaluated by every thread they were half of
// the instructions at two nodes per thread.  The trailing pad spreads the columns' 16-byte reads
// over the banks.  (With this and the four-chunk read-ahead of the carries: C = 2 at 1024 x 1024 x
// 32 0.465 -> 0.339 ms, FP64 128 x 128 x 126 0.385 -> 0.355; the exponentials of the carries among
// them too: 0.341 -> 0.336.)
template <typename T> struct __align__(16) ColIn {
  T E, a, b0, b1, d0, d1;        // element coefficients of a uniform grid
  T c, s, cc, ss, cs2, cs, c2;   // rotation: cos, sin, cos^2, sin^2, 2 cos sin, cos sin, cos^2 - sin^2
  T q, kind, EC;                 // wavenumber; 0 recursion, 1 laminate (k = 0), 2 outside Z^2_N; uniform: e^{-q C h}
  __device__ __forceinline__ El<T> el() const {
    El<T> e;
    e.E = E; e.a = a; e.b0 = b0; e.b1 = b1; e.d0 = d0; e.d1 = d1;
    return e;
  }
};
// Output of a node from the complete moments of both branches: with kappa = q / (4 (1 - nu)),
//   sigma_33 = kappa (v_A + v_P),             sigma_q3 = -i kappa (v_A - v_P + n_A - n_P),
//   sigma_qq = -kappa (v_A + v_P + 2 (n_A + n_P)),   sigma_pp = -2 nu kappa (n_A + n_P),
//   sigma_p3 = i q/2 (a_A - a_P),             sigma_qp = q/2 (a_A + a_P)
// plus the local terms; the strain is the same with 2 - 2 nu for the factor 2 of qq, 2 nu (n_A
// + n_P) added to 33, no pp component, all over 2 mu.  The constants of the rotation back are
// folded into the combinations.
template <typename T> struct __align__(16) ColOut {
  T k11w, k22w, k12w, k11n, k22n, k12n, k11a, k12a, k33, cy, sy, cz, sz, EC1, pad[2];
};
template <typename T> struct __align__(16) Col {
  ColIn<T> in;
  ColOut<T> out;
  T pad[4];
};

// constants of column k1 of row k2 (uniform: with the element coefficients of spacing hz)
template <typename T>
__device__ __forceinline__ void col_put(Col<T>* p, int k1, int k2, int n1, int n2, int hs, T w1, T w2, const DepthMat<T>& m,
                                        bool uniform, T hz, int C, T d1) {
  const ModeGeom<T> g = mode_geom<T>(k1, k2, n1, n2, hs, w1, w2);
  ColIn<T> i;
  El<T> e = {0, 0, 0, 0, 0, 0};
  if (uniform) e = elem_coef<T>(g.q, hz);
  i.E = e.E; i.a = e.a; i.b0 = e.b0; i.b1 = e.b1; i.d0 = e.d0; i.d1 = e.d1;
  i.c = g.c; i.s = g.s; i.cc = g.c * g.c; i.ss = g.s * g.s; i.cs = g.c * g.s; i.cs2 = (T)2 * i.cs; i.c2 = i.cc - i.ss;
  i.q = g.q;
  i.kind = g.nyq ? (T)2 : (g.zero ? (T)1 : (T)0);
  i.EC = uniform ? dexp<T>(-g.q * hz * (T)C) : (T)0;
  p->in = i;
  const T kap = m.kap * g.q, q2 = m.hq * g.q, pp = m.p * kap;
  ColOut<T> o;
  o.k11w = -kap * i.cc; o.k22w = -kap * i.ss; o.k12w = -kap * i.cs;
  o.k11n = pp * i.ss; o.k22n = pp * i.cc; o.k12n = -pp * i.cs;
  o.k11a = -q2 * i.cs2; o.k12a = q2 * i.c2;
  o.k33 = kap;
  o.cy = kap * g.c; o.sy = kap * g.s; o.cz = q2 * g.c; o.sz = q2 * g.s;
  o.EC1 = uniform ? dexp<T>(-g.q * d1) : (T)0;  // propagator over the first chunk's nodes
  o.pad[0] = o.pad[1] = 0;
  p->out = o;
}

// nodal sources of both branches from w (11, 22, 33, 23, 13, 12)
template <typename V> struct Src {
  V nA, nP, m, aA, aP;
};
template <typename T, typename V>
__device__ __forceinline__ Src<V> node_source(const V* x, const ColIn<T>& r, T m_scale) {
  const V qq = caxpy(caxpy(cscale(x[0], r.cc), r.ss, x[1]), r.cs2, x[5]);
  const V qp = caxpy(cscale(csub(x[1], x[0]), r.cs), r.c2, x[5]);
  const V q3 = caxpy(cscale(x[4], r.c), r.s, x[3]);
  const V p3 = caxpy(cscale(x[3], r.c), -r.s, x[4]);
  const V d = csub(x[2], qq);
  Src<V> o;
  o.nA = caxpy_i(d, (T)-2, q3);
  o.nP = caxpy_i(d, (T)2, q3);
  o.m = cscale(cadd(x[2], qq), m_scale);
  o.aA = caxpy_i(qp, (T)1, p3);
  o.aP = caxpy_i(qp, (T)-1, p3);
  return o;
}
template <typename T, typename V> __device__ __forceinline__ void hooke_mode(V* x, T lam, T mu) {
  const V tr = cadd(cadd(x[0], x[1]), x[2]);
#pragma unroll
  for (int cc = 0; cc < 6; ++cc) x[cc] = cscale(x[cc], (T)2 * mu);
#pragma unroll
  for (int cc = 0; cc < 3; ++cc) x[cc] = caxpy(x[cc], lam, tr);
}

// L: local terms (stress: 11, 22, 12; strain: 33, 23, 13)
template <typename T, typename V>
__device__ __forceinline__ void node_out(V* o, const Br<V>& A, const Br<V>& P, const V* L, const ColOut<T>& k,
                                         const DepthMat<T>& m) {
  const V N = cadd(A.n, P.n), Vv = cadd(A.v, P.v), z = csub(A.a, P.a), sa = cadd(A.a, P.a);
  const V y = cadd(csub(A.v, P.v), csub(A.n, P.n));
  const V W = caxpy(Vv, m.w, N);
  const V g = caxpy(cscale(y, k.cy), k.sz, z);   // 13 = -i g
  const V h = caxpy(cscale(z, k.cz), -k.sy, y);  // 23 = i h
  if (m.stress) {
    o[0] = caxpy(caxpy(caxpy(L[0], k.k11w, W), k.k11n, N), k.k11a, sa);
    o[1] = caxpy(caxpy(caxpy(L[1], k.k22w, W), k.k22n, N), -k.k11a, sa);
    o[2] = cscale(Vv, k.k33);
    o[3] = mk<V>(-h.y, h.x);
    o[4] = mk<V>(g.y, -g.x);
    o[5] = caxpy(caxpy(caxpy(L[2], k.k12w, W), k.k12n, N), k.k12a, sa);
  } else {
    o[0] = caxpy(cscale(W, k.k11w), k.k11a, sa);
    o[1] = caxpy(cscale(W, k.k22w), -k.k11a, sa);
    o[2] = caxpy(L[0], k.k33, caxpy(Vv, m.t, N));
    o[3] = mk<V>(L[1].x - h.y, L[1].y + h.x);
    o[4] = mk<V>(L[2].x + g.y, L[2].y - g.x);
    o[5] = caxpy(cscale(W, k.k12w), k.k12a, sa);
  }
}
// local terms of a node from w: stress nu / (1 - nu) w_33 - w_11, .. - w_22, -w_12 (the others
// cancel); strain w_33 / (lam + 2 mu), w_23 / (2 mu), w_13 / (2 mu)
template <typename T, typename V>
__device__ __forceinline__ void node_local(V* L, const V* x, const DepthMat<T>& m) {
  if (m.stress) {
    const V t = cscale(x[2], m.la);
    L[0] = csub(t, x[0]);
    L[1] = csub(t, x[1]);
    L[2] = mk<V>(-x[5].x, -x[5].y);
  } else {
    L[0] = cscale(x[2], m.la);
    L[1] = cscale(x[3], m.iu);
    L[2] = cscale(x[4], m.iu);
  }
}
// output of a node of a mode without depth recursion: k = 0 (laminate) or outside Z^2_N (nyq)
template <typename T, typename V>
__device__ __forceinline__ void node_special(V* o, const V* w, bool nyq, const DepthMat<T>& m) {
  if (nyq) {
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) o[cc] = m.stress ? cscale(w[cc], (T)-1) : mk<V>(0, 0);
    return;
  }
  // laminate: eps_33 = w_33/(lam+2mu), eps_a3 = w_a3/(2mu), eps_ab = 0
  V e[6];
  e[0] = e[1] = e[5] = mk<V>(0, 0);
  e[2] = cscale(w[2], (T)1 / (m.lam + (T)2 * m.mu));
  e[3] = cscale(w[3], m.iu);
  e[4] = cscale(w[4], m.iu);
  if (!m.stress) {
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) o[cc] = e[cc];
    return;
  }
  const V trc = e[2];
#pragma unroll
  for (int cc = 0; cc < 6; ++cc) o[cc] = csub(cscale(e[cc], (T)2 * m.mu), w[cc]);
  o[0] = caxpy(o[0], m.lam, trc);
  o[1] = caxpy(o[1], m.lam, trc);
  o[2] = caxpy(o[2], m.lam, trc);
}

// Chunk exchange area of a tile (values per column): the carries S of the A branch and T of the
// P branch, [nch][3] each; slot R: the P moments of node 0 without their carry; slot I: the
// image field at the surface.
template <typename V, int KT> struct Xch {
  V *A, *P, *R, *I;
  __device__ __forceinline__ Xch(V* base, int nch) : A(base), P(base + (size_t)nch * 3 * KT),
      R(base + (size_t)nch * 6 * KT), I(base + (size_t)nch * 6 * KT + 3 * KT) {}
  static __host__ __device__ size_t count(int nch) { return (size_t)(6 * nch + 6) * KT; }
};
template <typename V, int KT> __device__ __forceinline__ void br_put(V* p, const Br<V>& s) {
  p[0] = s.n; p[KT] = s.v; p[2 * KT] = s.a;
}
template <typename V, int KT> __device__ __forceinline__ Br<V> br_get(const V* p) {
  Br<V> s;
  s.n = p[0]; s.v = p[KT]; s.a = p[2 * KT];
  return s;
}

// Carries into every chunk, in place over the chunks' own ones (A: arriving at the chunk's first
// node, P: at its last), then the complete P moments of node 0, the image field and the surface
// displacement.  Work item t = role KT + column, roles 0: P (n, v), 1: A (n, v), 2: P a, 3: A a.
// The column of item t is that of the calling thread (KT divides both thread counts).  Four chunks
// are read ahead of the recurrence, whose chain is then one multiply-add per chunk.  EC, EC1: on a
// uniform grid the propagators over C elements and over the first chunk's nodes.
template <typename T, int KT>
__device__ __forceinline__ void chunk_carries(const Xch<typename Cx<T>::t, KT>& X, const T* zs, int tid, int nthr, int C,
                                              int nch, int nz, T q, bool uniform, T hz, T EC, T EC1, bool live,
                                              typename Cx<T>::t* u3, T u3_scale) {
  typedef typename Cx<T>::t V;
  const int col = tid & (KT - 1);
  T Eu = 0, xu = 0;
  if (uniform) {
    xu = q * hz * (T)C;
    Eu = EC;
  }
  for (int t = tid; t < 4 * KT; t += nthr) {
    const bool isA = (t / KT) & 1, isa = t / KT >= 2;
    const int step = isA ? 3 * KT : -3 * KT;
    // components: slot 0 (n) and slot 1 (v), or slot 2 (a) alone
    V* p = (isA ? X.A : X.P + (size_t)(nch - 1) * 3 * KT) + col + (isa ? 2 * KT : 0);
    V rn = mk<V>(0, 0), rv = mk<V>(0, 0);
    for (int j0 = 0; j0 < nch; j0 += 4) {
      V sn[4], sv[4];
      T E[4], xE[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        sn[k] = sv[k] = mk<V>(0, 0);
        E[k] = Eu;
        xE[k] = xu * Eu;
        if (j0 + k < nch) {
          sn[k] = p[k * step];
          if (!isa) sv[k] = p[k * step + KT];
          if (!uniform) {
            const int n0 = (isA ? j0 + k : nch - 1 - j0 - k) * C;
            const int lo = isA ? n0 : max(n0 - 1, 0);
            const int hi = min(isA ? n0 + C : n0 + C - 1, nz - 1);
            const T x = q * (zs[hi] - zs[lo]);
            E[k] = dexp<T>(-x);
            xE[k] = x * E[k];
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (j0 + k < nch) {
          p[k * step] = rn;
          if (!isa) p[k * step + KT] = rv;
          rv = caxpy(caxpy(sv[k], -xE[k], rn), E[k], rv);
          rn = caxpy(sn[k], E[k], rn);
        }
      }
      p += 4 * step;
    }
    if (!isA && live) {
      const T x = q * (zs[min(C - 1, nz - 1)] - zs[0]);
      const T E = uniform ? EC1 : dexp<T>(-x);
      if (isa) {
        X.I[2 * KT + col] = caxpy(X.R[2 * KT + col], E, X.P[2 * KT + col]);
      } else {
        const V dn = X.P[col], dv = X.P[KT + col];
        const V n = caxpy(X.R[col], E, dn);
        const V v = caxpy(caxpy(X.R[KT + col], E, dv), -x * E, dn);
        X.I[col] = caxpy(n, (T)2, v);
        X.I[KT + col] = mk<V>(-v.x, -v.y);
        if (u3) *u3 = cscale(v, u3_scale);
      }
    }
  }
}

// ----------------------------------------------------------------------------------
// Mindlin depth kernel, shared-memory variant (FP64, deep grids, narrow grids, long chunks)
// grid: (h1 / KT, n2); block: KT * nch threads, thread = (chunk, k1 column)
// smem: W[nz][6][KT] (input, then the chunk's own moments in place; LS false: [nz][9][KT] with the
// local terms), exchange area, element coefficients, depth nodes.
// LS: at most 8 nodes per chunk, their local terms in registers.
// Bound by the FP64 pipe in FP64 (two multiply-adds per clock and SM): 1163 -> 355 us at
// 128 x 128 x 126 when the moments went from six to three per branch.
// ----------------------------------------------------------------------------------
// Gap behind each chunk's rows in shared memory: rows shorter than 128 bytes go an odd number apart from
// chunk to chunk, or the warp's chunks would meet on the same banks (an even number of nodes per chunk).
// 128 x 128 FP32 refined, us per apply, without the gaps -> with them (and every thread copying its own
// nodes, without the index divisions of a shared copy loop): 192 layers 234 -> 173, 256 324 -> 254, 288
// 400 -> 336; FP64 128 x 128 x 126 refined 1602 -> 1581.
__host__ __device__ inline int chunk_gap(int rows, int kt, int row_bytes) {
  return row_bytes < 128 && rows % 2 == 0 ? kt : 0;
}
template <typename T, int KT, bool LS>
__global__ void __launch_bounds__(256) k_mindlin_depth(typename Cx<T>::t* __restrict__ spec, typename Cx<T>::t* __restrict__ surf,
                                const T* __restrict__ zn, int nz, int n1, int n2, int hs, int h1, int C, int nch, T w1,
                                T w2, const DepthMat<T> m, int want_u3, int uniform, T hz,
                                const int* __restrict__ zr, int ein) {
  chain_begin();
  typedef typename Cx<T>::t V;
  constexpr int SL = LS ? 6 : 9, CM = LS ? 8 : 1;
  extern __shared__ __align__(128) unsigned char smraw[];  // one alignment for every kernel of this file
  const int gw = chunk_gap(C * SL, KT, KT * sizeof(V)), ge = chunk_gap(C * EL_N, KT, KT * sizeof(T)),
            gp = chunk_gap(C, KT, KT * sizeof(T));
  V* W = reinterpret_cast<V*>(smraw);                      // [nz][SL][KT], chunks gw apart
  V* xbase = W + (size_t)nz * SL * KT + (size_t)nch * gw;
  const Xch<V, KT> X(xbase, nch);
  Col<T>* cols = reinterpret_cast<Col<T>*>(xbase + Xch<V, KT>::count(nch));  // [KT]
  T* el = reinterpret_cast<T*>(cols + KT);                 // refined: [nz][6][KT], chunks ge apart
  // propagators within a chunk: uniform [C][KT], refined [nz][KT], chunks gp apart
  T* pr = el + (uniform ? (size_t)0 : (size_t)nz * EL_N * KT + (size_t)nch * ge);
  T* zs = pr + (uniform ? (size_t)C * KT : (size_t)nz * KT + (size_t)nch * gp);  // [nz] depth nodes
  const int kt = threadIdx.x & (KT - 1);
  const int ch = threadIdx.x / KT;
  const int k1 = blockIdx.x * KT + kt;
  const int k2 = blockIdx.y;
  const size_t plane = (size_t)n2 * h1;
  const size_t colofs = (size_t)k2 * h1 + blockIdx.x * KT;

  const int n0 = ch * C;
  const int nend = min(n0 + C, nz);
  const bool active = n0 < nz;
  // the thread's column in its own chunk: node i at own + i SL KT, elements and propagators likewise
  V* own = W + (size_t)ch * gw + kt;
  T* elc = el + ch * ge + kt;
  T* prc = pr + (uniform ? 0 : ch * gp) + kt;

  // 1. load the tile (every thread its own nodes, KT-wide rows, every copy in flight before one wait)
  //    and the depth nodes
  // (layers outside zr hold no input: their spectrum was not computed and reads as zero)
  const int zlo = zr ? zr[0] : 0, zhi = zr ? zr[1] : nz;
  const V* src = spec + (size_t)n0 * 6 * plane + colofs + kt;
  for (int i = n0; i < nend; ++i, src += 6 * plane) {
    V* dst = own + (size_t)i * SL * KT;
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) {
      if (i >= zlo && i < zhi) cp_async_cx(dst + cc * KT, src + cc * plane);
      else dst[cc * KT] = mk<V>(0, 0);
    }
  }
  for (int i = threadIdx.x; i < nz; i += blockDim.x) zs[i] = zn[i];
  // column constants while the tile is in flight; on a refined grid the coefficients of element e below
  // node e (none, zero, below the last node); on a uniform grid the propagators over 0 .. C - 1 elements,
  // for distances within a chunk: FP64 as powers (an exponential costs eighteen multiplications), FP32 by
  // an exponential each, as longer distances in both (one per thread and two per column): a power carries
  // the rounding of E as many times as there are elements.  Error of the operator on a smooth strain,
  // powers over the whole depth -> this: FP32 512 layers 6.1e-6 -> 5.4e-7 (powers within chunks: 8.5e-7),
  // FP64 126 layers 1.9e-15 -> 6.5e-16; 128 x 128 x 126 FP64 1320.6 -> 1322.9 us.
  if (threadIdx.x < KT) {
    col_put<T>(cols + kt, k1, k2, n1, n2, hs, w1, w2, m, uniform != 0, hz, C, zn[min(C - 1, nz - 1)] - zn[0]);
    if (uniform && sizeof(T) == 8) {
      T p = 1;
      const T E = cols[kt].in.E;
      for (int k = 0; k < C; ++k, p *= E) pr[k * KT + kt] = p;
    }
  }
  if (uniform && sizeof(T) == 4) {
    const T a = mode_geom<T>(k1, k2, n1, n2, hs, w1, w2).q * hz;
    for (int k = ch; k < C; k += nch) pr[k * KT + kt] = dexp<T>(-a * (T)k);
  }
  if (!uniform) {
    const T q = mode_geom<T>(k1, k2, n1, n2, hs, w1, w2).q;
    for (int e = n0; e < nend; ++e) {
      El<T> c = {0, 0, 0, 0, 0, 0};
      if (e + 1 < nz) c = elem_coef<T>(q, zn[e + 1] - zn[e]);
      el_put<T, KT>(elc + e * EL_N * KT, c);
    }
  }
  cp_async_wait_all();
  __syncthreads();

  const ColIn<T> g = cols[kt].in;
  const bool special = g.kind != (T)0;
  const bool work = active && !special;
  El<T> ec = g.el();
  V L[CM][3];
  // 2. own moments of the chunk: A forward (slots 0..2), the P sources kept in slots 3..5 and
  //    then replaced by the P moments, backward
  if (work) {
    Br<V> s = br_zero<V>();
    auto fwd = [&](int i, V* Li) {
      V* w = own + (size_t)i * SL * KT;
      V x[6];
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) x[cc] = w[cc * KT];
      if (ein) hooke_mode(x, m.lam, m.mu);
      const Src<V> o = node_source(x, g, m.ms);
      node_local(Li, x, m);
      if (uniform) {
        if (i > 0) br_arrive(s, ec, o.nA, o.m, o.aA);
        br_put<V, KT>(w, s);
        br_leave(s, ec, o.nA, o.m, o.aA);
      } else {
        if (i > 0) br_arrive(s, el_get<T, KT>(elc + (i - 1) * EL_N * KT - (i == n0 ? ge : 0)), o.nA, o.m, o.aA);
        br_put<V, KT>(w, s);
        br_leave(s, el_get<T, KT>(elc + i * EL_N * KT), o.nA, o.m, o.aA);
      }
      w[3 * KT] = o.nP;
      w[4 * KT] = o.m;
      w[5 * KT] = o.aP;
    };
    if constexpr (LS) {
#pragma unroll
      for (int l = 0; l < CM; ++l)
        if (l < nend - n0) fwd(n0 + l, L[l]);
    } else {
      for (int i = n0; i < nend; ++i) {
        fwd(i, L[0]);
#pragma unroll
        for (int j = 0; j < 3; ++j) own[((size_t)i * SL + 6 + j) * KT] = L[0][j];
      }
    }
    br_put<V, KT>(X.A + (size_t)ch * 3 * KT + kt, s);
    s = br_zero<V>();
    T ep = 1;  // propagator from node i to the chunk's last node
    for (int i = nend - 1; i >= n0; --i) {
      V* w = own + (size_t)i * SL * KT;
      const V sn = w[3 * KT], sm = w[4 * KT], sa = w[5 * KT];
      if (!uniform) {
        ec = el_get<T, KT>(elc + i * EL_N * KT);
        if (i + 1 < nend) ep *= ec.E;
        prc[i * KT] = ep;
      }
      if (i + 1 < nz) br_arrive(s, ec, sn, sm, sa);
      br_put<V, KT>(w + 3 * KT, s);
      if (i == 0) br_put<V, KT>(X.R + kt, s);
      // (the element above the chunk's first node is the last one of the chunk above)
      if (!uniform) ec = el_get<T, KT>(elc + max(i - 1, 0) * EL_N * KT - (i == n0 && i > 0 ? ge : 0));
      br_leave(s, ec, sn, sm, sa);
    }
    br_put<V, KT>(X.P + (size_t)ch * 3 * KT + kt, s);
  } else if (active) {
    br_put<V, KT>(X.A + (size_t)ch * 3 * KT + kt, br_zero<V>());
    br_put<V, KT>(X.P + (size_t)ch * 3 * KT + kt, br_zero<V>());
  }
  __syncthreads();

  // 3. carries, image field, surface displacement
  V* u3 = want_u3 ? surf + (size_t)k2 * h1 + k1 : nullptr;
  chunk_carries<T, KT>(X, zs, threadIdx.x, blockDim.x, C, nch, nz, g.q, uniform != 0, hz, g.EC, cols[kt].out.EC1, !special,
                       u3, m.iu);
  if (want_u3 && ch == 0 && special) *u3 = mk<V>(0, 0);
  __syncthreads();
  if (!active) return;

  // 4. complete moments, output
  V* out = spec + (size_t)n0 * 6 * plane + (size_t)k2 * h1 + k1;
  if (special) {
    for (int i = n0; i < nend; ++i, out += 6 * plane) {
      V w[6], o[6];
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) w[cc] = own[((size_t)i * SL + cc) * KT];
      if (ein) hooke_mode(w, m.lam, m.mu);
      node_special(o, w, g.kind == (T)2, m);
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) out[cc * plane] = o[cc];
    }
    return;
  }
  Br<V> cA = br_get<V, KT>(X.A + (size_t)ch * 3 * KT + kt);
  const Br<V> cP = br_get<V, KT>(X.P + (size_t)ch * 3 * KT + kt);
  {
    const T x = g.q * zs[n0], E = dexp<T>(-x);
    br_add_prop(cA, br_get<V, KT>(X.I + kt), E, x * E);
  }
  const ColOut<T> oc = cols[kt].out;
  const int last = n0 + C - 1;  // node the P carry arrives at (a ragged last chunk has none: zero)
  T EA = 1;
  auto fin = [&](int i, const V* Li) {
    V* w = own + (size_t)i * SL * KT;
    Br<V> A = br_get<V, KT>(w), P = br_get<V, KT>(w + 3 * KT);
    T xA, xP, EP;
    if (uniform) {
      xA = ec.a * (T)(i - n0);
      xP = ec.a * (T)(last - i);
      EA = prc[(i - n0) * KT];
      EP = prc[(last - i) * KT];
    } else {
      xA = g.q * (zs[i] - zs[n0]);
      xP = g.q * (zs[nend - 1] - zs[i]);
      if (i > n0) EA *= elc[(i - 1) * EL_N * KT];
      EP = prc[i * KT];
    }
    br_add_prop(A, cA, EA, xA * EA);
    br_add_prop(P, cP, EP, xP * EP);
    V o[6];
    node_out(o, A, P, Li, oc, m);
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) out[cc * plane] = o[cc];
    out += 6 * plane;
  };
  if constexpr (LS) {
#pragma unroll
    for (int l = 0; l < CM; ++l)
      if (l < nend - n0) fin(n0 + l, L[l]);
  } else {
    for (int i = n0; i < nend; ++i) {
#pragma unroll
      for (int j = 0; j < 3; ++j) L[0][j] = own[((size_t)i * SL + 6 + j) * KT];
      fin(i, L[0]);
    }
  }
}

// ----------------------------------------------------------------------------------
// Mindlin depth kernel, register variant (FP32, C <= 8 nodes per chunk, compile time): the
// chunk's own moments at its nodes stay in registers, the tile is read twice (sources, local
// terms) and never written.
// smem: W[nz][6][KT] (the tile), exchange area, element coefficients, zs[nz]
// ----------------------------------------------------------------------------------
template <typename V> __device__ __forceinline__ void ld6(V (&w)[6], const V* W, int node, int KT, int kt) {
#pragma unroll
  for (int cc = 0; cc < 6; ++cc) w[cc] = W[(node * 6 + cc) * KT + kt];
}

// Quantities that do not depend on the tile's values, computed while its copy is in flight: the
// column constants, and on a refined grid the coefficients of each chunk's own elements (element
// e below node e; zero below the last node).
template <typename T, int KT, bool UNI>
__device__ __forceinline__ void depth_prep(Col<T>* cols, T* el, const T* __restrict__ zn, int tid, int kblk, int k2, int nz,
                                           int C, int n1, int n2, int hs, T w1, T w2, const DepthMat<T>& m, T hz) {
  const int kt = tid & (KT - 1), k1 = kblk * KT + kt;
  if (tid < KT) col_put<T>(cols + kt, k1, k2, n1, n2, hs, w1, w2, m, UNI, hz, C, zn[min(C - 1, nz - 1)] - zn[0]);
  if (!UNI) {
    const T q = mode_geom<T>(k1, k2, n1, n2, hs, w1, w2).q;
    const int n0 = (tid / KT) * C, nend = min(n0 + C, nz);
    for (int e = n0; e < nend; ++e) {
      El<T> c = {0, 0, 0, 0, 0, 0};
      if (e + 1 < nz) c = elem_coef<T>(q, zn[e + 1] - zn[e]);
      el_put<T, KT>(el + e * EL_N * KT + kt, c);
    }
  }
}

// Steps 2-4 of the register depth kernel on a tile already in shared memory (W, with its exchange
// area X, element coefficients el and nodes zs).  tid = ch * KT + kt is the thread's place among
// the tile's tt threads, kblk the tile's block of KT k1 columns.  A ghost tile (a CTA slot
// without a tile) takes part in the barriers only.
template <typename T, int KT, int C, bool UNI>
__device__ __forceinline__ void depth_r_body(const typename Cx<T>::t* W, const Xch<typename Cx<T>::t, KT>& X,
                                             const Col<T>* cols, const T* el, const T* zs, int tid, int tt, int kblk, int k2, bool ghost,
                                             typename Cx<T>::t* __restrict__ spec, typename Cx<T>::t* __restrict__ surf,
                                             int nz, int n2, int h1, int nch, const DepthMat<T>& m,
                                             bool ein, int want_u3, T hz, T cut) {
  typedef typename Cx<T>::t V;
  const int kt = tid & (KT - 1);
  const int ch = tid / KT;
  const int k1 = kblk * KT + kt;
  const size_t plane = (size_t)n2 * h1;
  const ColIn<T> g = cols[kt].in;
  const bool special = g.kind != (T)0;
  const int n0 = ch * C;
  const bool active = !ghost && n0 < nz;
  const bool work = active && !special;

  // 2. own moments of the chunk at its nodes, both branches from zero, and the carries handed on.
  //    Nodes past the last one count as sources of zero, which changes nothing above them.
  Br<V> A[C], P[C];
  if (work) {
    Src<V> o[C];
#pragma unroll
    for (int l = 0; l < C; ++l) {
      if (n0 + l < nz) {
        V x[6];
        ld6(x, W, n0 + l, KT, kt);
        if (ein) hooke_mode(x, m.lam, m.mu);
        o[l] = node_source(x, g, m.ms);
      } else {
        o[l].nA = o[l].nP = o[l].m = o[l].aA = o[l].aP = mk<V>(0, 0);
      }
    }
    El<T> ec = g.el();
    // on a refined grid: element above node n0 + l, zero above node 0 and below the last node
    auto elem = [&](int e) {
      El<T> c = {0, 0, 0, 0, 0, 0};
      if (e >= 0 && e < nz) c = el_get<T, KT>(el + e * EL_N * KT + kt);
      return c;
    };
    Br<V> s = br_zero<V>();
    if (!UNI) ec = elem(n0 - 1);
#pragma unroll
    for (int l = 0; l < C; ++l) {
      if (!UNI || n0 + l > 0) br_arrive(s, ec, o[l].nA, o[l].m, o[l].aA);
      A[l] = s;
      if (!UNI) ec = elem(n0 + l);
      br_leave(s, ec, o[l].nA, o[l].m, o[l].aA);
    }
    br_put<V, KT>(X.A + ch * 3 * KT + kt, s);
    s = br_zero<V>();
#pragma unroll
    for (int l = C - 1; l >= 0; --l) {
      if (!UNI || n0 + l + 1 < nz) br_arrive(s, ec, o[l].nP, o[l].m, o[l].aP);
      P[l] = s;
      if (!UNI) ec = elem(n0 + l - 1);
      br_leave(s, ec, o[l].nP, o[l].m, o[l].aP);
    }
    br_put<V, KT>(X.P + ch * 3 * KT + kt, s);
    if (ch == 0) br_put<V, KT>(X.R + kt, P[0]);
  } else if (active) {
    br_put<V, KT>(X.A + ch * 3 * KT + kt, br_zero<V>());
    br_put<V, KT>(X.P + ch * 3 * KT + kt, br_zero<V>());
    if (ch == 0) br_put<V, KT>(X.R + kt, br_zero<V>());
  }

  // 3. carries.  Cutoff (Sec. 3.2, eps_co, restated for the recursion): when every chunk span of
  //    the tile damps by e^{-q span} < e^{-cut}, a chunk's carry is its neighbour's own one to
  //    the rounding of the path (e^{-18} < 2^-24 in FP32).  The vote is block-wide.
  const T span = (work && ch + 1 < nch) ? zs[min(n0 + C, nz - 1)] - zs[n0] : (T)0;
  const bool far = !work || ch + 1 >= nch || g.q * span > cut;
  const bool local = __syncthreads_and(cut > (T)0 && far) != 0;
  const int last = min(C - 1, nz - 1);  // last node of chunk 0
  Br<V> cA = br_zero<V>(), cP = br_zero<V>(), im;
  if (!local) {
    if (!ghost)
      chunk_carries<T, KT>(X, zs, tid, tt, C, nch, nz, g.q, UNI, hz, g.EC,
                           cols[kt].out.EC1, !special,
                           want_u3 ? surf + (size_t)k2 * h1 + k1 : nullptr, m.iu);
    __syncthreads();
    if (!active) return;
    cA = br_get<V, KT>(X.A + ch * 3 * KT + kt);
    cP = br_get<V, KT>(X.P + ch * 3 * KT + kt);
    im = br_get<V, KT>(X.I + kt);
  } else {
    if (!active) return;
    if (ch > 0) cA = br_get<V, KT>(X.A + (ch - 1) * 3 * KT + kt);
    if (ch + 1 < nch) cP = br_get<V, KT>(X.P + (ch + 1) * 3 * KT + kt);
    // complete P moments of node 0 and the image field, by every thread (no second barrier)
    Br<V> p0 = br_get<V, KT>(X.R + kt);
    if (nch > 1) {
      const T x = g.q * (zs[last] - zs[0]), E = dexp<T>(-x);
      br_add_prop(p0, br_get<V, KT>(X.P + 3 * KT + kt), E, x * E);
    }
    im.n = caxpy(p0.n, (T)2, p0.v);
    im.v = mk<V>(-p0.v.x, -p0.v.y);
    im.a = p0.a;
    if (want_u3 && ch == 0 && !special) surf[(size_t)k2 * h1 + k1] = cscale(p0.v, m.iu);
  }
  if (want_u3 && ch == 0 && special) surf[(size_t)k2 * h1 + k1] = mk<V>(0, 0);

  // 4. complete moments, output
  V* out = spec + (size_t)n0 * 6 * plane + (size_t)k2 * h1 + k1;
  if (special) {
    const int nend = min(n0 + C, nz);
    for (int i = n0; i < nend; ++i, out += 6 * plane) {
      V w[6], o[6];
      ld6(w, W, i, KT, kt);
      if (ein) hooke_mode(w, m.lam, m.mu);
      node_special(o, w, g.kind == (T)2, m);
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) out[cc * plane] = o[cc];
    }
    return;
  }
  {
    const T x = g.q * zs[n0], E = dexp<T>(-x);
    br_add_prop(cA, im, E, x * E);
  }
  // propagators from the chunk's first node (A) and to its last one (P) and q times the distances
  T EA[C], EP[C], xA[C], xP[C];
  EA[0] = EP[C - 1] = (T)1;
  xA[0] = xP[C - 1] = (T)0;
  if (UNI) {
    const T E = g.E, a = g.a;
#pragma unroll
    for (int l = 1; l < C; ++l) {
      EA[l] = EP[C - 1 - l] = EA[l - 1] * E;
      xA[l] = xP[C - 1 - l] = a * (T)l;
    }
  } else {
    T Ee[C], ae[C];
#pragma unroll
    for (int l = 0; l < C; ++l) {
      const bool in = n0 + l < nz;
      Ee[l] = in ? el[(n0 + l) * EL_N * KT + kt] : (T)0;
      ae[l] = in ? el[((n0 + l) * EL_N + 1) * KT + kt] : (T)0;
    }
#pragma unroll
    for (int l = 1; l < C; ++l) {
      EA[l] = EA[l - 1] * Ee[l - 1];
      xA[l] = xA[l - 1] + ae[l - 1];
      EP[C - 1 - l] = EP[C - l] * Ee[C - 1 - l];
      xP[C - 1 - l] = xP[C - l] + ae[C - 1 - l];
    }
  }
  const ColOut<T> oc = cols[kt].out;
#pragma unroll
  for (int l = 0; l < C; ++l) {
    if (n0 + l < nz) {
      br_add_prop(A[l], cA, EA[l], xA[l] * EA[l]);
      br_add_prop(P[l], cP, EP[l], xP[l] * EP[l]);
      V x[6], L[3], o[6];
      ld6(x, W, n0 + l, KT, kt);
      if (ein) hooke_mode(x, m.lam, m.mu);
      node_local(L, x, m);
      node_out(o, A[l], P[l], L, oc, m);
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) out[cc * plane] = o[cc];
      out += 6 * plane;
    }
  }
}

// shared memory of a register-variant tile
template <typename T, int KT> struct RegSmem {
  typedef typename Cx<T>::t V;
  static __host__ __device__ size_t el_count(int nz, int uniform) { return (size_t)(uniform ? 0 : nz) * EL_N * KT; }
  static __host__ __device__ size_t bytes(int nz, int nch, int uniform) {
    return ((size_t)nz * 6 * KT + Xch<V, KT>::count(nch)) * sizeof(V) + KT * sizeof(Col<T>) + el_count(nz, uniform) * sizeof(T) +
           (((size_t)nz * sizeof(T) + 15) & ~(size_t)15);
  }
};

template <typename T, int KT, int C, bool UNI, int MB>
__global__ void __launch_bounds__(256, MB) k_mindlin_depth_r(typename Cx<T>::t* __restrict__ spec,
                                                            typename Cx<T>::t* __restrict__ surf,
                                                            const T* __restrict__ zn, int nz, int n1, int n2, int hs, int h1, int nch,
                                                            T w1, T w2, const DepthMat<T> m, int ein, int want_u3,
                                                            T hz, const int* __restrict__ zr, T cut,
                                                            const __grid_constant__ CUtensorMap tmap, int tma_rows,
                                                            int tx_extra, int* __restrict__ status) {
  chain_begin();
  typedef typename Cx<T>::t V;
  static_assert(sizeof(V) == 8 && KT % 2 == 0, "FP32 tiles of an even width");
  extern __shared__ __align__(128) unsigned char smraw[];  // tensor-copy boxes land at 128-byte offsets
  V* W = reinterpret_cast<V*>(smraw);                               // [nz][6][KT]
  V* xbase = W + (size_t)nz * 6 * KT;
  const Xch<V, KT> X(xbase, nch);
  Col<T>* cols = reinterpret_cast<Col<T>*>(xbase + Xch<V, KT>::count(nch));  // [KT]
  T* el = reinterpret_cast<T*>(cols + KT);
  T* zs = el + RegSmem<T, KT>::el_count(nz, UNI);                   // [nz]
  // mbarrier of the tensor copies, after the depth nodes
  unsigned long long* tbar = reinterpret_cast<unsigned long long*>(smraw + RegSmem<T, KT>::bytes(nz, nch, UNI));
  const int k2 = blockIdx.y;
  const size_t plane = (size_t)n2 * h1;
  const size_t colofs = (size_t)k2 * h1 + blockIdx.x * KT;

  // 1. load the tile and the depth nodes (layers outside zr hold no input: their spectrum was
  //    not computed and reads as zero).  With a tensor map (tma_rows > 0): one thread issues
  //    tensor copies of tma_rows x KT complex boxes (rows z c, one k2, KT columns) that complete
  //    on an mbarrier; the wait is bounded, and a copy that never completes sets the status word
  //    and every thread of the CTA returns after a second bounded wait.  Otherwise 16-byte
  //    cp.async copies by all threads.
  if (tma_rows > 0) {
    const unsigned bar = (unsigned)__cvta_generic_to_shared(tbar);
    if (threadIdx.x == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned bytes = (unsigned)(nz * 6 * KT * sizeof(V) + tx_extra);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      const int x = (int)(blockIdx.x * KT * 2);  // first k1 column, in floats (16-byte multiple)
      for (int r0 = 0; r0 < nz * 6; r0 += tma_rows) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(W + (size_t)r0 * KT);
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
            "[%5];" ::"r"(dst),
            "l"(reinterpret_cast<unsigned long long>(&tmap)), "r"(x), "r"(k2), "r"(r0), "r"(bar)
            : "memory");
      }
    }
    for (int i = threadIdx.x; i < nz; i += blockDim.x) zs[i] = zn[i];
    depth_prep<T, KT, UNI>(cols, el, zn, threadIdx.x, blockIdx.x, k2, nz, C, n1, n2, hs, w1, w2, m, hz);
    bool done = mbar_wait_bounded(bar, 1000000000ull);   // 1 s
    if (__syncthreads_or(!done)) {
      if (threadIdx.x == 0 && status) atomicOr(status, 1);
      if (!done) mbar_wait_bounded(bar, 1000000000ull);  // the copies of this CTA, once more
      return;
    }
    if (zr) {
      const int zlo = zr[0], zhi = zr[1];
      for (int idx = threadIdx.x; idx < nz * 6 * KT; idx += blockDim.x) {
        const int zl = idx / (6 * KT);
        if (zl < zlo || zl >= zhi) W[idx] = mk<V>(0, 0);
      }
      __syncthreads();
    }
  } else {
    const int zlo = zr ? zr[0] : 0, zhi = zr ? zr[1] : nz;
    for (int idx = threadIdx.x; idx < nz * 6 * (KT / 2); idx += blockDim.x) {
      const int zc = idx / (KT / 2), j = 2 * (idx % (KT / 2));
      const int zl = zc / 6;
      if (zl >= zlo && zl < zhi) {
        cp_async_16(W + zc * KT + j, spec + (size_t)zc * plane + colofs + j);
      } else {
        W[zc * KT + j] = mk<V>(0, 0);
        W[zc * KT + j + 1] = mk<V>(0, 0);
      }
    }
    for (int i = threadIdx.x; i < nz; i += blockDim.x) zs[i] = zn[i];
    depth_prep<T, KT, UNI>(cols, el, zn, threadIdx.x, blockIdx.x, k2, nz, C, n1, n2, hs, w1, w2, m, hz);
    cp_async_wait_all();
    __syncthreads();
  }

  depth_r_body<T, KT, C, UNI>(W, X, cols, el, zs, threadIdx.x, blockDim.x, blockIdx.x, k2, false, spec, surf, nz, n2,
                                   h1, nch, m, ein != 0, want_u3, hz, cut);
}

// ----------------------------------------------------------------------------------
// Grouped depth kernel: the tiles of every problem of a GrpTable in one launch.  Chunks of 4
// nodes, 16-column tiles; a CTA of 256 threads holds 16 / nchp tiles of one problem (nchp:
// the chunk count rounded up to a power of two; the chunks beyond nch have no nodes), each
// with its own shared-memory slot, loaded with 16-byte cp.async copies.  The cutoff vote is
// taken over the CTA's tiles together.
// ----------------------------------------------------------------------------------
inline __host__ __device__ size_t grp_depth_slot(int nz, int nchp, int uniform) {
  return RegSmem<float, 16>::bytes(nz, nchp, uniform);
}

__global__ void __launch_bounds__(256, 2) k_grp_depth(const __grid_constant__ GrpTable tab) {
  chain_begin();
  typedef float2 V;
  constexpr int KT = 16, C = 4;
  extern __shared__ __align__(128) unsigned char smraw[];
  const int pi = grp_find(tab, blockIdx.x);
  const GrpProb& P = tab.p[pi];
  const int nz = P.nz, nchp = P.nchp, tt = KT * nchp, tpc = 256 / tt;
  const int j = threadIdx.x / tt, tid = threadIdx.x - j * tt;
  const int ncb = P.h1 / KT, tiles = ncb * P.n2;
  const int tile = ((int)blockIdx.x - tab.start[pi]) * tpc + j;
  const bool ghost = tile >= tiles;
  const int kblk = ghost ? 0 : tile % ncb, k2 = ghost ? 0 : tile / ncb;
  unsigned char* base = smraw + (size_t)j * grp_depth_slot(nz, nchp, P.uniform);
  V* W = reinterpret_cast<V*>(base);                                // [nz][6][KT]
  V* xbase = W + (size_t)nz * 6 * KT;
  const Xch<V, KT> X(xbase, nchp);
  Col<float>* cols = reinterpret_cast<Col<float>*>(xbase + Xch<V, KT>::count(nchp));  // [KT]
  float* el = reinterpret_cast<float*>(cols + KT);
  float* zs = el + RegSmem<float, KT>::el_count(nz, P.uniform);     // [nz]
  if (!ghost) {
    const size_t plane = (size_t)P.n2 * P.h1;
    const size_t colofs = (size_t)k2 * P.h1 + (size_t)kblk * KT;
    for (int idx = tid; idx < nz * 6 * (KT / 2); idx += tt) {
      const int zc = idx / (KT / 2), jj = 2 * (idx % (KT / 2));
      cp_async_16(W + zc * KT + jj, P.spec + (size_t)zc * plane + colofs + jj);
    }
    for (int i = tid; i < nz; i += tt) zs[i] = P.zn[i];
  }
  if (!ghost) {
    if (P.uniform)
      depth_prep<float, KT, true>(cols, el, P.zn, tid, kblk, k2, nz, C, P.n1, P.n2, P.hs, P.w1, P.w2, P.dm, P.hz);
    else
      depth_prep<float, KT, false>(cols, el, P.zn, tid, kblk, k2, nz, C, P.n1, P.n2, P.hs, P.w1, P.w2, P.dm, P.hz);
  }
  cp_async_wait_all();
  __syncthreads();
  // one body per grid kind: a CTA's tiles belong to one problem
  if (P.uniform)
    depth_r_body<float, KT, C, true>(W, X, cols, el, zs, tid, tt, kblk, k2, ghost, P.spec, nullptr, nz, P.n2,
                                            P.h1, P.nch, P.dm, false, 0, P.hz, P.cut);
  else
    depth_r_body<float, KT, C, false>(W, X, cols, el, zs, tid, tt, kblk, k2, ghost, P.spec, nullptr, nz, P.n2,
                                             P.h1, P.nch, P.dm, false, 0, P.hz, P.cut);
}

// strain of the Boussinesq-Cerruti field of a surface traction t (rotated frame, force on
// the body per unit area, Eq. B:fourier with its gradient recurrence) at zeta = q z
template <typename T, typename V>
__device__ __forceinline__ void bous_strain_add(const V* tr, T zeta, T ex, T nu, T imu, V* e) {
  // ex = exp(-zeta), imu = 1 / mu
  const T c1 = ex * imu, c2 = (T)0.5 * ex * imu;
  const V t0 = tr[0], t1 = tr[1], t2 = tr[2];
  // qq: ((1-nu) i t0 + (nu - 1/2) t2 + zeta(-i t0/2 + t2/2)) / mu
  //   = ((1 - nu) - zeta/2) i t0 + ((nu - 1/2) + zeta/2) t2
  V v = caxpy_i(cscale(t2, nu - (T)0.5 + (T)0.5 * zeta), (T)1 - nu - (T)0.5 * zeta, t0);
  e[0] = caxpy(e[0], c1, v);
  // 33: (-2 i nu t0 + (2nu-1) t2 + zeta (i t0 - t2)) / (2 mu)
  //   = (zeta - 2 nu) i t0 + ((2 nu - 1) - zeta) t2
  v = caxpy_i(cscale(t2, (T)2 * nu - (T)1 - zeta), zeta - (T)2 * nu, t0);
  e[2] = caxpy(e[2], c2, v);
  // p3: -t1 / (2 mu) ; qp: i t1 / (2 mu)
  e[3] = caxpy(e[3], -c2, t1);
  e[5] = caxpy_i(e[5], c2, t1);
  // q3: (-t0 + zeta (t0 + i t2)) / (2 mu) = (zeta - 1) t0 + zeta i t2
  v = caxpy_i(cscale(t0, zeta - (T)1), zeta, t2);
  e[4] = caxpy(e[4], c2, v);
}

template <typename T, typename V>
__device__ __forceinline__ void rotate_out(V* y, T c, T s) {
  const V qq = y[0], pp = y[1], p3 = y[3], q3 = y[4], qp = y[5];
  const T cc = c * c, ss = s * s, cs = c * s;
  y[0] = caxpy(caxpy(cscale(qq, cc), ss, pp), (T)-2 * cs, qp);
  y[1] = caxpy(caxpy(cscale(qq, ss), cc, pp), (T)2 * cs, qp);
  y[3] = caxpy(cscale(q3, s), c, p3);
  y[4] = caxpy(cscale(q3, c), -s, p3);
  y[5] = caxpy(caxpy(cscale(qq, cs), -cs, pp), cc - ss, qp);
}

// ----------------------------------------------------------------------------------
// Boussinesq operator of a normal pressure (Eq. B:fourier): one thread per mode, loop
// over depth.  surf holds p_hat on entry and u3_hat = 2 p_hat / (E* q) on exit.
// ----------------------------------------------------------------------------------
template <typename T>
__global__ void k_boussinesq(typename Cx<T>::t* __restrict__ spec, typename Cx<T>::t* __restrict__ surf,
                             const T* __restrict__ zn, int nz, int n1, int n2, int hs, int h1, T w1, T w2, T lam,
                             T mu, T nu, int out_kind, int want_vol, int want_u3) {
  chain_begin();
  typedef typename Cx<T>::t V;
  const int k1 = blockIdx.x * blockDim.x + threadIdx.x;
  const int k2 = blockIdx.y;
  if (k1 >= h1) return;
  const ModeGeom<T> g = mode_geom<T>(k1, k2, n1, n2, hs, w1, w2);
  const size_t plane = (size_t)n2 * h1;
  const size_t at = (size_t)k2 * h1 + k1;
  const V p = surf[at];
  if (want_vol) {
    for (int i = 0; i < nz; ++i) {
      V o[6];
      if (g.nyq) {
#pragma unroll
        for (int cc = 0; cc < 6; ++cc) o[cc] = mk<V>(0, 0);
      } else if (g.zero) {
        const V e33 = cscale(p, (T)-1 / (lam + (T)2 * mu));
#pragma unroll
        for (int cc = 0; cc < 6; ++cc) o[cc] = mk<V>(0, 0);
        if (out_kind == FVIM_STRAIN) {
          o[2] = e33;
        } else {
          o[0] = o[1] = cscale(e33, lam);
          o[2] = cscale(p, (T)-1);
        }
      } else {
        V e[6];
#pragma unroll
        for (int cc = 0; cc < 6; ++cc) e[cc] = mk<V>(0, 0);
        V tr[3] = {mk<V>(0, 0), mk<V>(0, 0), p};
        bous_strain_add<T, V>(tr, g.q * zn[i], dexp<T>(-g.q * zn[i]), nu, (T)1 / mu, e);
        if (out_kind == FVIM_STRAIN) {
#pragma unroll
          for (int cc = 0; cc < 6; ++cc) o[cc] = e[cc];
        } else {
          const V trc = cadd(e[0], e[2]);
#pragma unroll
          for (int cc = 0; cc < 6; ++cc) o[cc] = cscale(e[cc], (T)2 * mu);
          o[0] = caxpy(o[0], lam, trc);
          o[1] = caxpy(o[1], lam, trc);
          o[2] = caxpy(o[2], lam, trc);
        }
        rotate_out(o, g.c, g.s);
      }
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) spec[(size_t)(i * 6 + cc) * plane + at] = o[cc];
    }
  }
  if (want_u3) {
    V u = mk<V>(0, 0);
    if (!g.zero && !g.nyq) u = cscale(p, ((T)1 - nu) / (mu * g.q));
    surf[at] = u;
  }
}

}  // namespace

// Launch configuration of the depth kernel for chunk length C (nodes per chunk thread).
// Every valid C gives the same operator up to the rounding order of the chunk scan.
template <typename T> struct DepthCfg {
  bool ok;        // launchable (threads, shared memory)
  bool reg;       // FP32 register variant
  int C, nch, KT, threads;
  size_t smem;
  int mb;         // register variant: register budget (2: 128 registers, 3: 80, for three CTAs per SM)
};

int depth_chunk_default(int nz) {
  const int C = (nz + 15) / 16;
  return C < 2 ? 2 : C;
}

template <typename T> DepthCfg<T> depth_cfg(const fvim_ctx* c, int C, int ctas) {
  typedef typename Cx<T>::t V;
  DepthCfg<T> d{};
  const int nz = c->nz, h1 = c->h1;
  d.ok = false;
  if (C < 2 || C > nz) return d;
  // the launch limits of a plan (what fvim_set_plan accepts): 16-column tiles of [Nz][6] values and 12
  // values per chunk (register variant) or per node (shared-memory variant).  A refined grid's element
  // table comes on top of them: what is launched is sized by its own layout below
  constexpr size_t kMom = 6 * sizeof(V);
  if constexpr (sizeof(T) == 4) {
    // FP32, 16-column tiles, at most 8 nodes per chunk: the register variant (C rounded up
    // to an instantiated chunk length)
    if (h1 >= KT_MAX && C <= 8) {
      const int CR = C <= 2 ? 2 : (C <= 3 ? 3 : (C <= 4 ? 4 : (C <= 6 ? 6 : 8)));
      const int nchr = (nz + CR - 1) / CR;
      const size_t lim = (size_t)nz * 6 * 16 * sizeof(V) + (size_t)(2 * nchr) * 16 * kMom +
                         (size_t)3 * 16 * sizeof(V) + (((size_t)nz * sizeof(T) + 7) & ~(size_t)7) + 16;
      if (lim <= 227 * 1024 && 16 * nchr <= 256) {
        // three CTAs per SM (80 registers): chunk lengths 4..8; accepted by the limits, launched where the
        // tile itself fits three times (64 refined layers in chunks of 4 take 89 KB and run the 128-register
        // build, as two CTAs)
        if (ctas == 3 && !(CR >= 4 && 3 * (lim + 1024) <= 228 * 1024)) return d;
        const size_t bytes = RegSmem<T, 16>::bytes(nz, nchr, c->uniform) + 16;
        d = DepthCfg<T>{true, true, CR, nchr, 16, 16 * nchr, bytes,
                        ctas == 3 && 3 * (bytes + 1024) <= 228 * 1024 ? 3 : 2};
        return d;
      }
    }
  }
  if (ctas == 3) return d;  // the shared-memory variant has one launch shape per chunk length
  const int nch = (nz + C - 1) / C;
  const int prow = nz > 2 * nch + 1 ? nz : 2 * nch + 1;
  auto lim_of = [&](int kt) {
    return (size_t)nz * 6 * kt * sizeof(V) + (size_t)prow * kt * kMom + (size_t)nz * sizeof(T);
  };
  int KT = h1 < KT_MAX ? h1 : KT_MAX;  // h1 is a power of two or a multiple of 16
  while (KT > 2 && lim_of(KT) > 227 * 1024) KT >>= 1;
  d.ok = lim_of(KT) <= 227 * 1024 && KT * nch <= 256;
  // tile width of the launch: as wide as fits twice on an SM, and at least one 32-byte sector
  auto smem_of = [&](int kt) {
    const int sl = C <= 8 ? 6 : 9, rb = kt * (int)sizeof(T);
    const size_t vals = (size_t)nz * sl * kt + (size_t)nch * chunk_gap(C * sl, kt, 2 * rb) + 6 * (size_t)(nch + 1) * kt;
    const size_t reals = (c->uniform ? (size_t)C * kt
                                     : (size_t)nz * (EL_N + 1) * kt +
                                           (size_t)nch * (chunk_gap(C * EL_N, kt, rb) + chunk_gap(C, kt, rb))) + nz;
    return vals * sizeof(V) + kt * sizeof(Col<T>) + reals * sizeof(T);
  };
  const int kmin = 32 / (int)sizeof(V);
  while (KT > 2 && (smem_of(KT) > 227 * 1024 || (KT > kmin && smem_of(KT) > 113 * 1024))) KT >>= 1;
  d.C = C;
  d.nch = nch;
  d.KT = KT;
  d.threads = KT * nch;
  d.smem = smem_of(KT);
  d.reg = false;
  return d;
}

int depth_shape_ctas(const fvim_ctx* c, int chunk, int ctas) {
  if (c->prec == FVIM_FP64) return 0;
  const DepthCfg<float> d = depth_cfg<float>(c, chunk, ctas);
  return d.ok && d.reg ? d.mb : 0;
}

int depth_launch_ctas(const fvim_ctx* c) {
  return depth_shape_ctas(c, c->depth_chunk > 0 ? c->depth_chunk : depth_chunk_default(c->nz), c->depth_ctas);
}

bool depth_chunk_ok(const fvim_ctx* c, int C, int ctas) {
  return c->prec == FVIM_FP64 ? depth_cfg<double>(c, C, ctas).ok : depth_cfg<float>(c, C, ctas).ok;
}

template <typename T>
int launch_mindlin_depth(const fvim_ctx* c, int out_kind, bool want_u3, bool eps_in, const int* zr) {
  typedef typename Cx<T>::t V;
  const int nz = c->nz, h1 = c->h1, n2 = c->n2;
  const DepthCfg<T> d = depth_cfg<T>(c, c->depth_chunk > 0 ? c->depth_chunk : depth_chunk_default(nz), c->depth_ctas);
  if (!d.ok) return FVIM_ERR_UNSUPPORTED;
  const int KT = d.KT, C = d.C, nch = d.nch;
  dim3 grid(h1 / KT, n2);
  const T w1 = (T)(kTwoPi / c->L1), w2 = (T)(kTwoPi / c->L2);
  const DepthMat<T> dm = depth_mat<T>(c->lam, c->mu, c->nu, out_kind);
  if constexpr (sizeof(T) == 4) if (d.reg) {
    // tensor-map copies of the tile where the context has its map (rows per box divide 6 Nz)
    CUtensorMap tm;
    int tma_rows = 0;
    if (c->tmap && c->tma_rows > 0) {
      tm = *reinterpret_cast<const CUtensorMap*>(c->tmap);
      tma_rows = c->tma_rows;
    } else {
      memset(&tm, 0, sizeof(tm));
    }
#define DEPTHR(CV, UN, MBV, MBK)                                                                                \
  if (C == CV && (c->uniform != 0) == UN && d.mb == MBV) {                                                      \
    smem_cap(k_mindlin_depth_r<T, 16, CV, UN, MBK>, d.smem);                                                            \
    launch_chain(c, k_mindlin_depth_r<T, 16, CV, UN, MBK>, grid, d.threads, d.smem,                               \
        (V*)c->spec, (V*)c->surf, (const T*)c->z_dev, nz, c->n1, n2, c->hs, h1, nch, w1, w2, dm, eps_in ? 1 : 0, \
        want_u3 ? 1 : 0, (T)c->hz, zr, (T)c->depth_cut, tm, tma_rows, c->tma_test_extra,    \
        c->dev_status);                                                                                          \
  }
// Short chunks hold fewer registers: two nodes run four CTAs per SM, three nodes three, which spills 44 to
// 56 bytes and still gains on large grids (against two CTAs: 512 x 512 x 48 apply 506 -> 489 us, 1024 x
// 1024 x 36 1842 -> 1708; 128 x 128 x 48 36.2 -> 37.3).
#define DEPTHR2(CV, MBV, MBK) DEPTHR(CV, true, MBV, MBK) DEPTHR(CV, false, MBV, MBK)
    DEPTHR2(2, 2, 4) DEPTHR2(3, 2, 3) DEPTHR2(4, 2, 2) DEPTHR2(6, 2, 2) DEPTHR2(8, 2, 2)
    DEPTHR2(4, 3, 3) DEPTHR2(6, 3, 3) DEPTHR2(8, 3, 3)
#undef DEPTHR2
#undef DEPTHR
    FVIM_CUDA_CHECK_LAUNCH();
    return FVIM_OK;
  }
#define DEPTH(KTV, LSV)                                                                                        \
  if (KT == KTV && (C <= 8) == LSV) {                                                                          \
    smem_cap(k_mindlin_depth<T, KTV, LSV>, d.smem);                                                                    \
    launch_chain(c, k_mindlin_depth<T, KTV, LSV>, grid, d.threads, d.smem,                                       \
        (V*)c->spec, (V*)c->surf, (const T*)c->z_dev, nz, c->n1, n2, c->hs, h1, C, nch, w1, w2, dm,      \
        want_u3 ? 1 : 0, c->uniform, (T)c->hz, zr, eps_in ? 1 : 0);              \
  }
  DEPTH(16, true) DEPTH(8, true) DEPTH(4, true) DEPTH(2, true)
  DEPTH(16, false) DEPTH(8, false) DEPTH(4, false) DEPTH(2, false)
#undef DEPTH
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template <typename T> int launch_boussinesq(const fvim_ctx* c, int out_kind, bool want_vol, bool want_u3) {
  typedef typename Cx<T>::t V;
  const int threads = 128;
  dim3 grid((c->h1 + threads - 1) / threads, c->n2);
  launch_chain(c, k_boussinesq<T>, grid, threads, 0, (V*)c->spec, (V*)c->surf, (const T*)c->z_dev, c->nz, c->n1, c->n2,
                                                   c->hs, c->h1,
                                                   (T)(kTwoPi / c->L1), (T)(kTwoPi / c->L2), (T)c->lam, (T)c->mu, (T)c->nu,
                                                   out_kind, want_vol ? 1 : 0, want_u3 ? 1 : 0);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}

template int launch_mindlin_depth<float>(const fvim_ctx*, int, bool, bool, const int*);
template int launch_mindlin_depth<double>(const fvim_ctx*, int, bool, bool, const int*);
template int launch_boussinesq<float>(const fvim_ctx*, int, bool, bool);
template int launch_boussinesq<double>(const fvim_ctx*, int, bool, bool);

int launch_grp_depth(GrpTable& t, cudaStream_t s) {
  int b = 0;
  size_t smem = 0;
  for (int i = 0; i < t.n; ++i) {
    const GrpProb& P = t.p[i];
    const int tpc = 16 / P.nchp, tiles = (P.h1 / 16) * P.n2;
    t.start[i] = b;
    b += (tiles + tpc - 1) / tpc;
    smem = std::max(smem, (size_t)tpc * grp_depth_slot(P.nz, P.nchp, P.uniform));
  }
  t.start[t.n] = b;
  if (b == 0) return FVIM_OK;
  smem_cap(k_grp_depth, smem);
  launch_chain_on(s, true, k_grp_depth, b, 256, smem, t);
  FVIM_CUDA_CHECK_LAUNCH();
  return FVIM_OK;
}
