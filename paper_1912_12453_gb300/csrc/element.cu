// Element kernels of the matrix-free CN-VMS CHNS operator (Sec. 3.4 fully
// discrete form, Sec. 3.1 time averages) on Q1 leaves with hanging nodes
// (Sec. 4), and the small node kernels around them.
//
// Thread mapping: an element owns 2^D consecutive lanes of a warp.  Lane c is
// corner c of the element while gathering and scattering, and Gauss point c
// (xi_a = +-1/sqrt(3) by bit a of c) while evaluating the physics.  Moving
// between the two uses the tensor-product structure of Q1 with the 2-point
// Gauss rule: per axis a butterfly between the lanes that differ in that
// axis' bit (one warp shuffle), which gives values, gradients and mixed second
// derivatives at all Gauss points, and its transpose, which contracts the
// Gauss-point coefficients with N_a and grad N_a.
//
// The Jacobian-vector product evaluates the same Gauss-point physics on dual
// numbers (value, derivative along w).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "chns_internal.h"
#include "kernels.h"
#include "launch.h"

namespace chns {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------- packed pairs
// Two floats in a register pair: one packed instruction (sm_100 and later)
// does what two scalar ones do in one issue slot.
struct F2 {
  unsigned long long v;
  F2() = default;
  __device__ __forceinline__ explicit F2(float a) : F2(a, a) {}
  __device__ __forceinline__ F2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
  __device__ __forceinline__ float lo() const { return __uint_as_float(unsigned(v)); }
  __device__ __forceinline__ float hi() const { return __uint_as_float(unsigned(v >> 32)); }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 &operator*=(F2 &a, F2 b) { return a = a * b; }

// ---------------------------------------------------------------- dual numbers
// mad(a, b, c) = a b + c, one rounding per fma
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

template <typename T>
struct Dl {
  T v, d;
  __device__ __forceinline__ Dl() {}
  __device__ __forceinline__ explicit Dl(T a) : v(a), d(T(0.0f)) {}
  __device__ __forceinline__ Dl(T a, T b) : v(a), d(b) {}
};
template <typename T> __device__ __forceinline__ Dl<T> operator+(Dl<T> a, Dl<T> b) { return Dl<T>(a.v + b.v, a.d + b.d); }
template <typename T> __device__ __forceinline__ Dl<T> operator-(Dl<T> a, Dl<T> b) { return Dl<T>(a.v - b.v, a.d - b.d); }
template <typename T> __device__ __forceinline__ Dl<T> operator*(Dl<T> a, Dl<T> b) { return Dl<T>(a.v * b.v, mad(a.d, b.v, a.v * b.d)); }
template <typename T> __device__ __forceinline__ Dl<T> operator*(Dl<T> a, T b) { return Dl<T>(a.v * b, a.d * b); }
template <typename T> __device__ __forceinline__ Dl<T> mad(Dl<T> a, Dl<T> b, Dl<T> c) {
  return Dl<T>(mad(a.v, b.v, c.v), mad(a.d, b.v, mad(a.v, b.d, c.d)));
}
template <typename T> __device__ __forceinline__ Dl<T> mad(Dl<T> a, T b, Dl<T> c) {
  return Dl<T>(mad(a.v, b, c.v), mad(a.d, b, c.d));
}
// a b + c with a constant c: the derivative of c is zero
template <typename T> __device__ __forceinline__ Dl<T> madc(Dl<T> a, T b, T c) { return Dl<T>(mad(a.v, b, c), a.d * b); }
template <typename T> __device__ __forceinline__ Dl<T> madc(Dl<T> a, Dl<T> b, T c) {
  return Dl<T>(mad(a.v, b.v, c), mad(a.d, b.v, a.v * b.d));
}
template <typename T> __device__ __forceinline__ T madc(T a, T b, T c) { return mad(a, b, c); }
template <typename T> __device__ __forceinline__ Dl<T> addc(Dl<T> a, T b) { return Dl<T>(a.v + b, a.d); }
template <typename T> __device__ __forceinline__ T addc(T a, T b) { return a + b; }
template <typename T> __device__ __forceinline__ Dl<T> subc(Dl<T> a, T b) { return Dl<T>(a.v - b, a.d); }
template <typename T> __device__ __forceinline__ T subc(T a, T b) { return a - b; }
template <typename T> __device__ __forceinline__ T val(Dl<T> a) { return a.v; }
__device__ __forceinline__ float val(float a) { return a; }
__device__ __forceinline__ double val(double a) { return a; }

// conditions: one per number, two per pair
struct B2 { bool lo, hi; };
template <typename T> struct Cond { using type = bool; };
template <> struct Cond<F2> { using type = B2; };
template <typename T> __device__ __forceinline__ bool abs_le1(T x) { return fabs(x) <= T(1); }
__device__ __forceinline__ B2 abs_le1(F2 x) { return {fabsf(x.lo()) <= 1.0f, fabsf(x.hi()) <= 1.0f}; }
template <typename T> __device__ __forceinline__ bool less(T a, T b) { return a < b; }
__device__ __forceinline__ B2 less(F2 a, F2 b) { return {a.lo() < b.lo(), a.hi() < b.hi()}; }
template <typename T> __device__ __forceinline__ T sign1(T x) { return x > T(0) ? T(1) : T(-1); }
__device__ __forceinline__ F2 sign1(F2 x) { return F2(sign1(x.lo()), sign1(x.hi())); }
__device__ __forceinline__ float sel(bool c, float a, float b) { return c ? a : b; }
__device__ __forceinline__ double sel(bool c, double a, double b) { return c ? a : b; }
__device__ __forceinline__ F2 sel(B2 c, F2 a, F2 b) { return F2(c.lo ? a.lo() : b.lo(), c.hi ? a.hi() : b.hi()); }
template <typename C, typename T> __device__ __forceinline__ Dl<T> sel(C c, Dl<T> a, Dl<T> b) {
  return Dl<T>(sel(c, a.v, b.v), sel(c, a.d, b.d));
}

// -1/x and -x^(-1/2) (negated: the weak form below then needs no negation of a pair)
__device__ __forceinline__ float nrcp_(float x) { return -(1.0f / x); }
__device__ __forceinline__ double nrcp_(double x) { return -(1.0 / x); }
__device__ __forceinline__ F2 nrcp_(F2 x) { return F2(nrcp_(x.lo()), nrcp_(x.hi())); }
template <typename T> __device__ __forceinline__ Dl<T> nrcp_(Dl<T> a) {
  const T r = nrcp_(a.v);
  return Dl<T>(r, a.d * (r * r));
}
__device__ __forceinline__ float nrsqrt_(float x) { return -rsqrtf(x); }
__device__ __forceinline__ double nrsqrt_(double x) { return -rsqrt(x); }
__device__ __forceinline__ F2 nrsqrt_(F2 x) { return F2(nrsqrt_(x.lo()), nrsqrt_(x.hi())); }
// derivative 1/2 x^(-3/2) x' = -1/2 r^3 x' with r = -x^(-1/2)
template <typename T> __device__ __forceinline__ Dl<T> nrsqrt_(Dl<T> a) {
  const T r = nrsqrt_(a.v);
  return Dl<T>(r, (a.d * T(-0.5f)) * (r * r) * r);
}

// x 2^k, exact, for constants (an infinity or NaN would come out as some number).
// In double on the exponent bits: the FP64 pipe issues one
// warp instruction every 16 cycles on this part, the integer pipe is idle (x
// is zero or normal, and so is the result for box extents between 1e-60 and
// 1e60 and levels up to 20: |k| <= 80).
__device__ __forceinline__ double scale2(double x, int k) {
  const int hi = __double2hiint(x);
  return __hiloint2double((hi << 1) == 0 ? hi : hi + k * (1 << 20), __double2loint(x));
}
__device__ __forceinline__ float scale2(float x, int k) { return x * __int_as_float((127 + k) << 23); }
__device__ __forceinline__ double flip_if(double x, bool f) {
  return __hiloint2double(__double2hiint(x) ^ (f ? int(0x80000000u) : 0), __double2loint(x));
}
__device__ __forceinline__ float flip_if(float x, bool f) {
  return __int_as_float(__float_as_int(x) ^ (f ? int(0x80000000u) : 0));
}
template <typename T> __device__ __forceinline__ Dl<T> flip_if(Dl<T> x, bool f) {
  return Dl<T>(flip_if(x.v, f), flip_if(x.d, f));
}

// ---------------------------------------------------------------- butterflies
// With g = 1/sqrt(3), CA = (1 + g)/2 and CB = (1 - g)/2, a corner pair (u own,
// o other) gives CA u + CB o at the own Gauss point and (u - o)/h (signed by
// the lane's bit) as derivative.  The common factor CA is taken out of every
// stage: a stage is u + TB o (TB = CB/CA, one fma) and u - o (one add), and
// each result is scaled once at the end (values by CA^D, derivatives by
// CA^(D-1) (+-1/h)), which leaves the differences of the corner data exact.
constexpr double CA = 0.78867513459481288225;
constexpr double TB = 0.26794919243112270647;  // CB / CA = 2 - sqrt(3)
template <int D> constexpr double CAD = D == 2 ? CA * CA : CA * CA * CA;

template <int D, typename T>
struct Stage {
  T v;      // factor of values
  T sg[D];  // factors of derivatives
  T sh[D];  // +-1 / h_a
  T cS;     // W CA^D: weight of S in the contraction (W = prod h/2)
  T cV[D];  // W CA^(D-1) (+-1/h_a): weight of V_a
};

// UNIT: the stage with its factor, CA u + CB o.  phi* is clipped at |phi| = 1,
// where both bulk phases sit, and J.w jumps there: in float the branch of a
// Gauss point hangs on the last bits of phi^{k+1}.  phi~ and the phi increment
// keep this evaluation in float, so that the branches stay what they were
// before the factors were taken out.
template <bool UNIT, typename T>
__device__ __forceinline__ T st_mix(T u, T o) {
  if (UNIT) return mad(T(0.5) + T(0.28867513459481288225), u, (T(0.5) - T(0.28867513459481288225)) * o);
  return mad(T(TB), o, u);
}
template <bool UNIT = false, typename T>
__device__ __forceinline__ void st_vd(T u, int m, T &v, T &d) {
  T o = __shfl_xor_sync(FULL, u, m);
  v = st_mix<UNIT>(u, o);
  d = u - o;
}
template <bool UNIT = false, typename T>
__device__ __forceinline__ T st_v(T u, int m) {
  return st_mix<UNIT>(u, __shfl_xor_sync(FULL, u, m));
}

// value only, without its factor
template <int D, typename T>
__device__ __forceinline__ T ip_v(T u) {
  T a = st_v(u, 1);
  a = st_v(a, 2);
  if (D == 3) a = st_v(a, 4);
  return a;
}

// value and gradient
template <int D, bool UNIT = false, typename T>
__device__ __forceinline__ void ip_vg(T u, const Stage<D, T> &s, T &v, T *g) {
  T A, Bx;
  st_vd<UNIT>(u, 1, A, Bx);
  if (D == 2) {
    st_vd<UNIT>(A, 2, v, g[1]);
    g[0] = st_v<UNIT>(Bx, 2);
  } else {
    T AA, AB;
    st_vd<UNIT>(A, 2, AA, AB);
    T BA = st_v<UNIT>(Bx, 2);
    st_vd<UNIT>(AA, 4, v, g[D - 1]);
    g[1] = st_v<UNIT>(AB, 4);
    g[0] = st_v<UNIT>(BA, 4);
  }
  if (!UNIT) v *= s.v;
#pragma unroll
  for (int a = 0; a < D; ++a) g[a] *= UNIT ? s.sh[a] : s.sg[a];
}

// value, gradient and mixed second derivatives (xy; xy, xz, yz in 3D); the
// pure second derivatives of Q1 vanish on an axis-aligned box.  The second
// derivatives come out as the product of the two derivative factors.
template <int D, bool UNIT = false, typename T>
__device__ __forceinline__ void ip_full(T u, const Stage<D, T> &s, T &v, T *g, T *hs) {
  const T *f = UNIT ? s.sh : s.sg;
  T A, Bx;
  st_vd<UNIT>(u, 1, A, Bx);
  if (D == 2) {
    st_vd<UNIT>(A, 2, v, g[1]);
    st_vd<UNIT>(Bx, 2, g[0], hs[0]);
    hs[0] *= f[0] * f[1];
  } else {
    T AA, AB, BA, BB;
    st_vd<UNIT>(A, 2, AA, AB);
    st_vd<UNIT>(Bx, 2, BA, BB);
    st_vd<UNIT>(AA, 4, v, g[D - 1]);
    st_vd<UNIT>(AB, 4, g[1], hs[2]);
    st_vd<UNIT>(BA, 4, g[0], hs[1]);
    hs[0] = st_v<UNIT>(BB, 4);
    hs[0] *= f[0] * f[1];
    hs[1] *= f[0] * f[D - 1];
    hs[2] *= f[1] * f[D - 1];
  }
  if (!UNIT) v *= s.v;
#pragma unroll
  for (int a = 0; a < D; ++a) g[a] *= f[a];
}

// transpose: r_node = W sum_gp N_node(gp) S(gp) + grad N_node(gp) . V(gp)
template <int D, typename T>
__device__ __forceinline__ T contract(T S, const T *V, const Stage<D, T> &s) {
  const T tb = T(TB);
  S *= s.cS;
  const T V0 = V[0] * s.cV[0], V1 = V[1] * s.cV[1];
  T X = S + V0 + __shfl_xor_sync(FULL, mad(tb, S, -V0), 1);
  T Y1 = mad(tb, __shfl_xor_sync(FULL, V1, 1), V1);
  if (D == 2) {
    return X + Y1 + __shfl_xor_sync(FULL, mad(tb, X, -Y1), 2);
  } else {
    const T V2 = V[D - 1] * s.cV[D - 1];
    T Y2 = mad(tb, __shfl_xor_sync(FULL, V2, 1), V2);
    T X2 = X + Y1 + __shfl_xor_sync(FULL, mad(tb, X, -Y1), 2);
    T Z2 = mad(tb, __shfl_xor_sync(FULL, Y2, 2), Y2);
    return X2 + Z2 + __shfl_xor_sync(FULL, mad(tb, X2, -Z2), 4);
  }
}

// ---------------------------------------------------------------- node gather / scatter
// Node blocks are N consecutive values at p = base + node * N: for even N the
// block starts on a 2-element boundary (float2 / double2 loads), for N = 4
// floats on a 16-byte boundary (float4).
template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

template <int N, typename T>
__device__ __forceinline__ void load_block(const T *__restrict__ p, T *out) {
  if constexpr (N == 4 && sizeof(T) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
  } else if constexpr (N % 2 == 0) {
    using P = typename Pair<T>::type;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const P v = __ldg(reinterpret_cast<const P *>(p) + k);
      out[2 * k] = v.x;
      out[2 * k + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) out[k] = __ldg(p + k);
  }
}

// corner value through the hanging constraint: mean of 2 or 4 parents
template <int N, typename T>
__device__ __forceinline__ void gather(int cn, const int32_t *__restrict__ hang,
                                       const T *__restrict__ src, T *out) {
  if (cn >= 0) {
    load_block<N>(src + (int64_t)cn * N, out);
  } else {
    const int4 p = reinterpret_cast<const int4 *>(hang)[-cn - 1];
    T a[N], b[N];
    load_block<N>(src + (int64_t)p.x * N, a);
    load_block<N>(src + (int64_t)p.y * N, b);
    if (p.z < 0) {
#pragma unroll
      for (int k = 0; k < N; ++k) out[k] = T(0.5) * (a[k] + b[k]);
    } else {
      T c[N], d[N];
      load_block<N>(src + (int64_t)p.z * N, c);
      load_block<N>(src + (int64_t)p.w * N, d);
#pragma unroll
      for (int k = 0; k < N; ++k) out[k] = T(0.25) * ((a[k] + b[k]) + (c[k] + d[k]));
    }
  }
}

// Sum and increments (v and phi) of two states at a corner.  A hanging corner takes
// the mean of its parents' increments: the difference of two means would carry the
// rounding of the states, over dt, however small the step.
template <int D, typename T>
__device__ __forceinline__ void state_pair(const T *__restrict__ a, const T *__restrict__ b, T *u, T *d) {
  constexpr int NF = D + 3;
  T x[NF], y[NF];
  load_block<NF>(a, x);
  load_block<NF>(b, y);
#pragma unroll
  for (int k = 0; k < NF; ++k) u[k] = x[k] + y[k];
#pragma unroll
  for (int k = 0; k < D; ++k) d[k] = x[k] - y[k];
  d[D] = x[D + 1] - y[D + 1];
}
template <int D, typename T>
__device__ __forceinline__ void gather_states(int cn, const int32_t *__restrict__ hang, const T *__restrict__ Un,
                                              const T *__restrict__ Uo, T *u, T *d) {
  constexpr int NF = D + 3, ND = D + 1;
  auto add = [&](int p) {
    T v[NF], e[ND];
    state_pair<D>(Un + (int64_t)p * NF, Uo + (int64_t)p * NF, v, e);
#pragma unroll
    for (int k = 0; k < NF; ++k) u[k] += v[k];
#pragma unroll
    for (int k = 0; k < ND; ++k) d[k] += e[k];
  };
  const bool hangs = cn < 0;
  const int4 p = hangs ? reinterpret_cast<const int4 *>(hang)[-cn - 1] : make_int4(cn, -1, -1, -1);
  state_pair<D>(Un + (int64_t)p.x * NF, Uo + (int64_t)p.x * NF, u, d);
  if (hangs) {
    add(p.y);
    T f = T(0.5);
    if (p.z >= 0) {
      add(p.z);
      add(p.w);
      f = T(0.25);
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) u[k] *= f;
#pragma unroll
    for (int k = 0; k < ND; ++k) d[k] *= f;
  }
}

template <int N, typename T, typename O>
__device__ __forceinline__ void add_block(O *__restrict__ p, const T *r, T wgt) {
  if constexpr (N % 2 == 0) {
    using P = typename Pair<O>::type;
    P *q = reinterpret_cast<P *>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      P v = q[k];
      v.x += O(wgt * r[2 * k]);
      v.y += O(wgt * r[2 * k + 1]);
      q[k] = v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] += O(wgt * r[k]);
  }
}

template <int N, typename T>
__device__ __forceinline__ void store_block(T *__restrict__ p, const T *r) {
  if constexpr (N % 2 == 0) {
    using P = typename Pair<T>::type;
    P *q = reinterpret_cast<P *>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      P v;
      v.x = r[2 * k];
      v.y = r[2 * k + 1];
      q[k] = v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = r[k];
  }
}

// non-atomic: elements of one launch (one colour) touch disjoint nodes
template <int N, typename T, typename O>
__device__ __forceinline__ void scatter(int cn, const int32_t *__restrict__ hang, O *__restrict__ dst,
                                        const T *r) {
  if (cn >= 0) {
    add_block<N>(dst + (int64_t)cn * N, r, T(1));
  } else {
    const int4 p = reinterpret_cast<const int4 *>(hang)[-cn - 1];
    T wgt = p.z < 0 ? T(0.5) : T(0.25);
    add_block<N>(dst + (int64_t)p.x * N, r, wgt);
    add_block<N>(dst + (int64_t)p.y * N, r, wgt);
    if (p.z >= 0) {
      add_block<N>(dst + (int64_t)p.z * N, r, wgt);
      add_block<N>(dst + (int64_t)p.w * N, r, wgt);
    }
  }
}

// ---------------------------------------------------------------- Gauss-point physics
template <int D, typename S>
struct GpIn {
  S vt[D], dvt[D][D];  // v~ and d_j v~_i (dvt[i][j])
  S pt, dpt[D];        // p~
  S phit, dphit[D], hphit[3];  // phi~, gradient, mixed second derivatives
  S mut, dmut[D];      // mu~
  S dv[D];             // v^{k+1} - v^k
  S dphi;              // phi^{k+1} - phi^k
  S phin, dphin[D];    // phi^{k+1} and its gradient
};

// Everything that depends only on the parameters and the box is folded on the
// host; what depends on the leaf is a power of two of its level.  Some are
// kept negated (n...): a pair has no negation for free.
template <typename T>
struct KEnd {      // float, and pairs of floats
  T end, inv_dtp;  // see kcoef
};
template <> struct KEnd<double> {};
template <typename T>
struct KPhys : KEnd<T> {
  T inv_dt, four_dt2, alpha, beta;
  T ngRe, gRe, xRe;        // eta / Re = gRe phi* + xRe (float: phi* + end, see kcoef)
  T jcP;                   // J / Pe = jcP grad mu
  T inv_We, ninv_We, CnWe, nCnWe, inv_PeCn, Cn2;
  T ngFr[3];               // - gravity / Fr
};
template <typename T> struct KBox {};
template <> struct KBox<double> {
  double f0, rf0, nk, rowp0;  // see kcube
};
template <typename T>
struct KCoef : KPhys<T>, KBox<T> {
  // geometry of a leaf of level 0; a leaf of level l has these times a power of 2^l
  T nG0[3];                // - G = - 4 / ext^2
  T CIGG0, inv_trG0;       // C_I G:G and 1 / tr G
  T sg0[3], sh0[3], cS0, cV0[3];  // Stage without the signs
  T W0;                    // prod ext / 2
};

template <int D> __device__ __forceinline__ int hidx(int i, int j) {
  // index of the mixed derivative d_i d_j (i != j) in hphit
  return D == 2 ? 0 : (i + j - 1);
}

// Weak-form coefficients at one Gauss point: the row of test function N_a
// receives W (N_a Sq[k] + sum_j d_j N_a Vq[k][j]) for equation k.  f: the
// nodal source at the Gauss point (HASF).  CnWeH: Cn/We over the factor left in
// hphit.  floored: whether the tau_m
// radicand was raised to 4/dt^2.
//
// The terms of Sec. 3.4 share factors.  With A_i = rho (dv_i/dt - g_i/Fr) - f_i,
// c_j = rho v~_j + J_j/Pe and t_i = tau_m R_m,i:
//   R_m,i        = A_i + d_j v~_i (c_j - d_j eta/Re) + capillary_i + d_i p~/We,
//   momentum S_i = A_i + d_j v~_i (c_j - t_j)
//                  (advection, flux and cross stress in one product),
//   momentum V_ij = (t_i/rho) (c_j - t_j) - Cn/We d_i phi~ d_j phi~ + eta/Re d_j v~_i
//                  (streamline, Reynolds and flux stabilisation in one product),
//   v~.G v~ + v~.G J/(rho Pe) = (1/rho) sum_i G_i v~_i c_i.
// That takes two matrix-vector products instead of four, one outer product
// instead of three, and the two quotients 1/rho and rad^(-1/2) only (tau_c =
// sqrt(rad)/tr G = rad tau_m/tr G).  Every quotient of the geometry is a power
// of two times a constant of the box.  In double bound by the FP64 pipe (86 % busy):
// residual of the level-6 octree (262,144 leaves) 1.41 ms, J.w of 77,932 adaptive
// leaves 0.75 ms, each with its node gather (CUBE: 1.26 and 0.68); term by term as
// in Sec. 3.4 and with a division per quotient of the geometry, 2.34 and 1.27 ms.
//
// nG, CI_GG, inv_trG, CnWeH come per leaf; T is the number type (a pair: two
// Gauss points), S is T or its dual.
//
// CUBE: a 3D box with equal sides (FP64; c: KCube).  Gradients come as plain
// differences of the corner data along the lane's own axes (own minus other
// corner: axis a is reversed where c.neg[a]), so d_a = f sign_a x difference with
// one f per leaf, and the factors sit in the constants: vt is f sign_i v~_i, cm is
// f sign_j c_j, V comes out for plain differences of the test functions, the
// continuity row over f.  Signs of the vector components that are not summed over
// are flipped back on the bits.  That saves the products of 21 gradients, three
// mixed derivatives and 18 contraction weights: 315 FP64 instructions a lane in the
// residual (general form 352), 557 in J.w (616).  Error against plain double code:
// residual 2.5e-16 (general form 2.7e-16; 7.3e-16 both with hanging nodes), J.w
// 2.6e-16 both.  In 2D J.w would go from 1.5e-16 to 1.7e-16, so 2D keeps the general
// form; so do other boxes, and union meshes, whose constants come from a table.
template <int D, bool HASF, bool CUBE, typename T, typename S, typename C>
__device__ __forceinline__ void gp_physics(const C &c, const T *nG, T CI_GG, T inv_trG, T CnWeH,
                                           const GpIn<D, S> &q, const T *f, S *Sq, S (*Vq)[D],
                                           typename Cond<T>::type &floored) {
  // phi* clip (Eq. phi_for_density) and mixture properties at t_{k+1}
  const T pn = val(q.phin);
  const auto inside = abs_le1(pn);
  S phis = sel(inside, q.phin, S(sign1(pn)));
  constexpr bool DBL = std::is_same<T, double>::value;
  if constexpr (!DBL) phis = addc(phis, c.end);
  const S rho = madc(phis, c.alpha, c.beta);
  const S etaRe = madc(phis, c.gRe, c.xRe);
  const S ninv_rho = nrcp_(rho);
  S cm[D], cR[D];  // c_j and c_j - d_j eta / Re
#pragma unroll
  for (int j = 0; j < D; ++j) {
    cm[j] = mad(rho, q.vt[j], q.dmut[j] * c.jcP);
    cR[j] = cm[j] + sel(inside, q.dphin[j] * c.ngRe, S(T(0.0f)));
  }
  // tau_m, tau_c with G = diag(4/h^2); radicand floored at 4/dt^2
  S nvGc = (q.vt[0] * cm[0]) * nG[0];
#pragma unroll
  for (int i = 1; i < D; ++i) nvGc = mad(q.vt[i] * cm[i], nG[i], nvGc);
  const S nvisc = etaRe * ninv_rho;
  S rad = mad(ninv_rho, nvGc, madc(nvisc * nvisc, CI_GG, c.four_dt2));
  floored = less(val(rad), c.four_dt2);
  rad = sel(floored, S(c.four_dt2), rad);
  const S ntau = nrsqrt_(rad);
  // strong residuals
  S A[D], nt[D];  // nt = - tau_m R_m
  S divv;
  if constexpr (CUBE) {
    divv = flip_if(q.dvt[0][0], c.neg[0]);
#pragma unroll
    for (int i = 1; i < D; ++i) divv = divv + flip_if(q.dvt[i][i], c.neg[i]);
  } else {
    divv = q.dvt[0][0];
#pragma unroll
    for (int i = 1; i < D; ++i) divv = divv + q.dvt[i][i];
  }
  if constexpr (HASF && CUBE) divv = subc(divv, f[D] * c.rf);
  else if (HASF) divv = subc(divv, f[D]);  // R_c
#pragma unroll
  for (int i = 0; i < D; ++i) {
    A[i] = rho * madc(q.dv[i], c.inv_dt, c.ngFr[i]);
    if (HASF) A[i] = subc(A[i], f[i]);
    S R;
    if constexpr (CUBE) R = mad(flip_if(q.dpt[i], c.neg[i]), c.inv_We, A[i]);
    else R = mad(q.dpt[i], c.inv_We, A[i]);
    S cap = D == 2 ? q.hphit[0] * q.dphit[1 - i] : S(T(0.0f));
    if (D == 3) {
      const int j0 = i == 0 ? 1 : 0, j1 = i == 2 ? 1 : 2;
      cap = mad(q.hphit[hidx<D>(i, j0)], q.dphit[j0], q.hphit[hidx<D>(i, j1)] * q.dphit[j1 < D ? j1 : 0]);
    }
    if constexpr (CUBE) cap = flip_if(cap, c.neg[i]);
    R = mad(cap, CnWeH, R);
#pragma unroll
    for (int j = 0; j < D; ++j) R = mad(q.dvt[i][j], cR[j], R);
    nt[i] = ntau * R;
  }
  // momentum rows
  const S ntau_c = (rad * ntau) * inv_trG;
  const S diag = mad(rho * ntau_c, divv, q.pt) * c.ninv_We;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    if constexpr (CUBE) cm[j] = mad(nt[j], c.fs[j], cm[j]);
    else cm[j] = cm[j] + nt[j];
  }
  S cphi[D];
#pragma unroll
  for (int i = 0; i < D; ++i) cphi[i] = q.dphit[i] * c.nCnWe;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    S Si = A[i];
#pragma unroll
    for (int j = 0; j < D; ++j) Si = mad(q.dvt[i][j], cm[j], Si);
    Sq[i] = Si;
    if constexpr (CUBE) Vq[D][i] = nt[i] * (ninv_rho * c.nk);
    else Vq[D][i] = nt[i] * ninv_rho;  // PSPG; tau_m R_m / rho
  }
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = i; j < D; ++j) {
      S cc = cphi[i] * q.dphit[j];
      if (i == j) cc = cc + diag;
      if constexpr (CUBE) {
        Vq[i][j] = mad(Vq[D][i], cm[j], mad(etaRe, q.dvt[i][j], flip_if(cc, c.neg[i])));
        if (i != j) Vq[j][i] = mad(Vq[D][j], cm[i], mad(etaRe, q.dvt[j][i], flip_if(cc, c.neg[j])));
      } else {
        Vq[i][j] = mad(Vq[D][i], cm[j], mad(etaRe, q.dvt[i][j], cc));
        if (i != j) Vq[j][i] = mad(Vq[D][j], cm[i], mad(etaRe, q.dvt[j][i], cc));
      }
    }
  if constexpr (CUBE)
#pragma unroll
    for (int i = 0; i < D; ++i) Vq[D][i] = flip_if(Vq[D][i], c.neg[i]);
  // continuity row
  Sq[D] = divv;
  // Cahn-Hilliard row
  if constexpr (DBL) Sq[D + 1] = q.dphi * c.inv_dt;
  else Sq[D + 1] = q.dphi * c.inv_dtp;
  S nphi;
  if constexpr (CUBE) nphi = q.phit * -c.nk;
  else nphi = q.phit * T(-1.0f);
#pragma unroll
  for (int i = 0; i < D; ++i) Vq[D + 1][i] = mad(q.vt[i], nphi, q.dmut[i] * c.inv_PeCn);
  // chemical-potential row, psi'(phi~) = phi~^3 - phi~
  Sq[D + 2] = q.phit * madc(q.phit, q.phit, T(-1.0f)) - q.mut;
#pragma unroll
  for (int i = 0; i < D; ++i) Vq[D + 2][i] = q.dphit[i] * c.Cn2;
  if (HASF) {
    Sq[D + 1] = subc(Sq[D + 1], f[D + 1]);
    Sq[D + 2] = subc(Sq[D + 2], f[D + 2]);
  }
}

template <int D, typename T>
struct Interp {  // one state interpolated at the lane's Gauss point
  T vt[D], dvt[D][D], pt, dpt[D], phit, dphit[D], hphit[3], mut, dmut[D];
};

// vs: factors of the velocity components (CUBE; others: the stage's)
template <int D, bool UNIT, bool CUBE = false, typename T>
__device__ __forceinline__ void interp_state(const T *u, const Stage<D, T> &s, Interp<D, T> &I,
                                             const T *vs = nullptr) {
#pragma unroll
  for (int i = 0; i < D; ++i) {
    Stage<D, T> si = s;
    if (CUBE) si.v = vs[i];
    ip_vg<D>(u[i], si, I.vt[i], I.dvt[i]);
  }
  ip_vg<D>(u[D], s, I.pt, I.dpt);
  I.hphit[1] = I.hphit[2] = T(0);
  ip_full<D, UNIT>(u[D + 1], s, I.phit, I.dphit, I.hphit);
  ip_vg<D>(u[D + 2], s, I.mut, I.dmut);
}

// The constants of the CUBE form, per leaf: those of kcube with the powers of two
// of the level
template <int D>
struct KCube : KPhys<double> {
  double f, rf, nk, fs[D];  // f, 1 / f, factor of V, f with the signs
  bool neg[D];
};

// Constants of a box with equal sides, gradients as plain differences (see
// gp_physics).  f = CA^(D-1) / h of level 0 is the factor of a gradient (half of
// it for the residual, which sums two states), ft that of the test functions'
// gradients; the contraction applies CA^D W to a row, so V is over CA^D.  Formed
// from the side in extended precision and rounded once: a constant's error is the
// same at every Gauss point, and of f it would enter to the third power.  Errors of
// the factors on the way are taken out as in kcoef.
KCoef<double> kcube(const PhysCoef &p, KCoef<double> c, bool raw) {
  typedef long double R;
  const R ca = R(0.5) + R(0.28867513459481288225457439025L), cad = ca * ca * ca;
  const R ext = p.ext[0], ft = ca * ca / ext, f = raw ? ft / 2 : ft, v = ft / cad;
  const R bv = R(CAD<3>) / cad;  // of values, as in kcoef
  const R W = ext * ext * ext / 8;
  c.cS0 = double(W * cad);
  const R bS = R(c.cS0) / (W * cad), G = 4 / (ext * ext);
  c.inv_dt = double(1 / (R(p.dt) * bv));
  c.jcP = double(R(p.jc) * p.inv_Pe * f * f);
  c.ngRe = double(-R(p.gamma) * p.inv_Re * f * f);
  c.gRe = double(R(p.gamma) * p.inv_Re * v * f / bS);
  c.xRe = double(R(p.xi) * p.inv_Re * v * f / bS);
  for (int a = 0; a < 3; ++a) {
    c.nG0[a] = double(-G / (f * f));
    c.ngFr[a] = double(-R(p.g[a]) * p.inv_Fr / bS);
  }
  c.CIGG0 = double(R(p.C_I) * 3 * G * G / (v * f * v * f) * bS * bS);
  c.inv_trG0 = double(f / (3 * G));
  c.CnWe = double(R(p.CnWe) * (raw ? 2 : 1) / cad * f * f * f);
  c.nCnWe = double(-R(p.CnWe) * v * f * f / bS);
  c.inv_We = double(R(p.inv_We) * f);
  c.ninv_We = double(-R(p.inv_We) * v / (bv * bS));
  c.inv_PeCn = double(R(p.inv_PeCn) * v * f / bS);
  c.Cn2 = double(R(p.Cn2) * v * f / bS);
  c.f0 = double(f);
  c.rf0 = double(1 / f);
  c.nk = double(v / f);
  c.rowp0 = double(W * cad * f);
  return c;
}
template <typename T>
bool is_cube(const KCoef<T> &c) { return c.sg0[0] == c.sg0[1] && c.sg0[0] == c.sg0[2]; }

// A constant's rounding is the same at every Gauss point: it shifts a whole row,
// where the roundings of the values average out (CA^2 as a float is off by 4e-8, once
// in a gradient and once in the test function's; CA^3 as a double by 4.7e-17).
//  - Each product's constant is over the errors of the rounded factors that its
//    terms meet on their way (values, gradients, test functions; the mean over the
//    axes), so that a term is off by the last rounding only.
//  - In float rho and eta are straight lines over phi* + end, from the lighter
//    phase's end of the range: alpha phi* + beta leaves the light phase with the
//    errors of two numbers that nearly cancel (2e-7 of rho at a ratio of 0.1).
// Error without -> with, geometric means over meshes and parameters of the tests'
// kind.  Float J.w against double: 2D -14 % (up to -44 %), 3D -5 %, momentum rows of
// a light phase by half; time -0.8 % (2D) to +0.7 % (3D with hanging nodes).  Double
// against 80 bits: J.w 2D -3 %, cubes (kcube) -7 %, residual of cubes -4 %.
// Errors are held as such, in double: long double is software on Arm, 2 us a call.
template <typename T>
void fit_constants(const PhysCoef &p, int dim, double W, double GG, KCoef<T> &c) {
  constexpr bool F = sizeof(T) == 4;
  constexpr long double ca = 0.5L + 0.28867513459481288225457439025L, ca2 = ca * ca, ca3 = ca2 * ca;
  constexpr double hi[3] = {double(ca), double(ca2), double(ca3)};
  constexpr double lo[3] = {double(ca - hi[0]), double(ca2 - hi[1]), double(ca3 - hi[2])};
  // error of x k as CA^n; of no use where x is beyond the range of T
  auto error = [&](double x, double k, int n) {
    const double e = (std::fma(x, k, -hi[n - 1]) - lo[n - 1]) / hi[n - 1];
    return std::fabs(e) < 1e-6 ? e : 0.0;
  };
  auto fit = [](double x, double e) { return T(std::fma(-e, x, x)); };  // x over 1 + e
  const double ev = error(T(dim == 2 ? CAD<2> : CAD<3>), 1.0, dim);  // of values
  double eg = 0.0, eh = 0.0, eV = 0.0;  // of gradients (in float phi's has 1/h alone), of test gradients
  for (int a = 0; a < dim; ++a) {
    const double x = p.ext[a], g = error(c.sg0[a], x, dim - 1), h = std::fma(double(c.sh0[a]), x, -1.0);
    c.cV0[a] = fit(W * hi[dim - 2] / x, F ? 0.0 : g);
    eg += g / dim;
    eh += (F ? (std::fabs(h) < 1e-6 ? h : 0.0) : g) / dim;
    eV += error(c.cV0[a], x / W, dim - 1) / dim;
  }
  // a value meets ev and eS; in float phi and its increment eS only.  In double 1/dt
  // leaves eS: the strong residual in the continuity row then matches div v
  c.cS0 = fit(W * hi[dim - 1], F ? 0.5 * ev : 0.0);
  const double eS = error(c.cS0, 1.0 / W, dim), et = std::fma(p.inv_dt, p.dt, -1.0);
  c.inv_dt = fit(p.inv_dt, et + ev + (F ? eS : 0.0));
  if constexpr (F) c.inv_dtp = fit(p.inv_dt, et + eS);
  for (int a = 0; a < 3; ++a) c.ngFr[a] = fit(-p.g[a] * p.inv_Fr, eS);
  c.jcP = fit(p.jc * p.inv_Pe, eg);
  c.inv_We = fit(p.inv_We, eg);
  c.ninv_We = fit(-p.inv_We, ev + eV);
  c.CnWe = fit(p.CnWe, F ? 3 * eh : 3 * eh - ev);  // in double 1 / CA^D follows
  c.nCnWe = fit(-p.CnWe, 2 * eh + eV);
  c.inv_PeCn = fit(p.inv_PeCn, eg + eV);
  c.Cn2 = fit(p.Cn2, eh + eV);
  c.ngRe = fit(-p.gamma * p.inv_Re, eg + eh);
  c.CIGG0 = fit(p.C_I * GG, -2.0 * (eg + eV));
  c.gRe = fit(p.gamma * p.inv_Re, eg + eV);
  double xi = p.xi;
  if constexpr (F) {
    c.end = p.alpha >= 0.0 ? 1.0f : -1.0f;
    c.beta = T(p.beta - c.end * p.alpha);
    xi -= c.end * p.gamma;
  }
  c.xRe = fit(xi * p.inv_Re, eg + eV);
}

template <typename T>
KCoef<T> kcoef(const PhysCoef &p, int dim) {
  KCoef<T> c{};
  c.four_dt2 = T(p.four_dt2);
  c.alpha = T(p.alpha);
  c.beta = T(p.beta);
  const double cad1 = dim == 2 ? CA : CA * CA;  // CA^(D-1)
  double trG = 0.0, GG = 0.0, W = 1.0;
  for (int a = 0; a < 3; ++a) {
    const double G = 4.0 / (p.ext[a] * p.ext[a]);
    c.nG0[a] = T(-G);
    c.sg0[a] = T(cad1 / p.ext[a]);
    c.sh0[a] = T(1.0 / p.ext[a]);
    if (a < dim) {
      trG += G;
      GG += G * G;
      W *= 0.5 * p.ext[a];
    }
  }
  c.inv_trG0 = T(1.0 / trG);
  c.W0 = T(W);
  fit_constants<T>(p, dim, W, GG, c);
  return c;
}

// ---------------------------------------------------------------- the element kernel
// MODE 0: residual into the element-local slots; MODE 1: J.w into the
// element-local slots; MODE 2: count of the Gauss points whose tau_m radicand
// is floored (O = unsigned long long, one counter); MODE 3: J.w scattered into
// the node vector (one launch per element colour,
// elements eperm[e_begin..e_end)).  MODE 0 and 2 read the
// states themselves (ut = U_new, dl = U_old: they are evaluated once per
// state), the J.w modes the prepared averages and increments.  MODE 1 takes
// gridDim.y directions at a time (w and out at strides).  BS, MINB: block size
// and minimum resident blocks per SM (the register budget).
template <int D, typename T, int MODE, bool HASF, typename O, int BS = 128, int MINB = 6, bool CUBE = false>
__global__ void __launch_bounds__(BS, MINB) k_element(
    const int32_t *__restrict__ conn, const uint8_t *__restrict__ level,
    const int32_t *__restrict__ hang, int64_t e_begin, int64_t e_end,
    const T *__restrict__ ut, const T *__restrict__ dl, const T *__restrict__ w,
    const T *__restrict__ f, O *__restrict__ out, KCoef<T> c0, const KCoef<T> *__restrict__ tab,
    const uint16_t *__restrict__ einst, int64_t wstride, int64_t ostride, const int32_t *__restrict__ eperm) {
  constexpr int NC = 1 << D, NF = D + 3, ND = D + 1;
  constexpr bool UNIT = sizeof(T) == 4, RAW = MODE == 0 || MODE == 2;
  static_assert(!(UNIT && RAW), "the residual is in double");
  static_assert(!CUBE || (!UNIT && D == 3 && (MODE == 0 || MODE == 1)), "FP64, one coefficient set");
  const int lc = threadIdx.x & (NC - 1);
  int64_t e = e_begin + ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> D);
  const bool active = e < e_end;
  if (!active) e = e_end - 1;  // keep the lanes alive for the shuffles
  if (MODE == 3) e = eperm[e];
  const int cn = conn[e * NC + lc];
  // batched meshes: the coefficients of the element's own problem instance
  const KCoef<T> c = tab ? tab[einst[e]] : c0;

  const int l = level[e];
  wait_previous(ut, dl, w, f, out);
  if (MODE == 1) {
    w += blockIdx.y * wstride;
    out += blockIdx.y * ostride;
  }

  // gather the corner's nodal blocks (MODE 0, 2: the sum of the states, twice
  // the average; the factors of the interpolation carry the half)
  T u[NF], d[ND];
  if constexpr (RAW) {
    gather_states<D>(cn, hang, ut, dl, u, d);
  } else {
    gather<NF>(cn, hang, ut, u);
    gather<ND>(cn, hang, dl, d);
  }
  T wn[NF];
  if (MODE == 1 || MODE == 3) gather<NF>(cn, hang, w, wn);
  T fn[NF];
  if (HASF) gather<NF>(cn, hang, f, fn);

  // geometry of this leaf
  Stage<D, T> s;
  T nG[D], vs[D], row = T(0), rowp = T(0);
  KCube<D> kc;
  s.v = T((RAW ? 0.5 : 1.0) * CAD<D>);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const bool neg = !((lc >> a) & 1);
    if constexpr (CUBE) {
      kc.neg[a] = neg;
      kc.fs[a] = flip_if(scale2(c.f0, l), neg);
      vs[a] = kc.fs[a] * s.v;
      s.sg[a] = s.sh[a] = s.cV[a] = T(1);  // folded away
      nG[a] = c.nG0[a];
    } else {
      s.sg[a] = flip_if(scale2(c.sg0[a], l - (RAW ? 1 : 0)), neg);
      s.sh[a] = UNIT ? flip_if(scale2(c.sh0[a], l), neg) : T(0);
      s.cV[a] = flip_if(scale2(c.cV0[a], (1 - D) * l - (RAW ? 0 : 1)), neg);
      nG[a] = scale2(c.nG0[a], 2 * l);
    }
  }
  T CI_GG, inv_trG, CnWeH;
  if constexpr (CUBE) {
    kc.inv_dt = c.inv_dt; kc.four_dt2 = c.four_dt2; kc.alpha = c.alpha; kc.beta = c.beta;
    for (int a = 0; a < 3; ++a) kc.ngFr[a] = c.ngFr[a];
    kc.jcP = scale2(c.jcP, 2 * l);
    kc.ngRe = scale2(c.ngRe, 2 * l);
    kc.gRe = scale2(c.gRe, 2 * l);
    kc.xRe = scale2(c.xRe, 2 * l);
    kc.nCnWe = scale2(c.nCnWe, 3 * l);
    kc.inv_We = scale2(c.inv_We, l);
    kc.ninv_We = scale2(c.ninv_We, l);
    kc.inv_PeCn = scale2(c.inv_PeCn, 2 * l);
    kc.Cn2 = scale2(c.Cn2, 2 * l);
    kc.f = scale2(c.f0, l);
    kc.rf = scale2(c.rf0, -l);
    kc.nk = c.nk;
    s.cS = T(1);
    row = scale2(c.cS0, -D * l - (RAW ? 0 : 1));
    rowp = scale2(c.rowp0, (1 - D) * l - (RAW ? 0 : 1));
    CI_GG = c.CIGG0;
    inv_trG = scale2(c.inv_trG0, -l);
    CnWeH = scale2(c.CnWe, 3 * l);
  } else {
    s.cS = scale2(c.cS0, -D * l - (RAW ? 0 : 1));
    CI_GG = scale2(c.CIGG0, 4 * l);
    inv_trG = scale2(c.inv_trG0, -2 * l);
    // d_a d_b = sg_a sg_b / CA^D (half of it with the halved factors)
    CnWeH = UNIT ? c.CnWe : c.CnWe * T((RAW ? 2.0 : 1.0) / CAD<D>);
  }

  // interpolate to the lane's Gauss point
  Interp<D, T> A;
  interp_state<D, UNIT, CUBE>(u, s, A, vs);
  T dvq[D], dphiq, dphig[D];
#pragma unroll
  for (int i = 0; i < D; ++i) dvq[i] = ip_v<D>(d[i]) * T(CAD<D>);
  ip_vg<D, UNIT>(d[D], s, dphiq, dphig);
  T fq[NF];
#pragma unroll
  for (int k = 0; k < NF; ++k) fq[k] = HASF ? ip_v<D>(fn[k]) * T(CAD<D>) : T(0);

  T r[NF];
  bool floored = false;
  if (RAW) {
    // dphiq, dphig: half the increment and half its gradient
    GpIn<D, T> q;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      q.vt[i] = A.vt[i];
      q.dv[i] = dvq[i];
      q.dpt[i] = A.dpt[i];
      q.dphit[i] = A.dphit[i];
      q.dmut[i] = A.dmut[i];
      q.dphin[i] = A.dphit[i] + dphig[i];
#pragma unroll
      for (int j = 0; j < D; ++j) q.dvt[i][j] = A.dvt[i][j];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) q.hphit[k] = A.hphit[k];
    q.pt = A.pt;
    q.phit = A.phit;
    q.mut = A.mut;
    q.dphi = T(2) * dphiq;
    q.phin = A.phit + dphiq;
    T Sq[NF], Vq[NF][D];
    if constexpr (CUBE) gp_physics<D, HASF, true, T, T>(kc, nG, CI_GG, inv_trG, CnWeH, q, fq, Sq, Vq, floored);
    else gp_physics<D, HASF, false, T, T>(c, nG, CI_GG, inv_trG, CnWeH, q, fq, Sq, Vq, floored);
    if constexpr (MODE == 2) {
      const unsigned b = __ballot_sync(FULL, floored && active);
      if ((threadIdx.x & 31) == 0 && b) atomicAdd(reinterpret_cast<unsigned long long *>(out), (unsigned long long)__popc(b));
    } else {
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        r[k] = contract<D>(Sq[k], Vq[k], s);
        if (CUBE) r[k] *= k == D ? rowp : row;
      }
    }
  } else {
    // perturbation U_new + 2 e w (the weights of the contraction carry the
    // half): the averages move by w, the increments and phi^{k+1} by 2 w
    Interp<D, T> B;
    T one[D], w2[D];  // CUBE: plain values of the velocities' perturbation first
#pragma unroll
    for (int i = 0; i < D; ++i) one[i] = T(1);
    interp_state<D, UNIT, CUBE>(wn, s, B, one);
    GpIn<D, Dl<T>> q;
    const T two = T(2), hf = T(0.5);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      w2[i] = (CUBE ? two * s.v : two) * B.vt[i];
      if (CUBE) B.vt[i] *= vs[i];
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
      q.vt[i] = Dl<T>(A.vt[i], B.vt[i]);
      q.dv[i] = Dl<T>(dvq[i], w2[i]);
      q.dpt[i] = Dl<T>(A.dpt[i], B.dpt[i]);
      q.dphit[i] = Dl<T>(A.dphit[i], B.dphit[i]);
      q.dmut[i] = Dl<T>(A.dmut[i], B.dmut[i]);
      q.dphin[i] = Dl<T>(mad(hf, dphig[i], A.dphit[i]), two * B.dphit[i]);
#pragma unroll
      for (int j = 0; j < D; ++j) q.dvt[i][j] = Dl<T>(A.dvt[i][j], B.dvt[i][j]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) q.hphit[k] = Dl<T>(A.hphit[k], B.hphit[k]);
    q.pt = Dl<T>(A.pt, B.pt);
    q.phit = Dl<T>(A.phit, B.phit);
    q.mut = Dl<T>(A.mut, B.mut);
    q.dphi = Dl<T>(dphiq, two * B.phit);
    q.phin = Dl<T>(mad(hf, dphiq, A.phit), two * B.phit);
    Dl<T> Sq[NF], Vq[NF][D];
    if constexpr (CUBE) gp_physics<D, HASF, true, T, Dl<T>>(kc, nG, CI_GG, inv_trG, CnWeH, q, fq, Sq, Vq, floored);
    else gp_physics<D, HASF, false, T, Dl<T>>(c, nG, CI_GG, inv_trG, CnWeH, q, fq, Sq, Vq, floored);
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      T Vk[D];
#pragma unroll
      for (int j = 0; j < D; ++j) Vk[j] = Vq[k][j].d;
      r[k] = contract<D>(Sq[k].d, Vk, s);
      if (CUBE) r[k] *= k == D ? rowp : row;
    }
  }
  if constexpr (MODE == 0 || MODE == 1) {
    // element-local output, slot (e, corner); k_gather_nodes sums the slots of
    // each node in a fixed order
    if (active) store_block<NF>(reinterpret_cast<T *>(out) + (e * NC + lc) * NF, r);
  } else if constexpr (MODE == 3) {
    // Lanes of one element may reach the same node: a hanging corner's parents
    // can be corners of the element or parents of its other hanging corner.
    // Warps that hold a hanging corner scatter one corner index at a time.
    if (__any_sync(FULL, cn < 0)) {
#pragma unroll 1
      for (int k = 0; k < NC; ++k) {
        if (active && lc == k) scatter<NF>(cn, hang, out, r);
        __syncwarp();
      }
    } else if (active) {
      scatter<NF>(cn, hang, out, r);
    }
  }
}

// ---------------------------------------------------------------- J.w in float, two Gauss points a lane
// As k_element MODE 1, with 2^(D-1) lanes per leaf: lane c holds the corners c
// and c + 2^(D-1) (the last axis' bit) and the two Gauss points of that pair.
// All arithmetic of the pair is packed, the last axis' stage stays in the lane.
// With one point a lane the issue slots bind (125 shuffles among the instructions
// of a Gauss point); packing halves the arithmetic's slots, the in-lane axis half of
// the shuffles: 37.5 M warp instructions on the level-6 octree, 7,028 flop a leaf.
// Bound by the latency of the gathers (54 % of the issue slots used, 128 registers,
// 14.6 warps an SM): 58 us, the whole apply with preparation and node gather 81 us
// and 457 us on 1,375,648 adaptive leaves; with one point a lane (schedule 5) 93 us.
template <int D>
struct Stage2 {
  F2 sg[D - 1];  // derivative factors of the lane axes, both halves
  F2 sh[D - 1];  // the same for UNIT data
  float sgl, shl;  // last axis: + for both halves (own - other, signed)
  F2 cS, cV[D - 1];
  float cVl;
};

__device__ __forceinline__ F2 shfl2(F2 x, int m) {
  return F2(__shfl_xor_sync(FULL, x.lo(), m), __shfl_xor_sync(FULL, x.hi(), m));
}
template <bool UNIT>
__device__ __forceinline__ F2 st_mix2(F2 u, F2 o) {
  constexpr float ca = 0.5f + 0.28867513459481288225f, cb = 0.5f - 0.28867513459481288225f;
  if (UNIT) return mad(F2(ca), u, F2(cb) * o);
  return mad(F2(float(TB)), o, u);
}
template <bool UNIT>
__device__ __forceinline__ void st_vd2(F2 u, int m, F2 &v, F2 &d) {
  const F2 o = shfl2(u, m);
  v = st_mix2<UNIT>(u, o);
  d = u - o;
}
template <bool UNIT>
__device__ __forceinline__ F2 st_v2(F2 u, int m) { return st_mix2<UNIT>(u, shfl2(u, m)); }
// the last axis, within the pair
template <bool UNIT>
__device__ __forceinline__ F2 in_v(F2 u) {
  return F2(st_mix<UNIT>(u.lo(), u.hi()), st_mix<UNIT>(u.hi(), u.lo()));
}
__device__ __forceinline__ F2 in_d(F2 u, float f) { return F2((u.hi() - u.lo()) * f); }

template <int D>
__device__ __forceinline__ F2 ip_v2(F2 u) {
  F2 a = st_v2<false>(u, 1);
  if (D == 3) a = st_v2<false>(a, 2);
  return in_v<false>(a) * F2(float(CAD<D>));
}

template <int D, bool UNIT = false>
__device__ __forceinline__ void ip_vg2(F2 u, const Stage2<D> &s, F2 &v, F2 *g) {
  const F2 *f = UNIT ? s.sh : s.sg;
  const float fl = UNIT ? s.shl : s.sgl;
  F2 A, Bx;
  st_vd2<UNIT>(u, 1, A, Bx);
  if (D == 2) {
    v = in_v<UNIT>(A);
    g[D - 1] = in_d(A, fl);
    g[0] = in_v<UNIT>(Bx) * f[0];
  } else {
    F2 AA, AB;
    st_vd2<UNIT>(A, 2, AA, AB);
    const F2 BA = st_v2<UNIT>(Bx, 2);
    v = in_v<UNIT>(AA);
    g[D - 1] = in_d(AA, fl);
    g[1] = in_v<UNIT>(AB) * f[D - 2];
    g[0] = in_v<UNIT>(BA) * f[0];
  }
  if (!UNIT) v *= F2(float(CAD<D>));
}

template <int D, bool UNIT = false>
__device__ __forceinline__ void ip_full2(F2 u, const Stage2<D> &s, F2 &v, F2 *g, F2 *hs) {
  const F2 *f = UNIT ? s.sh : s.sg;
  const float fl = UNIT ? s.shl : s.sgl;
  F2 A, Bx;
  st_vd2<UNIT>(u, 1, A, Bx);
  if (D == 2) {
    v = in_v<UNIT>(A);
    g[D - 1] = in_d(A, fl);
    g[0] = in_v<UNIT>(Bx) * f[0];
    hs[0] = in_d(Bx, fl) * f[0];
  } else {
    F2 AA, AB, BA, BB;
    st_vd2<UNIT>(A, 2, AA, AB);
    st_vd2<UNIT>(Bx, 2, BA, BB);
    v = in_v<UNIT>(AA);
    g[D - 1] = in_d(AA, fl);
    g[1] = in_v<UNIT>(AB) * f[D - 2];
    hs[2] = in_d(AB, fl) * f[D - 2];
    g[0] = in_v<UNIT>(BA) * f[0];
    hs[1] = in_d(BA, fl) * f[0];
    hs[0] = in_v<UNIT>(BB) * (f[0] * f[D - 2]);
  }
  if (!UNIT) v *= F2(float(CAD<D>));
}

template <int D>
__device__ __forceinline__ F2 contract2(F2 S, const F2 *V, const Stage2<D> &s) {
  const F2 tb{float(TB)}, ntb{float(-TB)};
  S *= s.cS;
  const float t = (V[D - 1].lo() + V[D - 1].hi()) * s.cVl;
  F2 X(fmaf(float(TB), S.hi(), S.lo()) - t, fmaf(float(TB), S.lo(), S.hi()) + t);
  F2 Y0 = in_v<false>(V[0] * s.cV[0]);
  if (D == 3) {
    const F2 Y1 = in_v<false>(V[1] * s.cV[D - 2]);
    X = (X + Y1) - shfl2(mad(ntb, X, Y1), 2);
    Y0 = mad(tb, shfl2(Y0, 2), Y0);
  }
  return (X + Y0) - shfl2(mad(ntb, X, Y0), 1);
}

template <int D>
__device__ __forceinline__ void interp_state2(const F2 *u, const Stage2<D> &s, Interp<D, F2> &I) {
#pragma unroll
  for (int i = 0; i < D; ++i) ip_vg2<D>(u[i], s, I.vt[i], I.dvt[i]);
  ip_vg2<D>(u[D], s, I.pt, I.dpt);
  ip_full2<D, true>(u[D + 1], s, I.phit, I.dphit, I.hphit);
  ip_vg2<D>(u[D + 2], s, I.mut, I.dmut);
}

template <int N>
__device__ __forceinline__ void gather_pair(int c0, int c1, const int32_t *__restrict__ hang,
                                            const float *__restrict__ src, F2 *out) {
  float a[N], b[N];
  gather<N>(c0, hang, src, a);
  gather<N>(c1, hang, src, b);
#pragma unroll
  for (int k = 0; k < N; ++k) out[k] = F2(a[k], b[k]);
}

// J.w of one leaf: u, d, wn hold the lane's two corners, r0, r1 their rows
template <int D>
__device__ __forceinline__ void pair_leaf(const KCoef<float> &c, const KPhys<F2> &cp, int lc, int l, const F2 *u,
                                          const F2 *d, const F2 *wn, float *r0, float *r1) {
  constexpr int NF = D + 3;
  Stage2<D> s;
#pragma unroll
  for (int a = 0; a < D - 1; ++a) {
    const bool neg = !((lc >> a) & 1);
    s.sg[a] = F2(flip_if(scale2(c.sg0[a], l), neg));
    s.sh[a] = F2(flip_if(scale2(c.sh0[a], l), neg));
  }
  s.sgl = scale2(c.sg0[D - 1], l);
  s.shl = scale2(c.sh0[D - 1], l);

  Interp<D, F2> A, B;
  interp_state2<D>(u, s, A);
  interp_state2<D>(wn, s, B);
  F2 dphi, dphig[D];
  ip_vg2<D, true>(d[D], s, dphi, dphig);
  GpIn<D, Dl<F2>> q;
  const F2 two(2.0f), hf(0.5f);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    q.vt[i] = Dl<F2>(A.vt[i], B.vt[i]);
    q.dv[i] = Dl<F2>(ip_v2<D>(d[i]), two * B.vt[i]);
    q.dpt[i] = Dl<F2>(A.dpt[i], B.dpt[i]);
    q.dphit[i] = Dl<F2>(A.dphit[i], B.dphit[i]);
    q.dmut[i] = Dl<F2>(A.dmut[i], B.dmut[i]);
    q.dphin[i] = Dl<F2>(mad(hf, dphig[i], A.dphit[i]), two * B.dphit[i]);
#pragma unroll
    for (int j = 0; j < D; ++j) q.dvt[i][j] = Dl<F2>(A.dvt[i][j], B.dvt[i][j]);
  }
#pragma unroll
  for (int k = 0; k < (D == 3 ? 3 : 1); ++k) q.hphit[k] = Dl<F2>(A.hphit[k], B.hphit[k]);
  q.pt = Dl<F2>(A.pt, B.pt);
  q.phit = Dl<F2>(A.phit, B.phit);
  q.mut = Dl<F2>(A.mut, B.mut);
  q.dphi = Dl<F2>(dphi, two * B.phit);
  q.phin = Dl<F2>(mad(hf, dphi, A.phit), two * B.phit);
  // the leaf's factors are made where they are used: kept from the start they
  // would sit in registers through the interpolation
  asm volatile("" : "+r"(l));
  F2 nG[D];
#pragma unroll
  for (int a = 0; a < D; ++a) nG[a] = F2(scale2(c.nG0[a], 2 * l));
  const F2 CI_GG(scale2(c.CIGG0, 4 * l)), inv_trG(scale2(c.inv_trG0, -2 * l));
  Dl<F2> Sq[NF], Vq[NF][D];
  B2 floored;
  gp_physics<D, false, false, F2, Dl<F2>>(cp, nG, CI_GG, inv_trG, cp.CnWe, q, static_cast<const F2 *>(nullptr), Sq, Vq,
                                   floored);
  asm volatile("" : "+r"(l));
#pragma unroll
  for (int a = 0; a < D - 1; ++a)
    s.cV[a] = F2(flip_if(scale2(c.cV0[a], (1 - D) * l - 1), !((lc >> a) & 1)));
  s.cVl = scale2(c.cV0[D - 1], (1 - D) * l - 1);
  s.cS = F2(scale2(c.cS0, -D * l - 1));
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    F2 Vk[D];
#pragma unroll
    for (int j = 0; j < D; ++j) Vk[j] = Vq[k][j].d;
    const F2 r = contract2<D>(Sq[k].d, Vk, s);
    r0[k] = r.lo();
    r1[k] = r.hi();
  }
}

// x rounded to T.  To float with integer instructions: the conversion
// instruction runs on the narrow FP64 pipe.  Round to nearest, ties to even, on
// the bits: the 29 discarded ones decide whether the kept ones go up by one
// (a carry moves into the exponent as it should).  Results that are not normal
// numbers go through the conversion instruction.
__device__ __forceinline__ float round_to(double x, float) {
  const unsigned hi = unsigned(__double2hiint(x)), lo = unsigned(__double2loint(x)), e = (hi >> 20) & 0x7ff;
  if (e - 897u < 253u) {
    unsigned b = ((hi << 3) | (lo >> 29)) - (896u << 23);  // exponent bias 1023 -> 127, modulo 2^32
    const unsigned rest = lo << 3;
    b += (rest > 0x80000000u || (rest == 0x80000000u && (b & 1u))) ? 1u : 0u;
    return __uint_as_float((b & 0x7fffffffu) | (hi & 0x80000000u));
  }
  if (((hi << 1) | lo) == 0) return __uint_as_float(hi);
  return float(x);
}
__device__ __forceinline__ double round_to(double x, double) { return x; }

// A node's prepared values straight from the states, rounded as k_prep rounds them
template <int D>
__device__ __forceinline__ void node_state(int64_t i, const double *__restrict__ Un, const double *__restrict__ Uo,
                                           float *u, float *d) {
  constexpr int NF = D + 3;
  double a[NF], b[NF];
  load_block<NF>(Un + i * NF, a);
  load_block<NF>(Uo + i * NF, b);
#pragma unroll
  for (int k = 0; k < NF; ++k) u[k] = 0.5f * round_to(a[k] + b[k], 0.0f);
#pragma unroll
  for (int k = 0; k < D; ++k) d[k] = round_to(a[k] - b[k], 0.0f);
  d[D] = round_to(a[D + 1] - b[D + 1], 0.0f);
}

// RAW: ut, dl are the states U_new, U_old themselves, on a mesh without hanging
// nodes (see launch_jacvec_states)
template <int D, int BS, int MINB, bool RAW>
__global__ void __launch_bounds__(BS, MINB) k_jv_pair(
    const int32_t *__restrict__ conn, const uint8_t *__restrict__ level, const int32_t *__restrict__ hang,
    int64_t n_elem, const void *__restrict__ ut, const void *__restrict__ dl, const float *__restrict__ w,
    float *__restrict__ out, const __grid_constant__ KCoef<float> c, const __grid_constant__ KPhys<F2> cp,
    int64_t wstride, int64_t ostride) {
  constexpr int NL = 1 << (D - 1), NC = 2 * NL, NF = D + 3, ND = D + 1;
  const int lc = threadIdx.x & (NL - 1);
  int64_t e = (int64_t(blockIdx.x) * BS + threadIdx.x) >> (D - 1);
  const bool active = e < n_elem;
  if (!active) e = n_elem - 1;
  const int c0 = conn[e * NC + lc], c1 = conn[e * NC + lc + NL], l = level[e];
  wait_previous(ut, dl, w, out);
  w += blockIdx.y * wstride;
  out += blockIdx.y * ostride;
  F2 u[NF], d[ND], wn[NF];
  if constexpr (RAW) {
    const double *Un = static_cast<const double *>(ut), *Uo = static_cast<const double *>(dl);
    float u0[NF], d0[ND], u1[NF], d1[ND];
    node_state<D>(c0, Un, Uo, u0, d0);
    node_state<D>(c1, Un, Uo, u1, d1);
#pragma unroll
    for (int k = 0; k < NF; ++k) u[k] = F2(u0[k], u1[k]);
#pragma unroll
    for (int k = 0; k < ND; ++k) d[k] = F2(d0[k], d1[k]);
  } else {
    gather_pair<NF>(c0, c1, hang, static_cast<const float *>(ut), u);
    gather_pair<ND>(c0, c1, hang, static_cast<const float *>(dl), d);
  }
  gather_pair<NF>(c0, c1, hang, w, wn);
  float r0[NF], r1[NF];
  pair_leaf<D>(c, cp, lc, l, u, d, wn, r0, r1);
  if (active) {
    store_block<NF>(out + (e * NC + lc) * NF, r0);
    store_block<NF>(out + (e * NC + lc + NL) * NF, r1);
  }
}

// ---------------------------------------------------------------- mass matrix
// Scalar corner value through the hanging constraint, field at offset k of
// node blocks of S values
template <int S>
__device__ __forceinline__ double gather1(int cn, const int32_t *__restrict__ hang, const double *__restrict__ u,
                                          int k) {
  if (cn >= 0) return __ldg(u + int64_t(cn) * S + k);
  const int4 p = reinterpret_cast<const int4 *>(hang)[-cn - 1];
  const double a = __ldg(u + int64_t(p.x) * S + k) + __ldg(u + int64_t(p.y) * S + k);
  if (p.z < 0) return 0.5 * a;
  return 0.25 * (a + (__ldg(u + int64_t(p.z) * S + k) + __ldg(u + int64_t(p.w) * S + k)));
}

// Conjugate gradients on the Q1 mass matrix (a scalar per node), preconditioned
// by its row sums, the whole iteration in one cooperative kernel.  With the
// 2-point Gauss rule the element matrix is the product over the axes of
// (h/6) [2 1; 1 2]: u + o/2 per axis and one factor W (2/3)^D, nine FP64
// instructions a lane.
//
// An iteration is three phases with a grid barrier after each: element products
// into the slots E, node sums with p.q, vector update with r.z and r.r.  Bound:
// the barriers, the sums and the first loads of each phase, about 12 us an
// iteration even on a mesh of 4,096 leaves; the FP64 pipe is worth about 8 of
// the 34 us on 77,932 leaves.  Whole call, in brackets with three launches an
// iteration: 77,932 leaves 2.45 ms (3.48), 4,096 uniform 1.13 (1.28), 262,144 2.57
// (3.44), 1,375,648 22.3 (25.6), 6,976,432 114 (110: there half the threads an SM
// could hold cost more than the launches do).
// Block shape, 77,932 / 4,096 leaves: 1,024 threads with two products in flight
// 2.48 / 1.13 ms, with four 2.52 / 1.31, 512 x 2 2.55 / 1.09, 512 x 3 2.95 /
// 1.03, 256 x 6 3.54 / 0.97: more blocks, more partial sums to add.
// Sums go through shared memory to one warp a scheduler: a shuffle sum in every
// warp is five FP64 instructions a warp of 64 cycles each.  Every block adds the
// blocks' partial sums itself, in the same order, so all of them take the same
// decisions.  What other blocks wrote is read past L1 (__ldcg).  Warps, not
// blocks, are dealt out over the nodes: the last round is spread over all SMs.
constexpr int kCgBlock = 1024, kCgPerSm = 1, kCgMaxGrid = 512, kCgUnroll = 2;
constexpr int kCgPolls = 1 << 25;  // about 20 s: a barrier that never fills ends as an error

struct CgArgs {
  const int32_t *conn, *hang, *gptr, *gent;
  const uint8_t *level;
  int64_t n_elem, n;
  double W0;  // of level 0, with the factor (2/3)^D
  double *E, *r, *x, *p, *q, *d, *z, *partial;
  unsigned *bar;
  CgState *s;
  int max_it;
  int polls;  // of a barrier, until it is given up
};

__device__ __forceinline__ double gather1_l2(int cn, const int32_t *__restrict__ hang, const double *u) {
  if (cn >= 0) return __ldcg(u + cn);
  const int4 p = reinterpret_cast<const int4 *>(hang)[-cn - 1];
  const double a = __ldcg(u + p.x) + __ldcg(u + p.y);
  if (p.z < 0) return 0.5 * a;
  return 0.25 * (a + (__ldcg(u + p.z) + __ldcg(u + p.w)));
}

// all blocks have arrived for the epoch-th time; false: given up
__device__ __forceinline__ bool cg_barrier(unsigned *bar, unsigned &epoch, int limit, int *given_up) {
  ++epoch;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned want = epoch * gridDim.x;
    unsigned have;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(have) : "l"(bar) : "memory");
    } while (have < want && --limit > 0);
    *given_up = have < want;
    __threadfence();
  }
  __syncthreads();
  return !*given_up;
}

// tot[v] = sum over all threads of the grid of acc[v], with a grid barrier
template <int N>
__device__ __forceinline__ bool cg_sum(const double (&acc)[N], double *tot, double *partial, unsigned *bar,
                                       unsigned &epoch, int limit, int *given_up) {
  __shared__ double all[N][kCgBlock], four[N][4];
  const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31;
#pragma unroll
  for (int v = 0; v < N; ++v) all[v][threadIdx.x] = acc[v];
  __syncthreads();
  if (wid < 4 * N) {
    const double *a = all[wid >> 2] + (wid & 3) * (kCgBlock / 4);
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < kCgBlock / 128; ++k) t += a[k * 32 + ln];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(FULL, t, o);
    if (ln == 0) four[wid >> 2][wid & 3] = t;
  }
  __syncthreads();
  if (threadIdx.x < N) {
    const double *f = four[threadIdx.x];
    __stcg(partial + threadIdx.x * gridDim.x + blockIdx.x, (f[0] + f[1]) + (f[2] + f[3]));
  }
  if (!cg_barrier(bar, epoch, limit, given_up)) return false;
  if (wid < N) {
    double t = 0.0;
    for (unsigned b = ln; b < gridDim.x; b += 32) t += __ldcg(partial + wid * gridDim.x + b);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(FULL, t, o);
    if (ln == 0) tot[wid] = t;
  }
  __syncthreads();
  return true;
}

__device__ __forceinline__ double cg_node_sum(const CgArgs &g, int64_t i) {
  double sum = 0.0;
  const int e1 = g.gptr[i + 1];
  constexpr int G = 8;  // independent loads, then the sum in list order
  for (int e = g.gptr[i]; e < e1; e += G) {
    uint32_t ent[G];
    double v[G];
#pragma unroll
    for (int k = 0; k < G; ++k) ent[k] = e + k < e1 ? uint32_t(g.gent[e + k]) : 0xffffffffu;
#pragma unroll
    for (int k = 0; k < G; ++k) v[k] = ent[k] != 0xffffffffu ? __ldcg(g.E + (ent[k] & 0x3fffffffu)) : 0.0;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const uint32_t code = ent[k] >> 30;  // 3: past the end, v = 0
      sum = fma(code == 0 ? 1.0 : (code == 1 ? 0.5 : 0.25), v[k], sum);
    }
  }
  return sum;
}

// E: the right-hand side's element parts; x = M^-1 (their node sums)
template <int D>
__global__ void __launch_bounds__(kCgBlock, kCgPerSm) k_cg(const __grid_constant__ CgArgs g) {
  constexpr int NC = 1 << D, U = kCgUnroll;
  const int lc = threadIdx.x & (NC - 1);
  const int64_t step = int64_t(gridDim.x) * kCgBlock;
  const int64_t t0 = (int64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  const int64_t slots = g.n_elem << D;
  __shared__ int given_up;
  __shared__ double tot[2], tpq[1], ash;
  unsigned epoch = 0;
  int err = 0, it = 0;
  for (int64_t i = t0; i < g.n; i += step) g.r[i] = cg_node_sum(g, i);
  if (!cg_barrier(g.bar, epoch, g.polls, &given_up)) { err = 2; goto end; }
  for (int64_t t = t0; t < slots; t += step)
    g.E[t] = scale2(g.W0, -D * int(g.level[t >> D])) * (D == 2 ? 2.25 : 3.375);  // the product with ones
  if (!cg_barrier(g.bar, epoch, g.polls, &given_up)) { err = 2; goto end; }
  {
    double acc[2] = {0.0, 0.0};
    for (int64_t i = t0; i < g.n; i += step) {
      const double m = cg_node_sum(g, i), di = m > 0.0 ? 1.0 / m : 0.0, ri = g.r[i], zi = di * ri;
      g.d[i] = di;
      g.z[i] = zi;
      g.x[i] = 0.0;
      g.p[i] = 0.0;
      acc[0] = fma(ri, zi, acc[0]);
      acc[1] = fma(ri, ri, acc[1]);
    }
    if (!cg_sum<2>(acc, tot, g.partial, g.bar, epoch, g.polls, &given_up)) { err = 2; goto end; }
  }
  {
    double rz = tot[0], rr = tot[1], beta = 0.0;
    const double stop = 1e-26 * fmax(rr, 1e-300);
    for (; it < g.max_it && rr > stop && rz > 0.0; ++it) {
      for (int64_t b = t0; b - (threadIdx.x & 31) < slots; b += U * step) {  // whole warps: shuffles
        int cn[U], l[U];
        double u[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int64_t t = b + k * step, e = (t < slots ? t : slots - NC + lc) >> D;
          cn[k] = g.conn[e * NC + lc];
          l[k] = g.level[e];
        }
#pragma unroll
        for (int k = 0; k < U; ++k) u[k] = fma(beta, gather1_l2(cn[k], g.hang, g.p), gather1_l2(cn[k], g.hang, g.z));
#pragma unroll
        for (int k = 0; k < U; ++k) {
#pragma unroll
          for (int a = 0; a < D; ++a) u[k] = fma(0.5, __shfl_xor_sync(FULL, u[k], 1 << a), u[k]);
          const int64_t t = b + k * step;
          if (t < slots) g.E[t] = scale2(g.W0, -D * l[k]) * u[k];
        }
      }
      if (!cg_barrier(g.bar, epoch, g.polls, &given_up)) { err = 2; break; }
      double pq[1] = {0.0}, acc[2] = {0.0, 0.0};
      for (int64_t i = t0; i < g.n; i += step) {
        const double sum = cg_node_sum(g, i), pi = fma(beta, g.p[i], g.z[i]);
        g.q[i] = sum;
        g.p[i] = pi;
        pq[0] = fma(pi, sum, pq[0]);
      }
      if (!cg_sum<1>(pq, tpq, g.partial + 2 * gridDim.x, g.bar, epoch, g.polls, &given_up)) { err = 2; break; }
      if (!(tpq[0] > 0.0)) { err = 1; break; }
      if (threadIdx.x == 0) ash = rz / tpq[0];  // one division a block: ten instructions of the FP64 pipe
      __syncthreads();
      const double a = ash;
      for (int64_t i = t0; i < g.n; i += step) {
        g.x[i] = fma(a, g.p[i], g.x[i]);
        const double ri = fma(-a, g.q[i], g.r[i]), zi = g.d[i] * ri;
        g.r[i] = ri;
        g.z[i] = zi;
        acc[0] = fma(ri, zi, acc[0]);
        acc[1] = fma(ri, ri, acc[1]);
      }
      if (!cg_sum<2>(acc, tot, g.partial, g.bar, epoch, g.polls, &given_up)) { err = 2; break; }
      if (threadIdx.x == 0) ash = tot[0] / rz;
      __syncthreads();
      beta = ash;
      rz = tot[0];
      rr = tot[1];
      __syncthreads();  // tot and ash are read before the next sums
    }
  }
end:
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    g.s->err = err;
    g.s->its = it;
  }
}

// Element-local part of the chemical-potential row at U_new = U_old = U:
// (N, psi'(phi) - mu) + Cn^2 (grad N, grad phi)
template <int D>
__global__ void __launch_bounds__(256) k_mu_row(const int32_t *__restrict__ conn, const uint8_t *__restrict__ level,
                                                const int32_t *__restrict__ hang, int64_t n_elem,
                                                const double *__restrict__ U, KCoef<double> c,
                                                double *__restrict__ E) {
  constexpr int NC = 1 << D, NF = D + 3;
  const int lc = threadIdx.x & (NC - 1);
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  int64_t e = t >> D;
  const bool active = e < n_elem;
  if (!active) e = n_elem - 1;
  const int cn = conn[e * NC + lc], l = level[e];
  Stage<D, double> s;
  s.v = CAD<D>;
  s.cS = scale2(c.cS0, -D * l);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const bool neg = !((lc >> a) & 1);
    s.sg[a] = flip_if(scale2(c.sg0[a], l), neg);
    s.cV[a] = flip_if(scale2(c.cV0[a], (1 - D) * l), neg);
  }
  double phi, g[D];
  ip_vg<D>(gather1<NF>(cn, hang, U, D + 1), s, phi, g);
  const double mu = ip_v<D>(gather1<NF>(cn, hang, U, D + 2)) * CAD<D>;
#pragma unroll
  for (int a = 0; a < D; ++a) g[a] *= c.Cn2;
  const double r = contract<D>(phi * fma(phi, phi, -1.0) - mu, g, s);
  if (active) E[t] = r;
}

// ---------------------------------------------------------------- node kernels
// v~ = (U_new + U_old)/2 for all fields; increments of v and phi, formed in
// double and rounded once (the half is taken after the rounding, exactly).  A
// thread per value.  FP64 pipe: two sums a value; with a thread per node (loads
// 48 B apart), products by 1/2 and ten conversions the pipe was 78 % busy.
// 274,625 nodes to float: 19.7 -> 12.1 us.
template <int D, typename T>
__global__ void __launch_bounds__(256) k_prep(const double *__restrict__ Un, const double *__restrict__ Uo, int64_t n,
                                              T *__restrict__ ut, T *__restrict__ dl) {
  constexpr int NF = D + 3, ND = D + 1;
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  wait_previous(Un, Uo, ut, dl);
  if (t >= n * NF) return;
  const unsigned i = unsigned(t / NF);
  const int k = int(t - int64_t(i) * NF);
  const double a = Un[t], b = Uo[t];
  ut[t] = T(0.5) * round_to(a + b, T());
  if (k < D || k == D + 1) dl[int64_t(i) * ND + (k < D ? k : D)] = round_to(a - b, T());
}

// y[i] = sum over the slots of node i of weight * E[slot] (fixed order), then
// the constrained rows (wall velocities, the pinned pressure): y = w for J.w,
// y = w - bc for the residual (kResidual: w = U_new, bc nullable).  kDefect:
// y = bc - J.w, the defect of bc.  A thread per pair
// of values (3D) or per value (2D) of a node, the threads of a node side by
// side: a warp's load then touches a third (a fifth) of the slots, and as many
// fewer cache lines, than with a thread per node.  Slots are fetched eight at a
// time (independent loads), then added in list order.
enum GatherOp { kApply, kResidual, kDefect };
template <int D, typename T, GatherOp OP>
__global__ void __launch_bounds__(256) k_gather_nodes(const int32_t *__restrict__ gptr,
                                                      const int32_t *__restrict__ gent,
                                                      const uint8_t *__restrict__ nflag, int64_t n_nodes,
                                                      const T *__restrict__ E, const T *w, const T *bc, T *y,
                                                      uint32_t fmask, int64_t estride) {
  constexpr int NF = D + 3, G = 8, L = NF % 2 == 0 ? 2 : 1, NP = NF / L;
  const int64_t t0 = blockIdx.x * int64_t(blockDim.x) + threadIdx.x, t = min(t0, n_nodes * NP - 1);
  const unsigned i = unsigned(t / NP);
  const int k0 = int(t - int64_t(i) * NP) * L;
  T acc[L];
#pragma unroll
  for (int k = 0; k < L; ++k) acc[k] = T(0);
  const int p0 = gptr[i], p1 = gptr[i + 1];
  const unsigned fl = nflag[i];
  uint32_t ent[G];
#pragma unroll
  for (int g = 0; g < G; ++g) ent[g] = p0 + g < p1 ? uint32_t(gent[p0 + g]) : 0xffffffffu;
  wait_previous(E, w, bc, y);
  if (t0 != t) return;
  E += blockIdx.y * estride;  // gridDim.y directions, one vector after another
  w += blockIdx.y * n_nodes * NF;
  y += blockIdx.y * n_nodes * NF;
  for (int pb = p0; pb < p1; pb += G) {
    if (pb != p0)
#pragma unroll
      for (int g = 0; g < G; ++g) ent[g] = pb + g < p1 ? uint32_t(gent[pb + g]) : 0xffffffffu;
    T v[G][L];
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (ent[g] != 0xffffffffu) load_block<L>(E + int64_t(ent[g] & 0x3fffffffu) * NF + k0, v[g]);
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (ent[g] != 0xffffffffu) {
        const uint32_t code = ent[g] >> 30;
        const T wt = code == 0 ? T(1) : (code == 1 ? T(0.5) : T(0.25));
#pragma unroll
        for (int k = 0; k < L; ++k) acc[k] = fma(wt, v[g][k], acc[k]);
      }
  }
#pragma unroll
  for (int k = 0; k < L; ++k) {
    const int q = k0 + k;
    if (((fl & 1) && q < D) || ((fl & 2) && q == D))
      acc[k] = w[int64_t(i) * NF + q] - (OP == kResidual && bc ? bc[int64_t(i) * NF + q] : T(0));
    else if (OP != kResidual && !((fmask >> q) & 1u)) acc[k] = w[int64_t(i) * NF + q];
    if (OP == kDefect) acc[k] = bc[int64_t(i) * NF + q] - acc[k];
  }
  store_block<L>(y + int64_t(i) * NF + k0, acc);
}

// One damped nodal block-Jacobi sweep on top of the element part of J.x in E:
// x += B (b - J.x), the node sums as in k_gather_nodes.  Eight lanes per node,
// lane q its component q: the slots, the rows of B and the vectors are read in
// pieces of a node's length, and the product needs six shuffles.  (A gather, then
// a sweep with a thread per node and its 144 B block, took a launch and a pass
// over y more.)
template <int D, typename T>
__global__ void __launch_bounds__(256) k_gather_smooth(const int32_t *__restrict__ gptr,
                                                       const int32_t *__restrict__ gent,
                                                       const uint8_t *__restrict__ nflag, int64_t n_nodes,
                                                       const T *__restrict__ E, const T *__restrict__ b,
                                                       const T *__restrict__ B, T *__restrict__ x, uint32_t fmask) {
  constexpr int NF = D + 3, G = 8;
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const int q = threadIdx.x & 7;
  const bool on = (t >> 3) < n_nodes && q < NF;
  const int64_t i = on ? t >> 3 : 0, at = i * NF + (on ? q : 0);
  T row[NF];
#pragma unroll
  for (int c = 0; c < NF; ++c) row[c] = B[at * NF + c];
  const unsigned fl = nflag[i];
  const int p0 = gptr[i], p1 = gptr[i + 1], k = int(at - i * NF);
  uint32_t ent[G];
#pragma unroll
  for (int g = 0; g < G; ++g) ent[g] = p0 + g < p1 ? uint32_t(gent[p0 + g]) : 0xffffffffu;
  wait_previous(E, b, x);
  const T xi = x[at], bi = b[at];
  T acc = T(0);
  for (int pb = p0; pb < p1; pb += G) {
    if (pb != p0)
#pragma unroll
      for (int g = 0; g < G; ++g) ent[g] = pb + g < p1 ? uint32_t(gent[pb + g]) : 0xffffffffu;
    T v[G];
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (ent[g] != 0xffffffffu) v[g] = E[int64_t(ent[g] & 0x3fffffffu) * NF + k];
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (ent[g] != 0xffffffffu) {
        const uint32_t code = ent[g] >> 30;
        acc = fma(code == 0 ? T(1) : (code == 1 ? T(0.5) : T(0.25)), v[g], acc);
      }
  }
  if (((fl & 1) && k < D) || ((fl & 2) && k == D) || !((fmask >> k) & 1u)) acc = xi;
  const T r = bi - acc;
  T s = T(0);
#pragma unroll
  for (int c = 0; c < NF; ++c) s = fma(row[c], __shfl_sync(FULL, r, c, 8), s);
  if (on) x[at] = xi + s;
}

// J.w by colour scatter: the constrained rows and the rows of fields outside
// fmask become y = w (as k_gather_nodes does after its sums)
template <int D, typename T>
__global__ void k_fix_rows(const uint8_t *__restrict__ nflag, int64_t n_nodes, const T *__restrict__ w,
                           T *__restrict__ y, uint32_t fmask) {
  constexpr int NF = D + 3;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n_nodes; i += int64_t(gridDim.x) * blockDim.x) {
    const uint8_t fl = nflag[i];
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const bool keep = ((fmask >> k) & 1u) && !((fl & 1) && k < D) && !((fl & 2) && k == D);
      if (!keep) y[i * NF + k] = w[i * NF + k];
    }
  }
}

// ---------------------------------------------------------------- diagnostics
// per block: energy, integral of phi, volume with phi < 0 (2^D Gauss rule).
// Bound by the FP64 pipe (16 cycles a warp instruction, 84 % busy).  A fixed
// grid strides over the leaves and each thread keeps its sums, so the block
// reduction runs once per thread and not once per leaf; quotients are exact
// scalings of host constants, the factors of the interpolation sit in the
// constants; comparisons and conversions of integers are done on the bits, and
// the volume is counted in cells of the finest level.  FP64 instructions a
// leaf's lane: 58 with the comparisons in double, 39 now.  381,256 leaves, the
// whole call: 0.33 ms; 0.84 with six divisions a lane and the sums on the host.
struct EnergyCoef {
  double kv;                 // CA^(2D) / 2: kinetic energy from unscaled velocities
  double kpsi, kg[3];        // Cn/(We 4 Cn^2) and Cn/(2 We) times the squared derivative factors
  double z0, zg[3];          // rho potential: z0 + sum zg_a (integer coordinate a)
  double alpha, beta, W0;
  double cell;               // volume weight of a Gauss point of the finest level
  int axes;                  // bit a: zg[a] is not 0
};

// an unsigned integer as a double, exactly: 2^52 + a has a in its low bits
__device__ __forceinline__ double uint_to_double(uint32_t a) {
  return __hiloint2double(0x43300000, int(a)) - 4503599627370496.0;
}

template <int D>
__global__ void __launch_bounds__(256) k_energy(
    const int32_t *__restrict__ conn, const uint8_t *__restrict__ level,
    const uint32_t *__restrict__ anchor, const int32_t *__restrict__ hang, int64_t n_elem, int max_level,
    const double *__restrict__ U, EnergyCoef c, double *__restrict__ partial) {
  constexpr int NC = 1 << D, NF = D + 3;
  const int lc = threadIdx.x & (NC - 1);
  double E = 0.0, M = 0.0;
  long long light = 0;
  const int64_t n = (n_elem + 256 / NC - 1) / (256 / NC);
  wait_previous(U, partial);
  for (int64_t blk = blockIdx.x; blk < n; blk += gridDim.x) {  // the same trips for all lanes: shuffles below
    int64_t e = blk * (256 / NC) + (threadIdx.x >> D);
    const bool active = e < n_elem;
    if (!active) e = n_elem - 1;
    const int cn = conn[e * NC + lc], l = level[e];
    double u[NF];
    gather<NF>(cn, hang, U, u);
    const double v0 = ip_v<D>(u[0]), v1 = ip_v<D>(u[1]);
    double v2 = fma(v1, v1, v0 * v0);
    if (D == 3) {
      const double vz = ip_v<D>(u[D - 1]);
      v2 = fma(vz, vz, v2);
    }
    Stage<D, double> s;
    s.v = CAD<D>;
#pragma unroll
    for (int a = 0; a < D; ++a) s.sg[a] = 1.0;  // folded away: raw derivatives, squared below
    double phi, g[D], t = 0.0;
    ip_vg<D>(u[D + 1], s, phi, g);
#pragma unroll
    for (int a = 0; a < D; ++a) t = fma(g[a] * g[a], scale2(c.kg[a], 2 * l), t);
    // phi*: bits of |phi| compare like the numbers; NaN stays NaN
    const int sg = __double2hiint(phi), hi = sg & 0x7fffffff;
    const double phis = hi < 0x3ff00000 || hi > 0x7ff00000 ? phi : flip_if(1.0, sg < 0);
    const double rho = fma(c.alpha, phis, c.beta);
    double z = c.z0;
#pragma unroll
    for (int a = 0; a < D; ++a)
      if ((c.axes >> a) & 1) {  // uniform: gravity along an axis needs one of them
        const double xi = scale2(((lc >> a) & 1) ? CA : 1.0 - CA, max_level - l);
        z = fma(c.zg[a], xi + uint_to_double(anchor[e * D + a]), z);
      }
    const double w = fma(phi, phi, -1.0);
    t = fma(c.kpsi * w, w, t);
    t = fma(rho, fma(c.kv, v2, z), t);
    if (active) {
      const double W = scale2(c.W0, -D * l);
      E = fma(W, t, E);
      M = fma(W, phi, M);
      // phi < 0 (not -0, not NaN)
      const bool neg = sg < 0 && hi <= 0x7ff00000 && (hi | __double2loint(phi)) != 0 &&
                       !(hi == 0x7ff00000 && __double2loint(phi) != 0);
      if (neg) light += 1ll << (D * (max_level - l));
    }
  }
  double Lt = c.cell * double(light);
  // deterministic block reduction
  __shared__ double sh[3][256 / 32];
  for (int o = 16; o > 0; o >>= 1) {
    E += __shfl_down_sync(FULL, E, o);
    M += __shfl_down_sync(FULL, M, o);
    Lt += __shfl_down_sync(FULL, Lt, o);
  }
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { sh[0][wid] = E; sh[1][wid] = M; sh[2][wid] = Lt; }
  __syncthreads();
  if (threadIdx.x < 3) {
    double a = 0;
    for (int k = 0; k < 256 / 32; ++k) a += sh[threadIdx.x][k];
    partial[blockIdx.x * 3 + threadIdx.x] = a;
  }
}

// out[k] = sum over the blocks b of partial[b * 3 + k], fixed order: a warp per
// sum, lanes over the blocks, a fixed shuffle tree
__global__ void k_energy_sum(const double *__restrict__ partial, int nb, double *__restrict__ out) {
  const int k = threadIdx.x >> 5, ln = threadIdx.x & 31;
  wait_previous(partial, out);
  double s = 0.0;
  for (int b = ln; b < nb; b += 32) s += partial[b * 3 + k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(FULL, s, o);
  if (ln == 0) out[k] = s;
}

}  // namespace

// ---------------------------------------------------------------- launchers
PhysCoef make_coef(const chns_params &p, const double *lo, const double *hi) {
  PhysCoef c;
  c.dt = p.dt;
  c.inv_dt = 1.0 / p.dt;
  c.four_dt2 = 4.0 / (p.dt * p.dt);
  c.alpha = 0.5 * (1.0 - p.rho_ratio);
  c.beta = 0.5 * (1.0 + p.rho_ratio);
  c.gamma = 0.5 * (1.0 - p.eta_ratio);
  c.xi = 0.5 * (1.0 + p.eta_ratio);
  c.jc = 0.5 * (p.rho_ratio - 1.0);
  c.inv_Pe = 1.0 / p.Pe;
  c.inv_We = 1.0 / p.We;
  c.inv_Re = 1.0 / p.Re;
  c.inv_Fr = 1.0 / p.Fr;
  c.CnWe = p.Cn / p.We;
  c.inv_PeCn = 1.0 / (p.Pe * p.Cn);
  c.Cn2 = p.Cn * p.Cn;
  c.C_I = p.C_I;
  for (int a = 0; a < 3; ++a) {
    c.g[a] = p.gravity[a];
    c.ext[a] = hi[a] - lo[a];
    c.lo[a] = lo[a];
  }
  c.fmask = 0xffu;
  return c;
}

namespace {
constexpr int kBlock = 256;
inline unsigned grid_for(int64_t threads) { return (unsigned)((threads + kBlock - 1) / kBlock); }
// element kernels: 128 threads (16 leaves in 3D), 6 blocks per SM (measured
// slightly ahead of 256 x 3 on the uniform and the adaptive meshes)
constexpr int kElemBlock = 128;
// FP64 element kernels: 3 blocks of 128 threads per SM (up to 170 registers)
constexpr int kFp64MinBlocks = 3;
inline unsigned grid_elem(int64_t threads) { return (unsigned)((threads + kElemBlock - 1) / kElemBlock); }
inline unsigned grid_nodes(int64_t n) {
  int64_t b = (n + kBlock - 1) / kBlock;
  return (unsigned)std::min<int64_t>(std::max<int64_t>(b, 1), 152 * 16);
}
}  // namespace

namespace {
template <int D>
unsigned grid_gather(int64_t n_nodes) { return grid_for(n_nodes * (D == 3 ? 3 : 5)); }
}  // namespace

template <typename T>
void launch_prep(const chns_mesh *m, const double *Un, const double *Uo, T *ut, T *dl, cudaStream_t st) {
  const unsigned g = grid_for(m->n_nodes * m->nf);
  if (m->dim == 2) launch_next(k_prep<2, T>, g, kBlock, st, Un, Uo, m->n_nodes, ut, dl);
  else launch_next(k_prep<3, T>, g, kBlock, st, Un, Uo, m->n_nodes, ut, dl);
  note_launches(1);
}
template void launch_prep<float>(const chns_mesh *, const double *, const double *, float *, float *, cudaStream_t);
template void launch_prep<double>(const chns_mesh *, const double *, const double *, double *, double *, cudaStream_t);

// Residual: all elements in one launch into the element-local buffer E, then
// the node gather with the constrained rows, as J.w.  One launch per element
// colour with in-place adds read and wrote every node once per colour, needed
// the output zeroed first and left eight partly filled last waves; E costs 96
// B per corner of L2 / HBM traffic instead: the gather takes 35 of 1,382 us on
// 262,144 leaves.
// U_new and U_old are averaged in the element kernel (10 FP64 instructions a
// lane) rather than by a node pass before it: a state is evaluated once.
template <int D, bool HASF>
static void residual_elemlocal(const chns_mesh *m, const PhysCoef &pc, const KCoef<double> &c, const double *Un, const double *Uo,
                               const double *f, const double *bc, double *E, double *F, cudaStream_t st) {
  if (D == 3 && !m->coef64 && is_cube(c))
    launch_next(k_element<D, double, 0, HASF, double, kElemBlock, kFp64MinBlocks, D == 3>, grid_elem(m->n_elem << D),
                kElemBlock, st, m->conn, m->level, m->hang, 0, m->n_elem, Un, Uo, nullptr, f, E, kcube(pc, c, true),
                nullptr, m->elem_inst, 0, 0, nullptr);
  else
    launch_next(k_element<D, double, 0, HASF, double, kElemBlock, kFp64MinBlocks>, grid_elem(m->n_elem << D),
                kElemBlock, st, m->conn, m->level, m->hang, 0, m->n_elem, Un, Uo, nullptr, f, E, c,
                reinterpret_cast<const KCoef<double> *>(m->coef64), m->elem_inst, 0, 0, nullptr);
  launch_next(k_gather_nodes<D, double, kResidual>, grid_gather<D>(m->n_nodes), kBlock, st, m->gptr, m->gent, m->nflag,
              m->n_nodes, E, Un, bc, F, 0xffu, 0);
  note_launches(2);
}

void launch_residual(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo, const double *f,
                     const double *bc, double *E, double *F, cudaStream_t st) {
  const KCoef<double> c = kcoef<double>(pc, m->dim);
  if (m->dim == 2) {
    if (f) residual_elemlocal<2, true>(m, pc, c, Un, Uo, f, bc, E, F, st);
    else residual_elemlocal<2, false>(m, pc, c, Un, Uo, f, bc, E, F, st);
  } else {
    if (f) residual_elemlocal<3, true>(m, pc, c, Un, Uo, f, bc, E, F, st);
    else residual_elemlocal<3, false>(m, pc, c, Un, Uo, f, bc, E, F, st);
  }
}

// J.w schedules (chosen per mesh by the autotuner, FP32 only; FP64 always
// uses the element-local buffer with 128-thread blocks, 3 per SM):
//   0-3: two Gauss points per lane (k_jv_pair), all elements at once into the
//      element-local buffer E (n_elem * 2^dim * nf values), then the node
//      gather with the constrained rows; (threads, blocks per SM) = (64, 8),
//      (128, 3), (64, 6), (128, 4).  0 is the default: 16 warps an SM hide the
//      scattered loads of an adaptive mesh better than 12 (455 against 491 us on
//      1,375,648 leaves, in spite of 124 bytes of spills) and cost 1 % on a
//      uniform one (81.0 against 80.4 us, 262,144 leaves)
//   4: element colours one launch after another, each element adding its
//      contributions into y (disjoint nodes within a colour; no E buffer),
//      then the constrained rows
//   5, 6: as 0 with one Gauss point per lane, 128 threads, 5 and 6 per SM; 5 is
//      what a batch's union mesh uses (each element has its own coefficients,
//      which as pairs would take twice the registers)
template <int D, typename T, int BS, int MINB>
static void elem_local(const chns_mesh *m, const PhysCoef &pc, const KCoef<T> &c, const KCoef<T> *tab, const T *ut, const T *dl,
                       const T *w, T *E, cudaStream_t st, int nv) {
  constexpr int NF = D + 3;
  const int64_t threads = m->n_elem << D;
  const dim3 ge((unsigned)((threads + BS - 1) / BS), (unsigned)nv);
  note_launches(1);
  if constexpr (sizeof(T) == 8 && D == 3)
    if (!tab && is_cube(c)) {
      launch_next(k_element<D, T, 1, false, T, BS, MINB, true>, ge, BS, st, m->conn, m->level, m->hang, 0, m->n_elem, ut,
                  dl, w, nullptr, E, kcube(pc, c, false), tab, m->elem_inst, m->n_nodes * NF, threads * NF, nullptr);
      return;
    }
  launch_next(k_element<D, T, 1, false, T, BS, MINB>, ge, BS, st, m->conn, m->level, m->hang, 0, m->n_elem, ut, dl, w,
              nullptr, E, c, tab, m->elem_inst, m->n_nodes * NF, threads * NF, nullptr);
}

static F2 host_pair(float a) {
  uint32_t b;
  std::memcpy(&b, &a, 4);
  F2 p;
  p.v = (uint64_t(b) << 32) | b;
  return p;
}
static KPhys<F2> pair_coef(const KPhys<float> &c) {
  KPhys<F2> p;
  static_assert(sizeof(KPhys<F2>) == 2 * sizeof(KPhys<float>), "plain arrays of constants");
  const float *x = reinterpret_cast<const float *>(&c);
  F2 *y = reinterpret_cast<F2 *>(&p);
  for (size_t k = 0; k < sizeof(KPhys<float>) / 4; ++k) y[k] = host_pair(x[k]);
  return p;
}

template <int D, int BS, int MINB>
static void elem_pair(const chns_mesh *m, const KCoef<float> &c, const float *ut, const float *dl, const float *w,
                      float *E, cudaStream_t st, int nv) {
  constexpr int NF = D + 3;
  const int64_t threads = m->n_elem << (D - 1);
  const dim3 ge((unsigned)((threads + BS - 1) / BS), (unsigned)nv);
  launch_next(k_jv_pair<D, BS, MINB, false>, ge, BS, st, m->conn, m->level, m->hang, m->n_elem, ut, dl, w, E, c, pair_coef(c),
              m->n_nodes * NF, (m->n_elem << D) * NF);
  note_launches(1);
}

template <int D, typename T>
static void jv_colours(const chns_mesh *m, const KCoef<T> &c, const KCoef<T> *tab, const T *ut, const T *dl,
                       const T *w, T *y, uint32_t fmask, cudaStream_t st) {
  cudaMemsetAsync(y, 0, sizeof(T) * m->n_nodes * (D + 3), st);
  for (int col = 0; col < m->n_colours; ++col) {
    const int64_t b = m->colour_start[col], e = m->colour_start[col + 1];
    if (e <= b) continue;
    k_element<D, T, 3, false, T><<<grid_elem((e - b) << D), kElemBlock, 0, st>>>(
        m->conn, m->level, m->hang, b, e, ut, dl, w, nullptr, y, c, tab, m->elem_inst, 0, 0, m->elem_perm);
    note_launches(1);
  }
  k_fix_rows<D, T><<<grid_nodes(m->n_nodes), kBlock, 0, st>>>(m->nflag, m->n_nodes, w, y, fmask);
  note_launches(1);
}

// element part of J.w into E (any schedule but the colours)
template <int D, typename T>
static void elem_dispatch(const chns_mesh *m, const PhysCoef &pc, int variant, const KCoef<T> &c, const KCoef<T> *tab, const T *ut,
                          const T *dl, const T *w, T *E, cudaStream_t st, int nv) {
  if constexpr (sizeof(T) == 8) {
    // FP64: bound by the narrow FP64 pipe, so occupancy matters less than
    // the register spills a 6-blocks-per-SM budget causes
    elem_local<D, T, 128, kFp64MinBlocks>(m, pc, c, tab, ut, dl, w, E, st, nv);
  } else {
    if (!tab) switch (variant) {
        case 0: elem_pair<D, 64, 8>(m, c, ut, dl, w, E, st, nv); return;
        case 1: elem_pair<D, 128, 3>(m, c, ut, dl, w, E, st, nv); return;
        case 2: elem_pair<D, 64, 6>(m, c, ut, dl, w, E, st, nv); return;
        case 3: elem_pair<D, 128, 4>(m, c, ut, dl, w, E, st, nv); return;
        default: break;
      }
    if (variant == 6) elem_local<D, T, 128, 6>(m, pc, c, tab, ut, dl, w, E, st, nv);
    else elem_local<D, T, 128, 5>(m, pc, c, tab, ut, dl, w, E, st, nv);  // 5, and the pair schedules on a union mesh
  }
}

template <int D, typename T>
static void jv_dispatch(const chns_mesh *m, const PhysCoef &pc, int variant, const KCoef<T> &c, const KCoef<T> *tab, const T *ut,
                        const T *dl, const T *w, T *E, T *y, uint32_t fmask, cudaStream_t st, int nv) {
  if constexpr (sizeof(T) == 4) {
    if (variant == 4 && nv == 1) {
      jv_colours<D, T>(m, c, tab, ut, dl, w, y, fmask, st);
      return;
    }
    if (variant == 4) variant = 0;  // the colour schedule takes one direction at a time
  }
  elem_dispatch<D, T>(m, pc, variant, c, tab, ut, dl, w, E, st, nv);
  const dim3 gn(grid_gather<D>(m->n_nodes), (unsigned)nv);
  launch_next(k_gather_nodes<D, T, kApply>, gn, kBlock, st, m->gptr, m->gent, m->nflag, m->n_nodes, E, w, nullptr, y,
              fmask, (m->n_elem << D) * (D + 3));
  note_launches(1);
}

// r = b - J x, and x += B (b - J x): the element part, then one node kernel.
// The colour schedule, which has no element-local buffer, is not used here.
template <int D, typename T>
static void jv_defect(const chns_mesh *m, const PhysCoef &pc, int variant, const KCoef<T> &c, const KCoef<T> *tab, const T *ut,
                      const T *dl, const T *b, const T *B, T *E, T *x, T *r, uint32_t fmask, cudaStream_t st) {
  elem_dispatch<D, T>(m, pc, variant == 4 ? 0 : variant, c, tab, ut, dl, x, E, st, 1);
  if (r)
    launch_next(k_gather_nodes<D, T, kDefect>, grid_gather<D>(m->n_nodes), kBlock, st, m->gptr, m->gent, m->nflag,
                m->n_nodes, E, x, b, r, fmask, 0);
  else
    launch_next(k_gather_smooth<D, T>, grid_for(m->n_nodes * 8), kBlock, st, m->gptr, m->gent, m->nflag, m->n_nodes, E,
                b, B, x, fmask);
  note_launches(1);
}

template <typename T>
void launch_jacvec(const chns_mesh *m, const PhysCoef &pc, const T *ut, const T *dl, const T *w, T *E, T *y,
                   cudaStream_t st, int variant, int nv) {
  KCoef<T> c = kcoef<T>(pc, m->dim);
  const KCoef<T> *tab = reinterpret_cast<const KCoef<T> *>(sizeof(T) == 8 ? m->coef64 : m->coef32);
  if (variant < 0) variant = sizeof(T) == 4 ? m->jv_variant : 0;
  if (m->dim == 2) jv_dispatch<2, T>(m, pc, variant, c, tab, ut, dl, w, E, y, pc.fmask, st, nv);
  else jv_dispatch<3, T>(m, pc, variant, c, tab, ut, dl, w, E, y, pc.fmask, st, nv);
}
template void launch_jacvec<float>(const chns_mesh *, const PhysCoef &, const float *, const float *,
                                   const float *, float *, float *, cudaStream_t, int, int);
template void launch_jacvec<double>(const chns_mesh *, const PhysCoef &, const double *, const double *,
                                    const double *, double *, double *, cudaStream_t, int, int);

// J.w straight from the states, without the preparation before it: two launches
// for a single apply.  On small meshes the host's launches are what an apply
// costs, back to back: 13.9..15.0 -> 11.7..12.7 us on uniform meshes of 64 to
// 16,384 leaves in 2D and 64 to 4,096 in 3D (a call waited for by itself: the
// same, 23..26 us).  Every corner of a leaf averages its node again, in double, so
// a large mesh loses: 32,768 leaves in 3D 15.6 -> 18.1 us, 65,536 in 2D
// 14.4 -> 13.8 but 31.1 -> 31.6 by itself.  With hanging nodes one corner
// averages up to four, one lane after another: 21,960 leaves 17.9 -> 31.8 us.
// false: the mesh, its schedule (one that the caller fixed runs as it is) or the
// states' alignment is not for this path.
bool launch_jacvec_states(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo, const float *w,
                          float *E, float *y, cudaStream_t st) {
  constexpr int64_t kStateCorners = 65536;
  if (m->n_hang || (m->n_elem << m->dim) > kStateCorners || m->jv_variant >= 4 || m->jv_fixed || m->coef32) return false;
  // node blocks of six doubles are read by pairs; the preparation reads single values
  if (m->dim == 3 && ((reinterpret_cast<uintptr_t>(Un) | reinterpret_cast<uintptr_t>(Uo)) & 15)) return false;
  const KCoef<float> c = kcoef<float>(pc, m->dim);
  const KPhys<F2> cp = pair_coef(c);
  const int64_t z = 0;
  if (m->dim == 2) {
    launch_next(k_jv_pair<2, 64, 8, true>, (unsigned)((m->n_elem * 2 + 63) / 64), 64, st, m->conn, m->level, m->hang,
                m->n_elem, Un, Uo, w, E, c, cp, z, z);
    launch_next(k_gather_nodes<2, float, kApply>, grid_gather<2>(m->n_nodes), kBlock, st, m->gptr, m->gent, m->nflag,
                m->n_nodes, E, w, nullptr, y, pc.fmask, z);
  } else {
    launch_next(k_jv_pair<3, 64, 6, true>, (unsigned)((m->n_elem * 4 + 63) / 64), 64, st, m->conn, m->level, m->hang,
                m->n_elem, Un, Uo, w, E, c, cp, z, z);
    launch_next(k_gather_nodes<3, float, kApply>, grid_gather<3>(m->n_nodes), kBlock, st, m->gptr, m->gent, m->nflag,
                m->n_nodes, E, w, nullptr, y, pc.fmask, z);
  }
  note_launches(2);
  return true;
}

template <typename T>
void launch_jacvec_defect(const chns_mesh *m, const PhysCoef &pc, const T *ut, const T *dl, const T *b, const T *B,
                          T *E, T *x, T *r, cudaStream_t st) {
  const KCoef<T> c = kcoef<T>(pc, m->dim);
  const KCoef<T> *tab = reinterpret_cast<const KCoef<T> *>(sizeof(T) == 8 ? m->coef64 : m->coef32);
  const int variant = sizeof(T) == 4 ? m->jv_variant : 0;
  if (m->dim == 2) jv_defect<2, T>(m, pc, variant, c, tab, ut, dl, b, B, E, x, r, pc.fmask, st);
  else jv_defect<3, T>(m, pc, variant, c, tab, ut, dl, b, B, E, x, r, pc.fmask, st);
}
template void launch_jacvec_defect<float>(const chns_mesh *, const PhysCoef &, const float *, const float *,
                                          const float *, const float *, float *, float *, float *, cudaStream_t);
template void launch_jacvec_defect<double>(const chns_mesh *, const PhysCoef &, const double *, const double *,
                                           const double *, const double *, double *, double *, double *,
                                           cudaStream_t);

// Gauss points with a floored tau_m radicand, added to *count (all elements
// in one launch, FP64 physics as in the residual)
void launch_tau_floor_count(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo,
                            unsigned long long *count, cudaStream_t st) {
  KCoef<double> c = kcoef<double>(pc, m->dim);
  const KCoef<double> *tab = reinterpret_cast<const KCoef<double> *>(m->coef64);
  if (m->dim == 2)
    k_element<2, double, 2, false, unsigned long long><<<grid_elem(m->n_elem << 2), kElemBlock, 0, st>>>(
        m->conn, m->level, m->hang, 0, m->n_elem, Un, Uo, nullptr, nullptr, count, c, tab, m->elem_inst, 0, 0,
        nullptr);
  else
    k_element<3, double, 2, false, unsigned long long><<<grid_elem(m->n_elem << 3), kElemBlock, 0, st>>>(
        m->conn, m->level, m->hang, 0, m->n_elem, Un, Uo, nullptr, nullptr, count, c, tab, m->elem_inst, 0, 0,
        nullptr);
  note_launches(1);
}

// x = M^-1 (node sums of E); v: six vectors of n_nodes; part: at least
// cg_partials() doubles; ctr: zero.  Status in *s (err 1: M not positive, 2: a
// barrier was given up).  polls: of a barrier, 0 for the default.
int cg_partials() { return 3 * kCgMaxGrid; }
cudaError_t launch_cg(const chns_mesh *m, const PhysCoef &pc, double *E, double *v, double *part, unsigned *ctr,
                      CgState *s, int max_it, int polls, cudaStream_t st) {
  CgArgs g{};
  const int64_t n = m->n_nodes;
  g.conn = m->conn; g.hang = m->hang; g.gptr = m->gptr; g.gent = m->gent; g.level = m->level;
  g.n_elem = m->n_elem; g.n = n;
  g.W0 = kcoef<double>(pc, m->dim).W0 * (m->dim == 2 ? 4.0 / 9.0 : 8.0 / 27.0);
  g.E = E; g.r = v; g.x = v + n; g.p = v + 2 * n; g.q = v + 3 * n; g.d = v + 4 * n; g.z = v + 5 * n;
  g.partial = part; g.bar = ctr; g.s = s; g.max_it = max_it;
  g.polls = polls > 0 ? polls : kCgPolls;
  int dev = 0, sms = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void *k = m->dim == 2 ? reinterpret_cast<const void *>(k_cg<2>) : reinterpret_cast<const void *>(k_cg<3>);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kCgBlock, 0);
  if (e != cudaSuccess) return e;
  // a warp of slots each is enough for a small mesh: fewer blocks, cheaper barriers
  const int64_t want = ((m->n_elem << m->dim) + kCgBlock - 1) / kCgBlock;
  const int grid = int(std::max<int64_t>(1, std::min<int64_t>({want, int64_t(sms) * per, kCgMaxGrid})));
  void *args[] = {&g};
  e = cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kCgBlock), args, 0, st);
  note_launches(1);
  return e;
}

void launch_mu_row(const chns_mesh *m, const PhysCoef &pc, const double *U, double *E, cudaStream_t st) {
  const KCoef<double> c = kcoef<double>(pc, m->dim);
  const unsigned g = grid_for(m->n_elem << m->dim);
  if (m->dim == 2) k_mu_row<2><<<g, kBlock, 0, st>>>(m->conn, m->level, m->hang, m->n_elem, U, c, E);
  else k_mu_row<3><<<g, kBlock, 0, st>>>(m->conn, m->level, m->hang, m->n_elem, U, c, E);
  note_launches(1);
}

chns_status upload_coef_tables(chns_mesh *m, const std::vector<PhysCoef> &pcs, cudaStream_t st) {
  const size_t n = pcs.size();
  if (!m->coef32) {
    CHNS_CUDA_TRY(cudaMalloc(&m->coef32, sizeof(KCoef<float>) * n));
    CHNS_CUDA_TRY(cudaMalloc(&m->coef64, sizeof(KCoef<double>) * n));
  }
  std::vector<KCoef<float>> a(n);
  std::vector<KCoef<double>> b(n);
  for (size_t i = 0; i < n; ++i) {
    a[i] = kcoef<float>(pcs[i], m->dim);
    b[i] = kcoef<double>(pcs[i], m->dim);
  }
  CHNS_CUDA_TRY(cudaMemcpyAsync(m->coef32, a.data(), sizeof(KCoef<float>) * n, cudaMemcpyHostToDevice, st));
  CHNS_CUDA_TRY(cudaMemcpyAsync(m->coef64, b.data(), sizeof(KCoef<double>) * n, cudaMemcpyHostToDevice, st));
  CHNS_CUDA_TRY(cudaStreamSynchronize(st));
  return CHNS_OK;
}

// the per-instance coefficient tables of src, copied to dst (same instances)
chns_status copy_coef_tables(const chns_mesh *src, chns_mesh *dst) {
  if (!src->coef32) { set_error("union mesh without coefficient tables"); return CHNS_ERR_ARG; }
  const size_t n = (size_t)src->n_inst;
  if (!dst->coef32) {
    CHNS_CUDA_TRY(cudaMalloc(&dst->coef32, sizeof(KCoef<float>) * n));
    CHNS_CUDA_TRY(cudaMalloc(&dst->coef64, sizeof(KCoef<double>) * n));
  }
  CHNS_CUDA_TRY(cudaMemcpy(dst->coef32, src->coef32, sizeof(KCoef<float>) * n, cudaMemcpyDeviceToDevice));
  CHNS_CUDA_TRY(cudaMemcpy(dst->coef64, src->coef64, sizeof(KCoef<double>) * n, cudaMemcpyDeviceToDevice));
  return CHNS_OK;
}

int64_t energy_blocks(const chns_mesh *m) { return std::min<int64_t>(grid_for(m->n_elem << m->dim), kEnergyBlocks); }

void launch_energy(const chns_mesh *m, const PhysCoef &pc, const double *U, double *partial, double *out3,
                   cudaStream_t st) {
  const int dim = m->dim;
  EnergyCoef c;
  double cad = 1.0, W = 1.0;
  for (int a = 0; a < dim; ++a) {
    cad *= CA;
    W *= 0.5 * pc.ext[a];
  }
  c.kv = 0.5 * cad * cad;
  // (1/(Cn We)) (psi + Cn^2/2 |grad phi|^2), psi = (phi^2 - 1)^2 / 4
  c.kpsi = 0.25 * pc.CnWe / pc.Cn2;
  c.z0 = 0.0;
  c.axes = 0;
  for (int a = 0; a < 3; ++a) {
    const double f = a < dim ? cad / (CA * pc.ext[a]) : 0.0;
    c.kg[a] = 0.5 * pc.CnWe * f * f;
    c.zg[a] = 0.0;
    if (a < dim) {
      c.z0 -= pc.g[a] * pc.inv_Fr * pc.lo[a];
      c.zg[a] = -pc.g[a] * pc.inv_Fr * pc.ext[a] / double(int64_t(1) << m->max_level);
      if (c.zg[a] != 0.0) c.axes |= 1 << a;
    }
  }
  c.alpha = pc.alpha;
  c.beta = pc.beta;
  c.W0 = W;
  c.cell = std::ldexp(W, -dim * m->max_level);
  const unsigned g = (unsigned)energy_blocks(m);
  if (dim == 2)
    launch_next(k_energy<2>, g, 256, st, m->conn, m->level, m->anchor, m->hang, m->n_elem, m->max_level, U, c, partial);
  else
    launch_next(k_energy<3>, g, 256, st, m->conn, m->level, m->anchor, m->hang, m->n_elem, m->max_level, U, c, partial);
  launch_next(k_energy_sum, 1, 96, st, partial, int(g), out3);
  note_launches(2);
}

}  // namespace chns
