// Shared-memory mixed-radix FFT core on pairs of lines.
//
// A point of a pair of lines is one float4 (re_a, re_b, im_a, im_b): the same
// point of line a and line b side by side.  Every butterfly then runs both
// lines at once in packed FP32 arithmetic (add / mul / fma .f32x2, one issue
// slot for two operations).  The FP32 pipe gives about 128 results per clock and
// SM either way: a register-only loop of 256 threads per CTA, two CTAs per SM,
// its time taken at 1.92 GHz, ran 65 complex additions per clock and SM as
// scalars and 67 packed, 22 complex multiply-adds as scalars and 34 packed.  A
// point is one 128-bit shared-memory access instead of two 64-bit ones, with one
// index and twiddle computation for both lines.
//
// Stage orders, plans, twiddle and position tables are those of fft.cuh.
#pragma once
#include <cuda_runtime.h>

#include "fft.cuh"
#include "mm_internal.h"

namespace mm {

typedef unsigned long long p2;  // two packed floats (a low, b high)

__device__ __forceinline__ p2 p2_pack(float a, float b) {
  p2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 p2_unpack(p2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ p2 p2_dup(float a) { return p2_pack(a, a); }
__device__ __forceinline__ p2 p2_add(p2 a, p2 b) {
  p2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 p2_mul(p2 a, p2 b) {
  p2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 p2_fma(p2 a, p2 b, p2 c) {
  p2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ p2 p2_sub(p2 a, p2 b) {
  p2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// the same point of two lines
struct c2 {
  p2 re, im;
};

__device__ __forceinline__ c2 c2_zero() { return c2{0ull, 0ull}; }
__device__ __forceinline__ c2 c2_make(float2 a, float2 b) { return c2{p2_pack(a.x, b.x), p2_pack(a.y, b.y)}; }
__device__ __forceinline__ float2 c2_a(c2 v) { return make_float2(p2_unpack(v.re).x, p2_unpack(v.im).x); }
__device__ __forceinline__ float2 c2_b(c2 v) { return make_float2(p2_unpack(v.re).y, p2_unpack(v.im).y); }
__device__ __forceinline__ c2 c2_load(const float4* p) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
  return c2{q.x, q.y};
}
__device__ __forceinline__ void c2_store(float4* p, c2 v) {
  *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.re, v.im);
}
__device__ __forceinline__ c2 operator+(c2 a, c2 b) { return c2{p2_add(a.re, b.re), p2_add(a.im, b.im)}; }
__device__ __forceinline__ c2 operator-(c2 a, c2 b) { return c2{p2_sub(a.re, b.re), p2_sub(a.im, b.im)}; }
// a + s b, s a real factor
__device__ __forceinline__ c2 c2_axpy(p2 s, c2 b, c2 a) { return c2{p2_fma(b.re, s, a.re), p2_fma(b.im, s, a.im)}; }
__device__ __forceinline__ c2 c2_scale(p2 s, c2 b) { return c2{p2_mul(b.re, s), p2_mul(b.im, s)}; }
// a + S i b and a - S i b (S = +-1)
template <int S> __device__ __forceinline__ c2 c2_add_i(c2 a, c2 b) {
  return S > 0 ? c2{p2_sub(a.re, b.im), p2_add(a.im, b.re)} : c2{p2_add(a.re, b.im), p2_sub(a.im, b.re)};
}
// a * (c + S i s)
template <int S> __device__ __forceinline__ c2 c2_mul(c2 a, p2 c, p2 s) {
  return S > 0 ? c2{p2_sub(p2_mul(a.re, c), p2_mul(a.im, s)), p2_fma(a.im, c, p2_mul(a.re, s))}
               : c2{p2_fma(a.re, c, p2_mul(a.im, s)), p2_sub(p2_mul(a.im, c), p2_mul(a.re, s))};
}
// a * exp(S 2 pi i j / N) for a constant angle of cosine c and sine s
template <int S> __device__ __forceinline__ c2 c2_rot(c2 a, float c, float s) {
  return c2_mul<S>(a, p2_dup(c), p2_dup(s));
}
// a * exp(S 2 pi i / 8) and a * exp(S 2 pi i 3 / 8)
template <int S> __device__ __forceinline__ c2 c2_rot8(c2 a) {
  const p2 h = p2_dup(0.70710678118654752440f);
  return S > 0 ? c2{p2_mul(h, p2_sub(a.re, a.im)), p2_mul(h, p2_add(a.re, a.im))}
               : c2{p2_mul(h, p2_add(a.re, a.im)), p2_mul(h, p2_sub(a.im, a.re))};
}
template <int S> __device__ __forceinline__ c2 c2_rot38(c2 a) {
  const p2 h = p2_dup(0.70710678118654752440f), nh = p2_dup(-0.70710678118654752440f);
  return S > 0 ? c2{p2_mul(nh, p2_add(a.re, a.im)), p2_mul(h, p2_sub(a.re, a.im))}
               : c2{p2_mul(h, p2_sub(a.im, a.re)), p2_mul(nh, p2_add(a.re, a.im))};
}
template <int S> __device__ __forceinline__ c2 c2_rot4(c2 a) {  // a * S i
  const p2 n = p2_dup(-1.f);
  return S > 0 ? c2{p2_mul(n, a.im), a.re} : c2{a.im, p2_mul(n, a.re)};
}

// Small DFTs y[k] = sum_n x[n] exp(S 2 pi i n k / R) in registers.
template <int R, int S> struct Dft2;

template <int S> struct Dft2<2, S> {
  static __device__ __forceinline__ void run(c2* x) {
    const c2 a = x[0], b = x[1];
    x[0] = a + b; x[1] = a - b;
  }
};
template <int S> struct Dft2<3, S> {
  static __device__ __forceinline__ void run(c2* x) {
    const float h = 0.86602540378443864676f;  // sqrt(3)/2
    const c2 t = x[1] + x[2], d = x[1] - x[2];
    const c2 m = c2_axpy(p2_dup(-0.5f), t, x[0]);
    const p2 hp = p2_dup(S > 0 ? h : -h), hn = p2_dup(S > 0 ? -h : h);
    x[0] = x[0] + t;
    x[1] = c2{p2_fma(d.im, hn, m.re), p2_fma(d.re, hp, m.im)};
    x[2] = c2{p2_fma(d.im, hp, m.re), p2_fma(d.re, hn, m.im)};
  }
};
template <int S> struct Dft2<4, S> {
  static __device__ __forceinline__ void run(c2* x) {
    const c2 a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = x[1] - x[3];
    x[0] = a + c; x[2] = a - c;
    x[1] = c2_add_i<S>(b, d); x[3] = c2_add_i<-S>(b, d);
  }
};
template <int S> struct Dft2<5, S> {
  static __device__ __forceinline__ void run(c2* x) {
    const p2 c1 = p2_dup(0.30901699437494742410f), c2_ = p2_dup(-0.80901699437494742410f);  // cos 2 pi/5, 4 pi/5
    const p2 s1 = p2_dup(0.95105651629515357212f), s2 = p2_dup(0.58778525229247312917f);     // sin
    const p2 n1 = p2_dup(-0.95105651629515357212f);
    const c2 t1 = x[1] + x[4], t2 = x[2] + x[3], d1 = x[1] - x[4], d2 = x[2] - x[3];
    const c2 a1 = c2_axpy(c1, t1, c2_axpy(c2_, t2, x[0]));
    const c2 a2 = c2_axpy(c2_, t1, c2_axpy(c1, t2, x[0]));
    const c2 b1 = c2_axpy(s1, d1, c2_scale(s2, d2));
    const c2 b2 = c2_axpy(s2, d1, c2_scale(n1, d2));
    x[0] = x[0] + (t1 + t2);
    x[1] = c2_add_i<S>(a1, b1); x[4] = c2_add_i<-S>(a1, b1);
    x[2] = c2_add_i<S>(a2, b2); x[3] = c2_add_i<-S>(a2, b2);
  }
};
// a * exp(S 2 pi i J / R) for the inner twiddles of the composite radices
template <int R, int J, int S> __device__ __forceinline__ c2 c2_root(c2 a) {
  constexpr int j = J % R;
  if constexpr (j == 0) return a;
  else if constexpr (4 * j == R) return c2_rot4<S>(a);
  else if constexpr (8 * j == R) return c2_rot8<S>(a);
  else if constexpr (8 * j == 3 * R) return c2_rot38<S>(a);
  else if constexpr (R == 16 && j == 1) return c2_rot<S>(a, 0.92387953251128675613f, 0.38268343236508977173f);
  else if constexpr (R == 16 && j == 3) return c2_rot<S>(a, 0.38268343236508977173f, 0.92387953251128675613f);
  else if constexpr (R == 16 && j == 9) return c2_rot<S>(a, -0.92387953251128675613f, -0.38268343236508977173f);
  else if constexpr (R == 9 && j == 1) return c2_rot<S>(a, 0.76604444311897803520f, 0.64278760968653932632f);
  else if constexpr (R == 9 && j == 2) return c2_rot<S>(a, 0.17364817766693034885f, 0.98480775301220805937f);
  else if constexpr (R == 9 && j == 4) return c2_rot<S>(a, -0.93969262078590838405f, 0.34202014332566873304f);
  else static_assert(R < 0, "no such inner twiddle");
}
// Composite R = A * B (DftComp's map): n = B n1 + n2, k = k1 + A k2
template <int A, int B, int S, int N2, int K1> __device__ __forceinline__ void comp_twiddles(c2 (*t)[A]) {
  if constexpr (N2 < B) {
    t[N2][K1] = c2_root<A * B, N2 * K1, S>(t[N2][K1]);
    if constexpr (K1 + 1 < A) comp_twiddles<A, B, S, N2, K1 + 1>(t);
    else comp_twiddles<A, B, S, N2 + 1, 1>(t);
  }
}
template <int A, int B, int S> struct Dft2Comp {
  static __device__ __forceinline__ void run(c2* x) {
    c2 t[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) t[n2][n1] = x[B * n1 + n2];
      Dft2<A, S>::run(t[n2]);
    }
    comp_twiddles<A, B, S, 1, 1>(t);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      c2 u[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][k1];
      Dft2<B, S>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) x[k1 + A * k2] = u[k2];
    }
  }
};
// Coprime R = A * B (DftPfa's map)
template <int A, int B, int S> struct Dft2Pfa {
  static __device__ __forceinline__ void run(c2* x) {
    constexpr int R = A * B;
    constexpr int eA = B * inv_mod(B % A, A), eB = A * inv_mod(A % B, B);
    c2 t[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) t[n2][n1] = x[(B * n1 + A * n2) % R];
      Dft2<A, S>::run(t[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      c2 u[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][k1];
      Dft2<B, S>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) x[(k1 * eA + k2 * eB) % R] = u[k2];
    }
  }
};
template <int S> struct Dft2<6, S> : Dft2Pfa<2, 3, S> {};
template <int S> struct Dft2<8, S> : Dft2Comp<2, 4, S> {};
template <int S> struct Dft2<9, S> : Dft2Comp<3, 3, S> {};
template <int S> struct Dft2<10, S> : Dft2Pfa<2, 5, S> {};
template <int S> struct Dft2<12, S> : Dft2Pfa<4, 3, S> {};
template <int S> struct Dft2<15, S> : Dft2Pfa<3, 5, S> {};
template <int S> struct Dft2<16, S> : Dft2Comp<4, 4, S> {};

// One stage of a plan: block length Lb = R M, L / R butterflies per line.  The
// lengths at run time, or (CtStage) as constants, so that the butterflies'
// shared-memory offsets fold into the instructions.
template <int R> struct RtStage {
  int L, Lb;
  unsigned mpl, mM;
  __device__ __forceinline__ RtStage(const FftPlanDev& P, int st)
      : L(P.L), Lb(P.blocklen[st]), mpl(P.magic_per_line[st]), mM(P.magic_M[st]) {}
  __device__ __forceinline__ int M() const { return Lb / R; }
  __device__ __forceinline__ int per_line() const { return L / R; }
  __device__ __forceinline__ int line(int b) const { return mpl ? (int)__umulhi((unsigned)b, mpl) : b; }
  __device__ __forceinline__ int block(int r) const { return mM ? (int)__umulhi((unsigned)r, mM) : r; }
};
template <int R, int L_, int Lb_> struct CtStage {
  static constexpr int Lb = Lb_;
  static __device__ __forceinline__ constexpr int M() { return Lb_ / R; }
  static __device__ __forceinline__ constexpr int per_line() { return L_ / R; }
  static __device__ __forceinline__ int line(int b) { return (int)((unsigned)b / (unsigned)per_line()); }
  static __device__ __forceinline__ int block(int r) { return (int)((unsigned)r / (unsigned)M()); }
};

// The block's butterflies of one stage over `nlines` lines:
// f(line, blk Lb + n1, n1) for each.
template <typename G, typename F> __device__ __forceinline__ void fft2_butterflies(const G& g, int nlines, F f) {
  const int nb = nlines * g.per_line();
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const int line = g.line(b);
    const int rem = b - line * g.per_line();
    const int blk = g.block(rem);
    const int n1 = rem - blk * g.M();
    f(line, blk * g.Lb + n1, n1);
  }
}

// Twiddles of a butterfly from the pair table: row n1 holds (c, c, s, s) of
// W^{n1 k} for k = 1 .. R-1, so the loads have constant offsets and feed the
// packed products as they are (half the table, widened in registers, measured
// 10% slower in the y pass).  The inverse takes conjugates.
template <int R, int S> __device__ __forceinline__ void fft2_twiddle(c2* v, const float4* row) {
#pragma unroll
  for (int k = 1; k < R; ++k) {
    const c2 w = c2_load(row + (k - 1));
    v[k] = c2_mul<-S>(v[k], w.re, w.im);
  }
}
__host__ __device__ constexpr int fft2_pitch(int R) { return (R - 1) | 1; }  // odd: rows spread over the banks

// A stage in place on lines of stride ldl.
template <int R, int MODE, typename G>
__device__ __forceinline__ void fft2_stage(const G& g, float4* buf, int ldl, int nlines, const float4* tw) {
  constexpr int S = MODE == kFwdDif ? -1 : 1;
  const int M = g.M();
  fft2_butterflies(g, nlines, [&](int line, int n0, int n1) {
    float4* p = buf + (line * ldl + n0);
    c2 v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = c2_load(p + k * M);
    if (MODE == kInvDit && M > 1) fft2_twiddle<R, S>(v, tw + n1 * fft2_pitch(R));
    Dft2<R, S>::run(v);
    if (MODE != kInvDit && M > 1) fft2_twiddle<R, S>(v, tw + n1 * fft2_pitch(R));
#pragma unroll
    for (int k = 0; k < R; ++k) c2_store(p + k * M, v[k]);
  });
}
// The first stage of a decimation-in-frequency transform, the points n0 + k M
// of a butterfly of line l read through ld(l, n0, M, v); twiddles from the
// plan's global table (coalesced).
template <int R, typename G, typename Ld>
__device__ __forceinline__ void fft2_first(const G& g, float4* buf, int ldl, int nlines,
                                           const float2* __restrict__ tw, Ld ld) {
  constexpr int S = -1;
  const int M = g.M();
  fft2_butterflies(g, nlines, [&](int line, int n0, int n1) {
    c2 v[R];
    ld(line, n0, M, v);
    Dft2<R, S>::run(v);
    if (M > 1) {
      const float2* col = tw + n1;
#pragma unroll
      for (int k = 1; k < R; ++k) {
        const float2 w = __ldg(col + (k - 1) * M);
        v[k] = c2_mul<-S>(v[k], p2_dup(w.x), p2_dup(w.y));
      }
    }
    float4* p = buf + (line * ldl + n0);
#pragma unroll
    for (int k = 0; k < R; ++k) c2_store(p + k * M, v[k]);
  });
}
// The last stage of a decimation-in-time inverse, the points n0 + k M of a
// butterfly of line l given to st(l, n0, M, v).
template <int R, typename G, typename St>
__device__ __forceinline__ void fft2_last(const G& g, const float4* buf, int ldl, int nlines, const float4* tw, St st) {
  const int M = g.M();
  fft2_butterflies(g, nlines, [&](int line, int n0, int n1) {
    const float4* p = buf + (line * ldl + n0);
    c2 v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = c2_load(p + k * M);
    if (M > 1) fft2_twiddle<R, 1>(v, tw + n1 * fft2_pitch(R));
    Dft2<R, 1>::run(v);
    st(line, n0, M, v);
  });
}

#define MM_RADICES(STAGE) STAGE(2) STAGE(3) STAGE(4) STAGE(5) STAGE(6) STAGE(8) STAGE(9) STAGE(10) STAGE(12) STAGE(15) STAGE(16)

// The transforms of a block with the plan at run time (the radices of RSET
// compiled in) ...
template <unsigned RSET> struct RtPair {
  static constexpr int kL = 0;
  // Forward (decimation-in-frequency) transforms of `nlines` lines of
  // buf (stride ldl): line l's points come from ld(l, n0, M, v); then also()
  // runs, before the first barrier (it may fill tw, the pair table, and what
  // else is needed later, while the first loads are on their way).  Ends with a
  // barrier.
  template <typename Ld, typename Also>
  static __device__ __forceinline__ void in(float4* buf, int ldl, int nlines, const FftTables& T, const float4* tw,
                                            Ld ld, Also also) {
    const FftPlanDev& P = T.plan;
    switch (P.radix[0]) {
#define MM_STAGE(R) \
  case R: if constexpr ((RSET & radix_bit(R)) != 0u) fft2_first<R>(RtStage<R>(P, 0), buf, ldl, nlines, T.tw_f, ld); break;
      MM_RADICES(MM_STAGE)
#undef MM_STAGE
      default: break;
    }
    also();
    __syncthreads();
    for (int s = 1; s < P.nstages; ++s) {
      const float4* ts = tw + T.tw2_off[s];
      switch (P.radix[s]) {
#define MM_STAGE(R) \
  case R: if constexpr ((RSET & radix_bit(R)) != 0u) fft2_stage<R, kFwdDif>(RtStage<R>(P, s), buf, ldl, nlines, ts); break;
        MM_RADICES(MM_STAGE)
#undef MM_STAGE
        default: break;
      }
      __syncthreads();
    }
  }
  // Decimation-in-time inverses of `nlines` lines of buf, the last stage's
  // points going to st(l, n0, M, v).  Ends with a barrier.
  template <typename St>
  static __device__ __forceinline__ void out(float4* buf, int ldl, int nlines, const FftTables& T, const float4* tw,
                                             St st) {
    const FftPlanDev& P = T.plan;
    for (int s = P.nstages - 1; s > 0; --s) {
      const float4* ts = tw + T.tw2_off[s];
      switch (P.radix[s]) {
#define MM_STAGE(R) \
  case R: if constexpr ((RSET & radix_bit(R)) != 0u) fft2_stage<R, kInvDit>(RtStage<R>(P, s), buf, ldl, nlines, ts); break;
        MM_RADICES(MM_STAGE)
#undef MM_STAGE
        default: break;
      }
      __syncthreads();
    }
    switch (P.radix[0]) {
#define MM_STAGE(R) \
  case R: if constexpr ((RSET & radix_bit(R)) != 0u) fft2_last<R>(RtStage<R>(P, 0), buf, ldl, nlines, tw, st); break;
      MM_RADICES(MM_STAGE)
#undef MM_STAGE
      default: break;
    }
    __syncthreads();
  }
};

// ... and for one plan R0 R1 R2 (R3) known at compile time, on lines of stride
// L + PAD.
template <int R0, int R1, int R2, int R3 = 1, int PAD = 0> struct CtPair {
  static constexpr int kL = R0 * R1 * R2 * R3, ldl = kL + PAD;
  static bool is(const FftPlanDev& P) {
    return P.nstages == (R3 > 1 ? 4 : 3) && P.radix[0] == R0 && P.radix[1] == R1 && P.radix[2] == R2 &&
           (R3 == 1 || P.radix[3] == R3);
  }
  template <typename Ld, typename Also>
  static __device__ __forceinline__ void in(float4* buf, int, int nlines, const FftTables& T, const float4* tw, Ld ld,
                                            Also also) {
    fft2_first<R0>(CtStage<R0, kL, kL>(), buf, ldl, nlines, T.tw_f, ld);
    also();
    __syncthreads();
    fft2_stage<R1, kFwdDif>(CtStage<R1, kL, R1 * R2 * R3>(), buf, ldl, nlines, tw + T.tw2_off[1]);
    __syncthreads();
    fft2_stage<R2, kFwdDif>(CtStage<R2, kL, R2 * R3>(), buf, ldl, nlines, tw + T.tw2_off[2]);
    __syncthreads();
    if constexpr (R3 > 1) {
      fft2_stage<R3, kFwdDif>(CtStage<R3, kL, R3>(), buf, ldl, nlines, tw);
      __syncthreads();
    }
  }
  template <typename St>
  static __device__ __forceinline__ void out(float4* buf, int, int nlines, const FftTables& T, const float4* tw, St st) {
    if constexpr (R3 > 1) {
      fft2_stage<R3, kInvDit>(CtStage<R3, kL, R3>(), buf, ldl, nlines, tw);
      __syncthreads();
    }
    fft2_stage<R2, kInvDit>(CtStage<R2, kL, R2 * R3>(), buf, ldl, nlines, tw + T.tw2_off[2]);
    __syncthreads();
    fft2_stage<R1, kInvDit>(CtStage<R1, kL, R1 * R2 * R3>(), buf, ldl, nlines, tw + T.tw2_off[1]);
    __syncthreads();
    fft2_last<R0>(CtStage<R0, kL, kL>(), buf, ldl, nlines, tw, st);
    __syncthreads();
  }
};

// The plans a pass on pair lines is compiled for.  A build is taken where every
// job's plan is its own, stage by stage (CtPair::is): a plan and the stages run
// over its tables cannot differ.  Else the plan at run time.
template <typename... Plans> struct PairPlans {
  static bool has(const FftPlanDev& P) { return (Plans::is(P) || ...); }
  static bool has_length(int L) { return ((Plans::kL == L) || ...); }
  // the kernel Pass::build<Fft>() of a launch, whose jobs hold the tables `t`;
  // lengths that never reach the pass (Pass::takes) get no build
  template <typename Pass, typename JobT>
  static auto kernel(const Launch<JobT>& L, FftTables JobT::*t) {
    unsigned rs = 0;
    for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set((L.job[i].*t).plan);
    auto k = (rs & ~kRadixSetB) == 0u ? Pass::template build<RtPair<kRadixSetB>>()
                                      : Pass::template build<RtPair<kAllRadices>>();
    auto all = [&](bool (*is)(const FftPlanDev&)) {
      for (int i = 0; i < L.njobs; ++i)
        if (!is((L.job[i].*t).plan)) return false;
      return true;
    };
    auto take = [&](auto plan) {
      if constexpr (Pass::takes(decltype(plan)::kL))
        if (all(&decltype(plan)::is)) k = Pass::template build<decltype(plan)>();
    };
    (take(Plans()), ...);
    return k;
  }
};

}  // namespace mm
