// Double-float arithmetic for the high-precision residuals of the mixed
// precision tracker.
//
// A double-float is the unevaluated sum hi + lo of two FP32 numbers
// (|lo| <= ulp(hi) / 2 after normalisation): about 48 significant bits with
// FP32's exponent range.  Its sums and products are built from error-free
// transformations:
//   TwoSum      (Knuth, TAOCP vol. 2, Sec. 4.2.2): s + e = a + b exactly,
//   TwoProd     with a fused multiply-add:          p + e = a * b exactly,
// in the arrangement of the double-word algorithms analysed by Joldes,
// Muller and Popescu, "Tight and rigorous error bounds for basic building
// blocks of double-word arithmetic" (ACM TOMS 44(2), 2017).  Everything runs
// on the FP32 pipe: GB300 issues FP64 FMAs at about 1/74 of its FP32 rate,
// so a double-float complex multiply-add (about 60 FP32 instructions) costs a
// fifth of the pipe time of the 4 native FP64 FMAs it replaces.
//
// What the tracker needs from it is a residual H(x, t) whose error is small
// against the size of the terms it sums (the backward-error scale): the
// accumulations below bound the absolute error of c + a b by a small
// multiple of u^2 (|c| + |a| |b|), u = 2^-24, which is what a cancelling sum
// needs; the relative error of a result that cancels is not bounded, and is
// not needed.
//
// The intrinsics __fadd_rn, __fsub_rn, __fmul_rn and __fmaf_rn are never
// contracted or reassociated by the compiler, which the transformations rely on.
#pragma once

#include "hc_device.cuh"

namespace hc {

// Besides the explicit functions below, df is an arithmetic type (the
// operators and overloads at the end of this file), so that the evaluators
// and the dense solve -- templates on their real type R -- run in
// double-floats with R = df: the kernels of the double-float precision
// (HC_PREC_DF) and of the last re-tracking tier of the mixed pipeline.
struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ constexpr explicit df(int v) : hi((float)v), lo(0.f) {}
  // nearest double-float to v (hi carries the leading 24 bits)
  __host__ __device__ explicit df(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
  __host__ __device__ explicit operator float() const { return hi + lo; }
  __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
};

// s + e = a + b exactly (six operations, no precondition)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// p + e = a * b exactly (barring underflow)
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}

// nearest double-float to a double (hi carries the leading 24 bits)
__device__ __forceinline__ df to_df(double v) {
  const float h = __double2float_rn(v);
  return df{h, __double2float_rn(v - (double)h)};
}
__device__ __forceinline__ float df_to_float(df a) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

// c + x1 y1 + x2 y2.  The two leading products are exact (TwoProd); their
// errors and the cross terms hi * lo go into the low part (the dropped
// lo * lo terms are below u^2 |x y|); the high parts are added by TwoSum and
// the result renormalised by a final TwoSum.
__device__ __forceinline__ df df_dot2(df c, df x1, df y1, df x2, df y2) {
  float p1, e1, p2, e2;
  two_prod(x1.hi, y1.hi, p1, e1);
  two_prod(x2.hi, y2.hi, p2, e2);
  float l = __fmaf_rn(x1.hi, y1.lo, __fmaf_rn(x1.lo, y1.hi, e1));
  l = __fadd_rn(l, __fmaf_rn(x2.hi, y2.lo, __fmaf_rn(x2.lo, y2.hi, e2)));
  float s, es, s2, es2;
  two_sum(c.hi, p1, s, es);
  two_sum(s, p2, s2, es2);
  const float lo = __fadd_rn(__fadd_rn(c.lo, l), __fadd_rn(es, es2));
  df r;
  two_sum(s2, lo, r.hi, r.lo);
  return r;
}

// a + b
__device__ __forceinline__ df df_add(df a, df b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  const float lo = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  df r;
  two_sum(s, lo, r.hi, r.lo);
  return r;
}

// Packed form: the real and the imaginary part of a complex double-float run
// the same operations, so each operation is one two-wide FP32 instruction
// (FADD2, FMUL2, FFMA2) over (re, im).  These round each half as the scalar
// instruction does -- the results are the scalar form's bit for bit -- and take
// the FP32 pipe as long as two scalar ones (measured: 2 cycles a warp
// instruction and scheduler, latency 5, negated operands free), but half the
// issue slots and half the code: a complex multiply-add 97 -> 70 cycles with
// one warp per scheduler and 73 -> 64 with four, and code is what the
// double-float kernels stall on (see run_tracker).
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// Complex double-float in registers, shared and global memory: one 16-byte
// word, high parts (re, im) then low parts.
template <>
struct __align__(16) cx<df> {
  float2 h, l;
};
__device__ __forceinline__ df re_of(cx<df> z) { return df{z.h.x, z.l.x}; }
__device__ __forceinline__ df im_of(cx<df> z) { return df{z.h.y, z.l.y}; }
template <>
__device__ __forceinline__ cx<df> mk<df>(df re, df im) {
  return cx<df>{make_float2(re.hi, im.hi), make_float2(re.lo, im.lo)};
}
template <>
__device__ __forceinline__ cx<df> czero<df>() {
  return cx<df>{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
}

// c + x1 y1 + x2 y2 in both halves (df_dot2)
__device__ __forceinline__ cx<df> dot2p(cx<df> c, cx<df> x1, cx<df> y1, cx<df> x2, cx<df> y2) {
  const float2 p1 = mul2(x1.h, y1.h), e1 = fma2(x1.h, y1.h, neg2(p1));
  const float2 p2 = mul2(x2.h, y2.h), e2 = fma2(x2.h, y2.h, neg2(p2));
  float2 l = fma2(x1.h, y1.l, fma2(x1.l, y1.h, e1));
  l = add2(l, fma2(x2.h, y2.l, fma2(x2.l, y2.h, e2)));
  float2 s, es, s2, es2;
  two_sum2(c.h, p1, s, es);
  two_sum2(s, p2, s2, es2);
  const float2 lo = add2(add2(c.l, l), add2(es, es2));
  cx<df> r;
  two_sum2(s2, lo, r.h, r.l);
  return r;
}
// x1 y1 + x2 y2 in both halves (df_sdot2)
__device__ __forceinline__ cx<df> sdot2p(cx<df> x1, cx<df> y1, cx<df> x2, cx<df> y2) {
  const float2 p1 = mul2(x1.h, y1.h), e1 = fma2(x1.h, y1.h, neg2(p1));
  const float2 p2 = mul2(x2.h, y2.h), e2 = fma2(x2.h, y2.h, neg2(p2));
  float2 l = fma2(x1.h, y1.l, fma2(x1.l, y1.h, e1));
  l = add2(l, fma2(x2.h, y2.l, fma2(x2.l, y2.h, e2)));
  float2 s, es;
  two_sum2(p1, p2, s, es);
  cx<df> r;
  two_sum2(s, add2(l, es), r.h, r.l);
  return r;
}
// x y in both halves (operator* of df)
__device__ __forceinline__ cx<df> mulp(cx<df> x, cx<df> y) {
  const float2 p = mul2(x.h, y.h);
  const float2 e = fma2(x.h, y.l, fma2(x.l, y.h, fma2(x.h, y.h, neg2(p))));
  cx<df> r;
  two_sum2(p, e, r.h, r.l);
  return r;
}
// operands of a complex product a b = (a.re b.re - a.im b.im,
// a.re b.im + a.im b.re): both halves a.re; (-a.im, a.im); b swapped
__device__ __forceinline__ cx<df> re_re(cx<df> a) { return {dup2(a.h.x), dup2(a.l.x)}; }
__device__ __forceinline__ cx<df> nim_im(cx<df> a) {
  return {make_float2(-a.h.y, a.h.y), make_float2(-a.l.y, a.l.y)};
}
__device__ __forceinline__ cx<df> im_re(cx<df> b) { return {swap2(b.h), swap2(b.l)}; }
__device__ __forceinline__ cx<df> neg(cx<df> a) { return {neg2(a.h), neg2(a.l)}; }

// The complex double-float of the residuals (tables, the mixed kernels' point
// copies): the same word.
struct __align__(16) cdf {
  float hr, hi_, lr, li;  // hi part (re, im), lo part (re, im)
  __host__ __device__ df re() const { return df{hr, lr}; }
  __host__ __device__ df im() const { return df{hi_, li}; }
};
__device__ __forceinline__ cx<df> to_cxdf(cdf z) {
  return {make_float2(z.hr, z.hi_), make_float2(z.lr, z.li)};
}
__device__ __forceinline__ cdf to_cdf(cx<df> z) { return cdf{z.h.x, z.h.y, z.l.x, z.l.y}; }

__device__ __forceinline__ cdf mk_cdf(df re, df im) { return cdf{re.hi, im.hi, re.lo, im.lo}; }
__device__ __forceinline__ cdf to_cdf(cx<double> z) { return mk_cdf(to_df(z.re), to_df(z.im)); }
__device__ __forceinline__ cdf cdf_zero() { return cdf{0.f, 0.f, 0.f, 0.f}; }
__device__ __forceinline__ cx<float> cdf_to_cf(cdf z) {
  return cx<float>{df_to_float(z.re()), df_to_float(z.im())};
}
__device__ __forceinline__ cx<double> cdf_to_cd(cdf z) {
  return cx<double>{df_to_double(z.re()), df_to_double(z.im())};
}

// acc + a b
__device__ __forceinline__ cdf cdf_fma(cdf a, cdf b, cdf acc) {
  const cx<df> pa = to_cxdf(a), pb = to_cxdf(b);
  return to_cdf(dot2p(to_cxdf(acc), re_re(pa), pb, nim_im(pa), im_re(pb)));
}
// a b
__device__ __forceinline__ cdf cdf_mul(cdf a, cdf b) { return cdf_fma(a, b, cdf_zero()); }
__device__ __forceinline__ cx<df> addp(cx<df> a, cx<df> b) {
  float2 s, e;
  two_sum2(a.h, b.h, s, e);
  cx<df> r;
  two_sum2(s, add2(e, add2(a.l, b.l)), r.h, r.l);
  return r;
}
__device__ __forceinline__ cdf cdf_add(cdf a, cdf b) { return to_cdf(addp(to_cxdf(a), to_cxdf(b))); }
__device__ __forceinline__ cdf cdf_sub(cdf a, cdf b) {
  return to_cdf(addp(to_cxdf(a), neg(to_cxdf(b))));
}
// a real double-float times a complex one
__device__ __forceinline__ cdf cdf_scale(df s, cdf a) {
  const cx<df> z = czero<df>();
  return to_cdf(dot2p(z, cx<df>{dup2(s.hi), dup2(s.lo)}, to_cxdf(a), z, z));
}

// host-side split of a complex double (tables and launch arguments)
inline cdf split_cdf_host(double re, double im) {
  const float hr = (float)re, hi = (float)im;
  return cdf{hr, hi, (float)(re - (double)hr), (float)(im - (double)hi)};
}

// |z| from the high parts (scales and tests need FP32 accuracy only)
__device__ __forceinline__ float cdf_abs_hi(cdf z) { return sqrtf(fmaf(z.hr, z.hr, z.hi_ * z.hi_)); }

// ---------------------------------------------------------------- df as R
// Real operations.  Sums: df_add (TwoSum of the high parts, the low parts
// added, renormalised).  Products: x y with the exact TwoProd of the high
// parts plus the cross terms.  Both are accurate to a small multiple of
// u^2 = 2^-48 relative to the operands' magnitudes.
__device__ __forceinline__ df operator+(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ df operator-(df a) { return df{-a.hi, -a.lo}; }
__device__ __forceinline__ df operator-(df a, df b) { return df_add(a, df{-b.hi, -b.lo}); }
__device__ __forceinline__ df operator*(df a, df b) {
  float p, e;
  two_prod(a.hi, b.hi, p, e);
  e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
  df r;
  two_sum(p, e, r.hi, r.lo);
  return r;
}

// x1 y1 + x2 y2 (df_dot2 without the addend)
__device__ __forceinline__ df df_sdot2(df x1, df y1, df x2, df y2) {
  float p1, e1, p2, e2;
  two_prod(x1.hi, y1.hi, p1, e1);
  two_prod(x2.hi, y2.hi, p2, e2);
  float l = __fmaf_rn(x1.hi, y1.lo, __fmaf_rn(x1.lo, y1.hi, e1));
  l = __fadd_rn(l, __fmaf_rn(x2.hi, y2.lo, __fmaf_rn(x2.lo, y2.hi, e2)));
  float s, es;
  two_sum(p1, p2, s, es);
  df r;
  two_sum(s, __fadd_rn(l, es), r.hi, r.lo);
  return r;
}

// 1 / d: one Newton step r = r0 + r0 (1 - d r0) from the FP32 reciprocal
// r0 of the high part; the residual 1 - d r0 is formed with df_dot2, which
// keeps it exact to u^2 while it cancels (accuracy about u^2 relative).
__device__ __forceinline__ df df_recip(df d) {
  const float r0 = __frcp_rn(d.hi);
  const df one{1.f, 0.f}, z{0.f, 0.f};
  const df e = df_dot2(one, df{-d.hi, -d.lo}, df{r0, 0.f}, z, z);
  return df_add(df{r0, 0.f}, df{r0, 0.f} * e);
}

// Complex operations on cx<df> (overloads of the templates in
// hc_device.cuh; a complex product is two two-term dot products).
__device__ __forceinline__ cx<df> operator+(cx<df> a, cx<df> b) { return addp(a, b); }
__device__ __forceinline__ cx<df> operator-(cx<df> a) { return neg(a); }
__device__ __forceinline__ cx<df> operator-(cx<df> a, cx<df> b) { return addp(a, neg(b)); }
__device__ __forceinline__ cx<df> operator*(df s, cx<df> a) {
  return mulp(cx<df>{dup2(s.hi), dup2(s.lo)}, a);
}
__device__ __forceinline__ cx<df> operator*(cx<df> a, cx<df> b) {
  return sdot2p(re_re(a), b, nim_im(a), im_re(b));
}
__device__ __forceinline__ cx<df> cfma(cx<df> a, cx<df> b, cx<df> acc) {
  return dot2p(acc, re_re(a), b, nim_im(a), im_re(b));
}
__device__ __forceinline__ cx<df> cfms(cx<df> a, cx<df> b, cx<df> acc) {
  return dot2p(acc, neg(re_re(a)), b, neg(nim_im(a)), im_re(b));
}
// 1/z = conj(z) / |z|^2 (|z| must stay inside FP32's range, as for the
// FP32 solve: a pivot outside it gives a non-finite reciprocal and the step
// is rejected)
__device__ __forceinline__ cx<df> crecip(cx<df> z) {
  const df re = re_of(z), im = im_of(z);
  const df inv = df_recip(df_sdot2(re, re, im, im));
  const cx<df> r = mulp(z, cx<df>{dup2(inv.hi), dup2(inv.lo)});
  return {make_float2(r.h.x, -r.h.y), make_float2(r.l.x, -r.l.y)};
}
// magnitudes for pivot choice and tests: FP32 accuracy from the high parts
__device__ __forceinline__ float cabs1(cx<df> z) { return fabsf(z.h.x) + fabsf(z.h.y); }
__device__ __forceinline__ float cnorm2(cx<df> z) { return fmaf(z.h.x, z.h.x, z.h.y * z.h.y); }
__device__ __forceinline__ float cabs2(cx<df> z) { return sqrtf(cnorm2(z)); }
// complex double <-> complex double-float
__device__ __forceinline__ cx<df> to_cxdf(cx<double> z) { return mk<df>(df(z.re), df(z.im)); }
// butterfly sum over the lanes xor o (o = L .. L * PARTS / 2) of a warp
__device__ __forceinline__ df shfl_xor_df(df v, int o) {
  return df{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ cx<df> shfl_xor_df(cx<df> v, int o) {
  return {make_float2(__shfl_xor_sync(0xffffffffu, v.h.x, o),
                      __shfl_xor_sync(0xffffffffu, v.h.y, o)),
          make_float2(__shfl_xor_sync(0xffffffffu, v.l.x, o),
                      __shfl_xor_sync(0xffffffffu, v.l.y, o))};
}

// The elimination of gj_solve (hc_device.cuh) for double-float rows held in
// shared memory: entry j of row r at A[j * LR + r], LR = lanes per row replica,
// PARTS replicas (lane gl: row gl mod LR, columns j with j mod PARTS = gl / LR).
// Rolled over the pivots and over the columns (UNROLL of a lane's columns at a
// time, to cover the chain of a multiply-add): unrolled with the row in
// registers, the solve alone was 60 to 150 KB of code, and a path's warp,
// often the only one of its scheduler, waited for instructions at 5.6 cycles
// each (see run_tracker).  Measured with the packed arithmetic and rolled
// evaluations, ms: precision DF on cubic n = 8 (16 systems) 3464 -> 430, on quadratic
// n = 6 (64) 27.7 -> 7.4; re-tracking of cubic n = 8 31.5 -> 18.9.  The same
// operations in the same order per entry, so the same results.  W columns: N and the right-hand sides.  pv: W entries.  On
// return the lanes of part 0 hold in col the column they pivoted on (-1: none)
// and in dinv 1 / pivot: that component of x is dinv times the right-hand side.
template <int N, int LR, int PARTS, bool MEET>
__device__ __forceinline__ bool gj_solve_df(const Group& g, cx<df>* A, cx<df>* pv, int W,
                                            cx<df>& dinv, int& col) {
  constexpr int L = LR * PARTS;
  constexpr int UNROLL = PARTS >= 4 ? 2 : 3;
  const int r = g.gl & (LR - 1), part = PARTS > 1 ? g.gl / LR : 0;
  bool used = r >= N;
  dinv = mk<df>(df(1), df(0));
  unsigned lo = 0xffffffffu, hi = 0u;
  col = -1;
#pragma unroll 1
  for (int k = 0; k < N; ++k) {
    const cx<df> ak = A[k * LR + r];
    const float m = cabs1(ak);
    const unsigned key = used ? 0u : ((__float_as_uint(m) & ~31u) | (unsigned)(31 - r));
    const unsigned kmax = gmaxu<L, MEET>(g, key);
    const cx<df> inv = crecip(ak);
    lo = min(lo, kmax);
    hi = max(hi, kmax);
    const int rp = min(31 - (int)(kmax & 31u), LR - 1);  // the pivot row
    const bool me = r == rp;
    for (int j = k + 1 + g.gl; j < W; j += L) pv[j] = A[j * LR + rp];
    if (me) {
      if (part == 0) pv[k] = inv;
      used = true;
      dinv = inv;
      col = k;
    }
    __syncwarp(g.meet);
    const cx<df> l = me ? czero<df>() : ak * pv[k];
    const cx<df> lr = neg(re_re(l)), li = neg(nim_im(l));
    // a lane's first column behind k
    const int j0 = k + 1 + (PARTS > 1 ? ((part - (k + 1)) & (PARTS - 1)) : 0);
#pragma unroll 1
    for (int j = j0; j < W; j += UNROLL * PARTS) {
      cx<df> a[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        // (behind the last column: this lane's own j, as another lane may be storing W - 1)
        const int ju = j + u * PARTS < W ? j + u * PARTS : j;
        const cx<df> p = pv[ju];
        a[u] = dot2p(A[ju * LR + r], lr, p, li, im_re(p));
      }
#pragma unroll
      for (int u = 0; u < UNROLL; ++u)
        if (j + u * PARTS < W) A[(j + u * PARTS) * LR + r] = a[u];
    }
    __syncwarp(g.meet);
  }
  if (part != 0 || r >= N) col = -1;
  return (lo & ~31u) != 0u && (hi & ~31u) < 0x7f800000u;
}

}  // namespace hc
