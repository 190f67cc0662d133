// Shared device/host helpers for the DDA CUDA path: complex types and
// arithmetic, error plumbing.  Nothing here is specific to one kernel.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cstdio>
#include <type_traits>
#include <string>

namespace dda {

// ---- double-float reals -------------------------------------------------------
// A value hi + lo held in two floats (|lo| <= ulp(hi)/2), with arithmetic by
// error-free transformations: Knuth's two-sum for addition and the FMA
// two-product (exact product of two floats as p + fma(a, b, -p)) for
// multiplication (Dekker 1971; Shewchuk 1997).  About 44 significant bits:
// an FFT matvec in this arithmetic is accurate to ~1e-12 relative, far below
// the residual tolerances it checks, and runs on the FP32 pipes, which on
// GB300 have ~58x the FP64 throughput.  Addition uses the cheaper variant
// whose error is bounded relative to |a| + |b| (enough for FFT sums).
struct dfl {
    float hi, lo;
    dfl() = default;
    __host__ __device__ constexpr dfl(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ dfl(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ dfl(int i) : hi((float)i), lo(0.f) {}
    __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
};

__host__ __device__ __forceinline__ dfl operator-(dfl a) { return dfl(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ dfl operator+(dfl a, dfl b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    float e = (a.hi - (s - bb)) + (b.hi - bb);  // two-sum error of the leading parts
    e += a.lo + b.lo;
    const float h = s + e;
    return dfl(h, e - (h - s));
}
__host__ __device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
__host__ __device__ __forceinline__ dfl operator*(dfl a, dfl b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);  // exact error of the float product
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float h = p + e;
    return dfl(h, e - (h - p));
}

// Complex double-float: the leading floats of the two parts side by side, then
// their corrections, so that one packed instruction (add, mul, fma .f32x2) works
// on both parts.  Packed instructions run the same operations per clock in half
// the issue slots, and the double-float passes issue little else.  Aligned to its
// 16 bytes, so that it moves in one load or store (as four floats it took four).
struct __align__(16) cdfl {
    float2 hi, lo;
};
__host__ __device__ __forceinline__ cdfl make_cdfl(dfl re, dfl im) {
    cdfl r;
    r.hi = make_float2(re.hi, im.hi);
    r.lo = make_float2(re.lo, im.lo);
    return r;
}

template <typename T> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <> struct cplx_of<dfl> { using type = cdfl; };
template <typename T> using cx = typename cplx_of<T>::type;

template <typename C> struct real_of;
template <> struct real_of<float2> { using type = float; };
template <> struct real_of<double2> { using type = double; };
template <> struct real_of<cdfl> { using type = dfl; };

__host__ __device__ __forceinline__ float2 mk(float re, float im) { return make_float2(re, im); }
__host__ __device__ __forceinline__ double2 mk(double re, double im) { return make_double2(re, im); }

template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) { C r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) { C r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
// g0 p0 + g1 p1 + g2 p2 (a row of the 3x3 product in Fourier space) as one
// FMA chain per part: 12 instructions for complex64 instead of the 16 of
// three products and two sums (IEEE rules forbid the compiler this
// reassociation)
template <typename C> __host__ __device__ __forceinline__ C cdot3(C g0, C p0, C g1, C p1, C g2, C p2) {
    C r;
    if constexpr (std::is_same<C, float2>::value) {
        r.x = fmaf(g0.x, p0.x, fmaf(-g0.y, p0.y, fmaf(g1.x, p1.x, fmaf(-g1.y, p1.y, fmaf(g2.x, p2.x, -g2.y * p2.y)))));
        r.y = fmaf(g0.x, p0.y, fmaf(g0.y, p0.x, fmaf(g1.x, p1.y, fmaf(g1.y, p1.x, fmaf(g2.x, p2.y, g2.y * p2.x)))));
    } else {
        static_assert(std::is_same<C, double2>::value, "double-float: the overload below");
        r.x = fma(g0.x, p0.x, fma(-g0.y, p0.y, fma(g1.x, p1.x, fma(-g1.y, p1.y, fma(g2.x, p2.x, -g2.y * p2.y)))));
        r.y = fma(g0.x, p0.y, fma(g0.y, p0.x, fma(g1.x, p1.y, fma(g1.y, p1.x, fma(g2.x, p2.y, g2.y * p2.x)))));
    }
    return r;
}
// a * conj(b)
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
    C r;
    r.x = a.x * b.x + a.y * b.y;
    r.y = a.y * b.x - a.x * b.y;
    return r;
}
template <typename C, typename S> __host__ __device__ __forceinline__ C cscale(C a, S s) { C r; r.x = a.x * s; r.y = a.y * s; return r; }
template <typename C> __host__ __device__ __forceinline__ C cmake(typename real_of<C>::type re, typename real_of<C>::type im) {
    C r;
    r.x = re;
    r.y = im;
    return r;
}
template <typename C> __host__ __device__ __forceinline__ C czero() { return cmake<C>(0, 0); }
template <typename C> __host__ __device__ __forceinline__ C cneg(C a) { C r; r.x = -a.x; r.y = -a.y; return r; }
template <typename C> __host__ __device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }
// multiply by +i (sgn > 0) or -i (sgn < 0)
template <int SGN, typename C> __host__ __device__ __forceinline__ C cmul_i(C a) {
    C r;
    if (SGN > 0) { r.x = -a.y; r.y = a.x; }
    else         { r.x = a.y;  r.y = -a.x; }
    return r;
}
template <typename D, typename S> __host__ __device__ __forceinline__ D ccast(S a) {
    D r;
    r.x = static_cast<typename real_of<D>::type>(a.x);
    r.y = static_cast<typename real_of<D>::type>(a.y);
    return r;
}

// ---- packed FP32 pairs ---------------------------------------------------------
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f32x2 pk(float2 a) { return pk(a.x, a.y); }
__device__ __forceinline__ float2 upk(f32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// ---- complex double-float ------------------------------------------------------
// The operations of dfl on both parts at once, in the same order: the same bits.
// (Products summed before they are normalized, 38 operations in place of 50 for
// a complex product, were 20 % faster still and 8 % less accurate.)
// a * b for pairs, n = -b.hi
__device__ __forceinline__ cdfl df_mul(f32x2 ah, f32x2 al, f32x2 bh, f32x2 bl, f32x2 nbh) {
    const f32x2 n = mul2(ah, nbh), e = fma2(al, bh, fma2(ah, bl, fma2(ah, bh, n))), h = sub2(e, n);
    cdfl r;
    r.hi = upk(h);
    r.lo = upk(sub2(e, add2(h, n)));
    return r;
}
__device__ __forceinline__ cdfl cadd(cdfl a, cdfl b) {
    const f32x2 ah = pk(a.hi), bh = pk(b.hi), s = add2(ah, bh), bb = sub2(s, ah);
    const f32x2 e = add2(add2(sub2(ah, sub2(s, bb)), sub2(bh, bb)), add2(pk(a.lo), pk(b.lo))), h = add2(s, e);
    cdfl r;
    r.hi = upk(h);
    r.lo = upk(sub2(e, sub2(h, s)));
    return r;
}
__device__ __forceinline__ cdfl csub(cdfl a, cdfl b) {
    const f32x2 ah = pk(a.hi), bh = pk(b.hi), s = sub2(ah, bh), bb = sub2(s, ah);
    const f32x2 e = add2(sub2(sub2(ah, sub2(s, bb)), add2(bh, bb)), sub2(pk(a.lo), pk(b.lo))), h = add2(s, e);
    cdfl r;
    r.hi = upk(h);
    r.lo = upk(sub2(e, sub2(h, s)));
    return r;
}
// re(a) b + im(a) (i b)
__device__ __forceinline__ cdfl cmul(cdfl a, cdfl b) {
    const cdfl p = df_mul(pk(a.hi.x, a.hi.x), pk(a.lo.x, a.lo.x), pk(b.hi), pk(b.lo), pk(-b.hi.x, -b.hi.y));
    const cdfl q = df_mul(pk(a.hi.y, a.hi.y), pk(a.lo.y, a.lo.y), pk(-b.hi.y, b.hi.x), pk(-b.lo.y, b.lo.x),
                          pk(b.hi.y, -b.hi.x));
    return cadd(p, q);
}
__device__ __forceinline__ cdfl cscale(cdfl a, dfl s) {
    return df_mul(pk(a.hi), pk(a.lo), pk(s.hi, s.hi), pk(s.lo, s.lo), pk(-s.hi, -s.hi));
}
__device__ __forceinline__ cdfl cdot3(cdfl g0, cdfl p0, cdfl g1, cdfl p1, cdfl g2, cdfl p2) {
    return cadd(cadd(cmul(g0, p0), cmul(g1, p1)), cmul(g2, p2));
}
__host__ __device__ __forceinline__ cdfl cneg(cdfl a) {
    cdfl r;
    r.hi = make_float2(-a.hi.x, -a.hi.y);
    r.lo = make_float2(-a.lo.x, -a.lo.y);
    return r;
}
__host__ __device__ __forceinline__ cdfl cconj(cdfl a) {
    a.hi.y = -a.hi.y;
    a.lo.y = -a.lo.y;
    return a;
}
template <> __host__ __device__ __forceinline__ cdfl cmake<cdfl>(dfl re, dfl im) { return make_cdfl(re, im); }
template <int SGN> __device__ __forceinline__ cdfl cmul_i(cdfl a) {
    cdfl r;
    r.hi = SGN > 0 ? make_float2(-a.hi.y, a.hi.x) : make_float2(a.hi.y, -a.hi.x);
    r.lo = SGN > 0 ? make_float2(-a.lo.y, a.lo.x) : make_float2(a.lo.y, -a.lo.x);
    return r;
}
template <> __host__ __device__ __forceinline__ cdfl ccast<cdfl, double2>(double2 a) {
    return make_cdfl(dfl(a.x), dfl(a.y));
}
template <> __host__ __device__ __forceinline__ double2 ccast<double2, cdfl>(cdfl a) {
    return make_double2((double)a.hi.x + (double)a.lo.x, (double)a.hi.y + (double)a.lo.y);
}

// Index of site s in the per-RHS 1/alpha and weight tables: its composition
// code, or, with per-site materials (no composition array), s + 1.
__device__ __forceinline__ int table_index(const uint8_t* __restrict__ comp_of, int64_t s) {
    return comp_of != nullptr ? (int)comp_of[s] : (int)(s + 1);
}

// How the x-inverse pass finds a site's 1/alpha (a template parameter of its
// kernels): the scalar of the site's composition, row c of its composition's
// tensor, or the scalar of the site itself (per-site materials).
enum { kDiagComp = 0, kDiagTensor = 1, kDiagSite = 2 };
template <int DIAG, typename C>
__device__ __forceinline__ C diag_entry(const C* __restrict__ br, const uint8_t* __restrict__ comp_of, int64_t s,
                                        int c) {
    if constexpr (DIAG == kDiagTensor) return br[comp_of[s] * 3 + c];
    else if constexpr (DIAG == kDiagSite) return br[s + 1];
    else return br[comp_of[s]];
}

}  // namespace dda
