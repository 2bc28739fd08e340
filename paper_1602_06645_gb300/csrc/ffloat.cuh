// Float-float ("double-single") arithmetic: a value is the unevaluated sum
// hi + lo of two binary32 numbers, about 48 significant bits.  Built from the
// error-free transformations of Knuth (TwoSum: a + b = s + e exactly) and
// Dekker (FastTwoSum, for |a| >= |b|), with the product error taken by one
// fused multiply-add (a * b = p + fmaf(a, b, -p) exactly, Ogita, Rump and
// Oishi 2005).  Correct only without contraction or reassociation of the
// written operations: the library is compiled with --fmad=false and no
// fast-math.
#pragma once

namespace tsdf {

struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff fast_two_sum(float a, float b) {  // |a| >= |b| (or a == 0)
    const float s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}

__device__ __forceinline__ ff two_prod(float a, float b) {
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
    const ff s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}

__device__ __forceinline__ ff ff_add(ff a, float b) {
    const ff s = two_sum(a.hi, b);
    return fast_two_sum(s.hi, s.lo + a.lo);
}

__device__ __forceinline__ ff ff_mul(ff a, float b) {
    const ff p = two_prod(a.hi, b);
    return fast_two_sum(p.hi, fmaf(a.lo, b, p.lo));
}

// y = R x + t for one row r of a binary32 3x3 R and t, x in float-float.
__device__ __forceinline__ ff ff_row(const float* R, float t, const ff x[3]) {
    ff acc = ff_mul(x[0], R[0]);
    acc = ff_add(acc, ff_mul(x[1], R[1]));
    acc = ff_add(acc, ff_mul(x[2], R[2]));
    return ff_add(acc, t);
}

// a / b to float-float accuracy: q = hi(a) / hi(b) corrected once by the
// residual a - q b (computed in float-float).
__device__ __forceinline__ ff ff_div(ff a, ff b) {
    const float q = __fdiv_rn(a.hi, b.hi);
    const ff qb = two_prod(q, b.hi);
    const ff r = ff_add(a, ff{-qb.hi, -fmaf(q, b.lo, qb.lo)});
    return fast_two_sum(q, __fdiv_rn(r.hi, b.hi));
}

// A sum of binary32 terms as three binary32 numbers: the running sum, the sum
// of its rounding errors, and the sum of that sum's.  Both additions are
// error-free (TwoSum), so only the third component rounds: the total carries
// about 70 bits, more than a binary64 sum of the same terms, without the
// binary64 pipe (some 64 cycles per warp instruction on this GPU).
struct fsum3 {
    float hi, mid, lo;
};

__device__ __forceinline__ void fsum3_add(fsum3& s, float x) {
    const ff a = two_sum(s.hi, x), b = two_sum(s.mid, a.lo);
    s.hi = a.hi;
    s.mid = b.hi;
    s.lo += b.lo;
}

// Adds x y, whose rounding error one fused multiply-add gives exactly.
__device__ __forceinline__ void fsum3_add_product(fsum3& s, float x, float y) {
    const ff p = two_prod(x, y), a = two_sum(s.hi, p.hi), b = two_sum(s.mid, p.lo), c = two_sum(b.hi, a.lo);
    s.hi = a.hi;
    s.mid = c.hi;
    s.lo += b.lo + c.lo;
}

__device__ __forceinline__ fsum3 fsum3_merge(const fsum3& s, const fsum3& t) {
    const ff a = two_sum(s.hi, t.hi), b = two_sum(s.mid, t.mid), c = two_sum(b.hi, a.lo);
    return {a.hi, c.hi, (s.lo + t.lo) + (b.lo + c.lo)};
}

// (An infinite or NaN running sum is the sum: its rounding errors are then NaN.)
__device__ __forceinline__ double fsum3_value(const fsum3& s) {
    return isfinite(s.hi) ? (double)s.hi + ((double)s.mid + (double)s.lo) : (double)s.hi;
}

__device__ __forceinline__ fsum3 fsum3_shfl_xor(const fsum3& s, int lanes) {
    return {__shfl_xor_sync(0xffffffffu, s.hi, lanes), __shfl_xor_sync(0xffffffffu, s.mid, lanes),
            __shfl_xor_sync(0xffffffffu, s.lo, lanes)};
}

}  // namespace tsdf
