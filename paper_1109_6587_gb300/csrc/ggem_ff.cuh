// Double-float arithmetic: a value is the unevaluated sum hi + lo of two
// floats, about 48 significant bits.  GB300 issues FP64 at 1/64 of its FP32
// rate, so FP64-accurate pair sums run faster in float pairs than in doubles.
// Built on Knuth's two-sum and the exact product of a fused multiply-add
// (a*b - fl(a*b) = fma(a, b, -fl(a*b))), after Dekker (1971) and Hida, Li and
// Bailey (2001).  Sums and products are left unnormalised -- lo up to a few
// 2^-23 of the largest term, not half an ulp of hi -- as every operation takes
// its operands' lo parts to first order anyway; the dropped lo * lo products
// and the rounding of the lo parts are about 2^-46 of the largest term.  The
// rounded products are __fmul_rn: a plain multiply could be contracted with the
// addition that follows it, whose error term then counts twice.  The
// renormalising steps (3 operations each) are kept where a value is compared,
// accumulated over many pairs or fed to the reciprocal square root.
#pragma once

struct ff {
    float hi, lo;
};

// FP64 -> pair (setup code only: it issues FP64 instructions)
__device__ __forceinline__ ff ff_from_double(double x) {
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - (double)h)};
}
__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.hi + (double)a.lo; }

// s + e = a + b exactly (Knuth)
__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
// s + e = a + b exactly when |a| >= |b| (Dekker)
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ ff ff_norm(ff a) { return fast_two_sum(a.hi, a.lo); }
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = __fmul_rn(a.hi, b.hi);
    return {p, fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, fmaf(a.hi, b.hi, -p)))};
}
__device__ __forceinline__ ff ff_sqr(ff a) {
    const float p = __fmul_rn(a.hi, a.hi);
    return {p, fmaf(a.hi, a.lo + a.lo, fmaf(a.hi, a.hi, -p))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    const ff s = two_sum(a.hi, b.hi);
    return {s.hi, (a.lo + b.lo) + s.lo};
}
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, {-b.hi, -b.lo}); }
// a + b + c of products
__device__ __forceinline__ ff ff_sum3(ff a, ff b, ff c) {
    const ff s = two_sum(a.hi, b.hi), t = two_sum(s.hi, c.hi);
    return {t.hi, ((a.lo + b.lo) + (c.lo + s.lo)) + t.lo};
}
__device__ __forceinline__ ff ff_dot(const ff* a, const ff* b) {
    return ff_sum3(ff_mul(a[0], b[0]), ff_mul(a[1], b[1]), ff_mul(a[2], b[2]));
}
// acc += p, acc normalised
__device__ __forceinline__ void ff_acc(ff& acc, ff p) { acc = ff_norm(ff_add(acc, p)); }

// y = 1/sqrt(x), x > 0 normalised: the hardware estimate e (about 2^-22.4
// relative) corrected by e r (1/2 + 3 r / 8), r = 1 - x e^2.  r and the
// correction are themselves kept in pairs and y is normalised: 1/r^5 takes five
// times y's error (8e-16 rms this way, 5e-15 with r and the correction as single
// floats: 3 times the error of the pair terms for 12 operations of about 420).
__device__ __forceinline__ ff ff_rsqrt(ff x) {
    float e;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x.hi));
    const float p = __fmul_rn(e, e), pl = fmaf(e, e, -p);
    const float t = __fmul_rn(x.hi, p), t0 = fmaf(x.hi, p, -t);
    const float tl = fmaf(x.lo, p, __fmul_rn(x.hi, pl));
    const ff a = fast_two_sum(1.0f - t, -t0);        // 1 - t is exact
    const float r = a.hi - tl;
    const float rl = ((a.hi - r) - tl) + a.lo;
    const float h = 0.5f * r, c = __fmul_rn(e, h);
    const float cl = fmaf(e, 0.5f * rl, fmaf(0.75f * c, r, fmaf(e, h, -c)));
    ff y = fast_two_sum(e, c);
    y.lo += cl;
    return y;
}
