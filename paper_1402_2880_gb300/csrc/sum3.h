// A sum of floats that carries more than FP64 does, off the FP64 pipe (two
// lanes per clock and SM).
#pragma once

namespace sscf {

// s + e = a + b exactly, s the rounded sum
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// Three floats, each what the roundings of the one before dropped. Only the
// third rounds: an addition is off by 2^-24 of it, about 2^-70 of the largest
// sum so far. An infinite sum stays infinite (its remainders are NaN).
struct Sum3 {
    float h, l, m;
    __device__ __forceinline__ void add(float v) {
        float e, d;
        two_sum(h, v, h, e);
        two_sum(l, e, l, d);
        m = __fadd_rn(m, d);
    }
    __device__ __forceinline__ void add(float2 v) {
        float d;
        add(v.x);
        two_sum(l, v.y, l, d);
        m = __fadd_rn(m, d);
    }
    __device__ __forceinline__ void add(const Sum3& o) {
        add(make_float2(o.h, o.l));
        m = __fadd_rn(m, o.m);
    }
    __device__ __forceinline__ double value() const {
        return isfinite(h) ? ((double)h + (double)l) + (double)m : (double)h;
    }
};

// Two of them in packed arithmetic. A term must not come from a packed product:
// the compiler fuses one with the additions here (their results then differ in
// the last bits), which it does with no product of __fmul_rn.
struct Sum3x2 {
    float2 h, l, m;
    __device__ __forceinline__ static float2 sub(float2 a, float2 b) {
        return __fadd2_rn(a, make_float2(-b.x, -b.y));
    }
    __device__ __forceinline__ static void two_sums(float2 a, float2 b, float2& s, float2& e) {
        s = __fadd2_rn(a, b);
        const float2 t = sub(s, a);
        e = __fadd2_rn(sub(a, sub(s, t)), sub(b, t));
    }
    __device__ __forceinline__ void add(float2 v) {
        float2 e, d;
        two_sums(h, v, h, e);
        two_sums(l, e, l, d);
        m = __fadd2_rn(m, d);
    }
};

}  // namespace sscf
