// Device helpers shared by the libfengine kernels: complex arithmetic, the
// quantiser and an in-register radix-2 FFT.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace fe {

__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// Requantise to an 8-bit Gaussian-integer component (Sec. 2.1 step 6,
// Sec. 3.6): saturate to [-127, 127], round half away from zero. Adding the
// largest float below 1/2 with the sign of t and truncating rounds ties away
// from zero and everything else to nearest for |t| <= 127 (FP32 addition is
// correctly rounded, so t + 0.49999997 reaches the next integer exactly when
// frac(|t|) >= 1/2). This is the rule on the host; the kernels apply it to
// four components at a time, with other steps (quant8x4).
inline int quant8(float x) {
    const float t = fminf(fmaxf(x, -127.0f), 127.0f);
    return (int)(t + copysignf(0.49999997f, t));
}

// quant8 of two complex values as one word of 8-bit cells (re0, im0, re1, im1
// from the low byte up): the sum of value and half in packed adds, a
// truncating conversion, and the saturation at +127 in the 8-bit pack
// (integer pipes; 16 instructions for four components against 20 with four
// conversions to 8 bits).
__device__ __forceinline__ unsigned quant8x4(float2 v0, float2 v1) {
    const float2 a = make_float2(fmaxf(v0.x, -127.0f), fmaxf(v0.y, -127.0f));
    const float2 b = make_float2(fmaxf(v1.x, -127.0f), fmaxf(v1.y, -127.0f));
    const float2 ra = __fadd2_rn(a, make_float2(copysignf(0.49999997f, a.x), copysignf(0.49999997f, a.y)));
    const float2 rb = __fadd2_rn(b, make_float2(copysignf(0.49999997f, b.x), copysignf(0.49999997f, b.y)));
    unsigned hi, r;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"((int)rb.y), "r"((int)rb.x), "r"(0));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"((int)ra.y), "r"((int)ra.x), "r"(hi));
    return r;
}

template <int NN>
__host__ __device__ constexpr int bitrev(int i) {
    int r = 0;
    for (int b = 1; b < NN; b <<= 1) {
        r = (r << 1) | (i & 1);
        i >>= 1;
    }
    return r;
}

// cos(2 pi q / 64) for q in [0, 32] (FP64 values rounded to FP32; the exact
// values 0 and +-1 are written exactly so that multiplications by them fold).
__host__ __device__ constexpr float cos64(int q) {
    constexpr float c[33] = {
        1.0f, 9.951847196e-01f, 9.807852507e-01f, 9.569403529e-01f, 9.238795042e-01f,
        8.819212914e-01f, 8.314695954e-01f, 7.730104327e-01f, 7.071067691e-01f, 6.343932748e-01f,
        5.555702448e-01f, 4.713967443e-01f, 3.826834261e-01f, 2.902846634e-01f, 1.950903237e-01f,
        9.801714122e-02f, 0.0f, -9.801714122e-02f, -1.950903237e-01f, -2.902846634e-01f,
        -3.826834261e-01f, -4.713967443e-01f, -5.555702448e-01f, -6.343932748e-01f, -7.071067691e-01f,
        -7.730104327e-01f, -8.314695954e-01f, -8.819212914e-01f, -9.238795042e-01f, -9.569403529e-01f,
        -9.807852507e-01f, -9.951847196e-01f, -1.0f};
    return c[q];
}

// The in-register transforms are radix-2 decimations in time with every index
// and twiddle a compile-time constant. A real DFT of NN points (bins 0..NN/2 of
// X[k] = sum_t x[t] exp(-2 pi i k t / NN)) takes the half-length DFTs E and O of
// the even and odd samples (both real sequences, so E[NN/2 - k] = conj E[k]):
//   X[k] = E[k] + w^k O[k],  X[NN/2 - k] = conj(E[k] - w^k O[k]),  k <= NN/4,
// w = exp(-2 pi i / NN); w^(NN/4) = -i and the k = 0 terms are real.

// ---- two sequences at a time ----
//
// A cpair holds one complex value of two independent sequences (two spectra):
// x the two real parts, y the two imaginary parts. Every operation is one
// packed FP32x2 instruction for both sequences (round to nearest in each
// half), so a transform of two sequences costs half the instructions per
// sequence wherever the scalar form needs one per component: complex
// products 4 for two instead of 8, and products by -i none (the halves are
// not swapped). Which product of a complex product's component is rounded
// and which is fused is written out, so that the results do not depend on
// how a compiler contracts a * b + c * d.
struct cpair {
    float2 x, y;
};
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("{\n\t.reg .b64 p, q;\n\tmov.b64 p, {%1, %2};\n\tmov.b64 q, {%3, %4};\n\tsub.rn.f32x2 %0, p, q;\n\t}"
        : "=l"(r)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}

// a b with the real part fma(a.x, b.x, -(a.y b.y)); the imaginary part is
// fma(a.y, b.x, a.x b.y) with IMB, else fma(a.x, b.y, a.y b.x)
template <bool IMB>
__device__ __forceinline__ cpair cmulp(cpair a, cpair b) {
    cpair r;
    r.x = __ffma2_rn(a.x, b.x, __fmul2_rn(neg2(a.y), b.y));   // (a negated factor is free, a negated addend is not)
    if constexpr (IMB) r.y = __ffma2_rn(a.y, b.x, __fmul2_rn(a.x, b.y));
    else r.y = __ffma2_rn(a.x, b.y, __fmul2_rn(a.y, b.x));
    return r;
}

// a conj(b): real part fma(a.x, b.x, a.y b.y), imaginary part fma(a.y, b.x, -(a.x b.y))
__device__ __forceinline__ cpair cmulp_conj(cpair a, cpair b) {
    cpair r;
    r.x = __ffma2_rn(a.x, b.x, __fmul2_rn(a.y, b.y));
    r.y = __ffma2_rn(a.y, b.x, __fmul2_rn(neg2(a.x), b.y));
    return r;
}
__device__ __forceinline__ cpair as_cpair(float4 v) { return cpair{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 as_float4(cpair c) { return make_float4(c.x.x, c.x.y, c.y.x, c.y.y); }

// a * exp(-2 pi i Q / 64) for a compile-time Q (not 0 or 16): signs go with the
// variable factors, where they are free, so that the constants are the seven
// cosines in (0, 1) and stay in registers
template <int Q, bool IMB>
__device__ __forceinline__ cpair cmulp_w64(cpair a) {
    static_assert(Q > 0 && Q < 32 && Q != 16, "twiddle index");
    constexpr float c = cos64(Q < 16 ? Q : 32 - Q), s = cos64(Q < 16 ? 16 - Q : Q - 16);   // |cos|, sin
    const float2 xc = Q < 16 ? a.x : neg2(a.x), yc = Q < 16 ? a.y : neg2(a.y);
    cpair r;
    r.x = __ffma2_rn(xc, dup2(c), __fmul2_rn(a.y, dup2(s)));
    if constexpr (IMB) r.y = __ffma2_rn(yc, dup2(c), __fmul2_rn(neg2(a.x), dup2(s)));
    else r.y = __ffma2_rn(neg2(a.x), dup2(s), __fmul2_rn(yc, dup2(c)));
    return r;
}

// A load of what an earlier kernel of the call wrote (programmatic launches: after pdl_wait()). Not __ldg, whose
// loads a compiler may move above the wait, as loads of memory that nothing writes while the kernel runs.
template <class V>
__device__ __forceinline__ V ld_dep(const V *p) {
    return *p;
}

namespace detail {

template <int NN, int K>
__device__ __forceinline__ void dit_combine2(cpair (&z)[NN], const cpair (&e)[NN / 2], const cpair (&o)[NN / 2]) {
    if constexpr (K < NN / 2) {
        constexpr int Q = K * (64 / NN);
        if constexpr (Q == 16) {   // times -i
            z[K].x = __fadd2_rn(e[K].x, o[K].y);
            z[K].y = sub2(e[K].y, o[K].x);
            z[K + NN / 2].x = sub2(e[K].x, o[K].y);
            z[K + NN / 2].y = __fadd2_rn(e[K].y, o[K].x);
        } else {
            cpair t = o[K];
            if constexpr (Q != 0) t = cmulp_w64<Q, Q < 16 && Q != 8>(o[K]);
            z[K].x = __fadd2_rn(e[K].x, t.x);
            z[K].y = __fadd2_rn(e[K].y, t.y);
            z[K + NN / 2].x = sub2(e[K].x, t.x);
            z[K + NN / 2].y = sub2(e[K].y, t.y);
        }
        dit_combine2<NN, K + 1>(z, e, o);
    }
}

template <int NN, int K>
__device__ __forceinline__ void rdit_combine2(cpair (&X)[NN / 2 + 1], const cpair (&E)[NN / 4 + 1],
                                              const cpair (&O)[NN / 4 + 1]) {
    if constexpr (K < NN / 4) {
        constexpr int Q = K * (64 / NN);
        const cpair t = cmulp_w64<Q, Q < 8>(O[K]);
        X[K].x = __fadd2_rn(E[K].x, t.x);
        X[K].y = __fadd2_rn(E[K].y, t.y);
        X[NN / 2 - K].x = sub2(E[K].x, t.x);
        X[NN / 2 - K].y = sub2(t.y, E[K].y);
        rdit_combine2<NN, K + 1>(X, E, O);
    }
}

}  // namespace detail

// Real DFTs of two sequences (x[t]: sample t of both), NN = 2, 4, ..., 32.
template <int NN>
__device__ __forceinline__ void rdft_reg2(const float2 (&x)[NN], cpair (&X)[NN / 2 + 1]) {
    if constexpr (NN == 2) {
        X[0].x = __fadd2_rn(x[0], x[1]);
        X[1].x = sub2(x[0], x[1]);
        X[0].y = X[1].y = dup2(0.0f);
    } else {
        constexpr int H = NN / 2, Q = NN / 4;
        float2 xe[H], xo[H];
#pragma unroll
        for (int t = 0; t < H; t++) {
            xe[t] = x[2 * t];
            xo[t] = x[2 * t + 1];
        }
        cpair E[Q + 1], O[Q + 1];
        rdft_reg2<H>(xe, E);
        rdft_reg2<H>(xo, O);
        X[0].x = __fadd2_rn(E[0].x, O[0].x);
        X[H].x = sub2(E[0].x, O[0].x);
        X[0].y = X[H].y = dup2(0.0f);
        detail::rdit_combine2<NN, 1>(X, E, O);
        X[Q].x = E[Q].x;
        X[Q].y = neg2(O[Q].x);
    }
}

// In-register NN-point complex DFTs of two sequences (NN = 1, 2, 4, ..., 64),
// natural order in and out: recursive radix-2 decimation in time, every index
// and twiddle a compile-time constant.
template <int NN>
__device__ __forceinline__ void fft_regc2(cpair (&z)[NN]) {
    if constexpr (NN > 1) {
        cpair e[NN / 2], o[NN / 2];
#pragma unroll
        for (int t = 0; t < NN / 2; t++) {
            e[t] = z[2 * t];
            o[t] = z[2 * t + 1];
        }
        fft_regc2<NN / 2>(e);
        fft_regc2<NN / 2>(o);
        detail::dit_combine2<NN, 0>(z, e, o);
    }
}

// The member of a grouped launch (GroupArgs) that owns block b: the last m
// with start[m] <= b (binary search over the n members' first blocks).
template <class G>
__device__ __forceinline__ int group_member(const G &g, int b) {
    int lo = 0, hi = g.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.start[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

}  // namespace fe
