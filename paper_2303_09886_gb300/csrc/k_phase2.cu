// Phase 2 of the fused F-engine: the N2-point FFT over t2 of the four-step
// split, then fine-delay rotation and bandpass gain (Sec. 2.1 steps 4-5),
// requantisation (Sec. 2.1 step 6, Sec. 3.6) and the channel-major corner
// turn into heaps (Sec. 2.2, Sec. 3.6).
//
// One CTA owns one first-stage index k1 in [0, N1/2] for R2 consecutive
// spectra of both polarisations of one antenna. The FFT of B[k1][.] gives
// F[k2] = X[k1 + N1 k2]. For k2 < N2/2 that is channel k = k1 + N1 k2
// directly; for k2 >= N2/2 it is a channel above n, whose conjugate is
// channel N - k (the real input's Hermitian symmetry), which belongs to the
// class N1 - k1. Classes k1 = 0 and k1 = N1/2 map onto themselves, so their
// CTAs keep only the lower half. Every channel in [0, n) is written once.
//
// FFT: in-place decimation in frequency, radix 16 while possible, then one
// radix-2/4/8 stage; each thread holds 16 points in registers per stage. The
// result is left in digit-reversed order and read back through the index map
// in the epilogue. Shared memory rows are padded by one complex per 16 so
// that every stage and the epilogue are free of bank conflicts.
//
// Rotation: exp(i phi) exp(-2 pi i delta k / N) for k = k1 + N1 k2 is the
// product of a per-(spectrum, pol) table over the high bits of k2 (with the
// exp(i phi) and k1 factors folded in) and one over the low 5 bits, built
// with sincospif at the start of the CTA.
//
// The CTA writes, for each of its channels, R2 consecutive spectra x 2 pols
// x (re, im) = 4 R2 contiguous bytes of one heap row.
#include <cuda_fp16.h>

#include "fe_device.cuh"
#include "fe_internal.cuh"

namespace fe {

namespace {

constexpr int kP2Threads = 256;

template <int I>
struct P2Int {
    static constexpr int value = I;
};

// exp(-2 pi i q / 16), q = 0..15, as compile-time constants.
__device__ __forceinline__ float2 w16(int q) {
    constexpr float c1 = 0.92387953251128674f, s1 = 0.38268343236508977f, h = 0.70710678118654752f;
    constexpr float re[16] = {1.f, c1, h, s1, 0.f, -s1, -h, -c1, -1.f, -c1, -h, -s1, 0.f, s1, h, c1};
    constexpr float im[16] = {0.f, -s1, -h, -c1, -1.f, -c1, -h, -s1, 0.f, s1, h, c1, 1.f, c1, h, s1};
    return make_float2(re[q], im[q]);
}

// In-register R-point DFT (R = 2, 4, 8, 16), natural order in and out,
// radix-2 decimation in time with compile-time twiddles.
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&v)[R]) {
#pragma unroll
    for (int i = 0; i < R; i++) {
        const int j = bitrev<R>(i);
        if (i < j) {
            float2 t = v[i];
            v[i] = v[j];
            v[j] = t;
        }
    }
#pragma unroll
    for (int len = 2; len <= R; len <<= 1) {
#pragma unroll
        for (int i = 0; i < R; i += len) {
#pragma unroll
            for (int j = 0; j < len / 2; j++) {
                const float2 w = w16(j * (16 / len));
                float2 b = v[i + j + len / 2];
                if (j != 0) b = cmul(b, w);
                const float2 a = v[i + j];
                v[i + j] = cadd(a, b);
                v[i + j + len / 2] = csub(a, b);
            }
        }
    }
}

// padded shared-memory index of element e of a sequence
__device__ __forceinline__ int pad(int e) { return e + (e >> 4); }

template <int N2>
struct P2Shape {
    static constexpr int P = N2 < 16 ? N2 : 16;                   // points per thread per stage
    static constexpr int TPS = N2 / P;                            // threads per sequence
    static constexpr int R2 = phase2_R2_for(N2);                  // spectra per CTA
    static constexpr int LD = N2 + N2 / 16 + 1;                   // padded row stride
    static constexpr int LO = N2 < 32 ? N2 : 32;                  // rotation low table size
    static constexpr int HI = N2 / LO;                            // rotation high table size
};

// One DIF stage of radix R over spans of length Lspan (R divides Lspan).
// Butterfly (block b, j): v[r] = x[b Lspan + j + r Lspan/R]; V = DFT_R(v);
// x[b Lspan + j + k Lspan/R] = V[k] exp(-2 pi i j k / Lspan).
template <int N2, int R, int Lspan>
__device__ __forceinline__ void dif_stage(float2 *buf, int nseq, const float2 *tw) {
    using S = P2Shape<N2>;
    constexpr int PER = S::P / R;                 // butterflies per thread (16 points total)
    constexpr int sub = Lspan / R;
    constexpr int seq_per_round = kP2Threads / S::TPS;
    constexpr int tws = N2 / Lspan;               // twiddle table stride
    for (int s0 = 0; s0 < nseq; s0 += seq_per_round) {
        const int sq = s0 + (int)threadIdx.x / S::TPS;
        const int tl = (int)threadIdx.x % S::TPS;
        if (sq < nseq) {
            float2 *x = buf + sq * S::LD;
#pragma unroll
            for (int u = 0; u < PER; u++) {
                const int bf = tl + u * S::TPS;   // butterfly index in [0, per_seq)
                const int blk = bf / sub, j = bf - blk * sub;
                const int base = blk * Lspan + j;
                // pad(base + r sub) = pad(base) + padc(r sub): (base & 15) + (r sub & 15)
                // never carries into bit 4 (j < sub when sub < 16; r sub & 15 = 0
                // otherwise; base & 15 <= 12 with r < 4 when Lspan < 16)
                float2 *xb = x + pad(base);
                float2 v[R];
#pragma unroll
                for (int r = 0; r < R; r++) v[r] = xb[(r * sub) + ((r * sub) >> 4)];
                dft_reg<R>(v);
                if constexpr (Lspan != R) {
                    const int js = j * tws;
#pragma unroll
                    for (int k = 1; k < R; k++) v[k] = cmul(v[k], __ldg(tw + k * js));
                }
#pragma unroll
                for (int r = 0; r < R; r++) xb[(r * sub) + ((r * sub) >> 4)] = v[r];
            }
        }
    }
    __syncthreads();
}

// All DIF stages: radix 16 while the span allows, then the remaining radix.
template <int N2, int Lspan>
__device__ __forceinline__ void dif_all(float2 *buf, int nseq, const float2 *tw) {
    if constexpr (Lspan >= 16) {
        dif_stage<N2, 16, Lspan>(buf, nseq, tw);
        dif_all<N2, Lspan / 16>(buf, nseq, tw);
    } else if constexpr (Lspan > 1) {
        dif_stage<N2, Lspan, Lspan>(buf, nseq, tw);
    }
}

// Position of F[k2] after the DIF stages (digit reversal of k2 in the radix
// sequence 16, 16, ..., R_last).
template <int N2>
__device__ __forceinline__ int dif_pos(int k2) {
    int p = 0, L = N2, k = k2;
#pragma unroll
    for (int s = 0; s < 12; s++) {
        if (L <= 1) break;
        const int R = L >= 16 ? 16 : L;
        L /= R;
        p += (k % R) * L;
        k /= R;
    }
    return p;
}

}  // namespace

// The tiles of one plan's second stage (CAP = 1) or of several plans' (same
// N2) in one grid.
template <int N2, int IN, int CAP>
__global__ void __launch_bounds__(kP2Threads, 3) k_phase2(const __grid_constant__ GroupArgs<Phase2Params, CAP> ga) {
    const int m = CAP == 1 ? 0 : group_member(ga, (int)blockIdx.x);
    const Phase2Params &p = ga.p[m];
    const int blk = (int)blockIdx.x - (CAP == 1 ? 0 : ga.start[m]), gy = ga.aux[m];
    using S = P2Shape<N2>;
    constexpr int R2 = S::R2, LD = S::LD;
    extern __shared__ float2 sm[];
    float2 *buf = sm;                                  // [2 R2][LD]
    constexpr int HP = S::HI + 1, LP = S::LO + 1;      // padded table rows (no bank conflicts)
    float2 *thi = buf + 2 * R2 * LD;                   // [2 R2][HP]
    float2 *tlo = thi + 2 * R2 * HP;                   // [2 R2][LP]
    float2 *qup = tlo + 2 * R2 * LP;                   // [2 R2] upper-class factor
    long long *rowoff = reinterpret_cast<long long *>(qup + 2 * R2);   // [R2] heap row byte offset
    int *rowstride = reinterpret_cast<int *>(rowoff + R2);             // [R2] bytes per channel row

    const int k1 = blk % ga.gx, ant = blk / (ga.gx * gy);
    const int q0 = p.q_begin + ((blk / ga.gx) % gy) * R2;
    pdl_release();
    pdl_wait();
#include "k_phase2_tile.inc"
}

// ---------------------------------------------------------------------------
// N2 = 256 and 512 (1024 and 2048 channels): the same transform and epilogue on
// pairs of spectra in packed FP32x2 arithmetic, with the roundings of k_phase2
// (the results are the same bits). A thread loads the 16 points of its first
// radix-16 butterfly straight from the intermediate, the only transpose goes
// through shared memory within the sequence's half or whole warp, and the last
// butterfly's outputs are rotated, scaled and quantised in registers; a CTA
// synchronises twice (tables and gains; the staged cells). The corner turn
// stores four spectra, 16 bytes, at a time.
//
// What bounds it: issue (16 warps per SM; rotation tables 15 %, epilogue 45 %
// of the instructions). 16384 spectra, 2 polarisations of 2048 channels: 0.322
// ms against 0.390 with one spectrum per thread, four passes over shared
// memory and 4-byte stores.
template <int N2>
struct P2Pair {
    static constexpr int R2 = phase2_R2_for(N2);       // spectra per CTA (8)
    static constexpr int NP = R2 / 2, NS = 2 * NP;     // pairs per polarisation, pair sequences per CTA
    static constexpr int TPS = N2 / 16, THREADS = NS * TPS;
    static constexpr int SUB = N2 / 16;                // points between a butterfly's
    // transpose rows: 16 blocks of SUB points, padded so that a quarter warp's 16-byte accesses hit 32 banks
    static constexpr int XR = N2 == 256 ? 17 : 34, XS = 16 * XR;
    static constexpr int LO = 32, HI = N2 / 32;        // rotation tables: k2 = 32 a + b
    static constexpr int NG = R2 / 4;                  // groups of four spectra
    static constexpr int PITCH = 2 * N2 + 32 / NG;     // staged words of a (polarisation, group)
    struct Smem {
        union {
            float4 x[NS][XS];
            unsigned stg[2 * NG * PITCH];              // (after the transforms)
        };
        float4 th[NS][HI + 1], tl[NS][LO + 1], qu[NS];
        float2 gain[2][N2];                            // of the first spectrum's gain set, [pol][k2]
    };
    static_assert(R2 == 8 && THREADS <= 256, "a group is four spectra");
};

// dft_reg<16> of two sequences, with its roundings
template <int LEN, int J>
__device__ __forceinline__ void p2_butterflies(cpair (&v)[16]) {
    if constexpr (J < LEN / 2) {
        constexpr int q = J * (16 / LEN);
#pragma unroll
        for (int i = J; i < 16; i += LEN) {
            const cpair a = v[i];
            cpair t = v[i + LEN / 2];
            if constexpr (q == 4) t = cpair{t.y, neg2(t.x)};   // times -i
            else if constexpr (q != 0) t = cmulp_w64<4 * q, (q != 6)>(t);
            v[i] = cpair{__fadd2_rn(a.x, t.x), __fadd2_rn(a.y, t.y)};
            v[i + LEN / 2] = cpair{sub2(a.x, t.x), sub2(a.y, t.y)};
        }
        p2_butterflies<LEN, J + 1>(v);
    }
}
__device__ __forceinline__ void p2_dft16(cpair (&z)[16]) {
    cpair v[16];
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = z[bitrev<16>(i)];
    p2_butterflies<2, 0>(v);
    p2_butterflies<4, 0>(v);
    p2_butterflies<8, 0>(v);
    p2_butterflies<16, 0>(v);
#pragma unroll
    for (int i = 0; i < 16; i++) z[i] = v[i];
}

template <int N2, int IN, int CAP>
__global__ void __launch_bounds__(P2Pair<N2>::THREADS, N2 == 256 ? 4 : 2)
    k_phase2_pairs(const __grid_constant__ GroupArgs<Phase2Params, CAP> ga) {
    using S = P2Pair<N2>;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    typename S::Smem &sm = *reinterpret_cast<typename S::Smem *>(sm_raw);
    const int m = CAP == 1 ? 0 : group_member(ga, (int)blockIdx.x);
    const Phase2Params &p = ga.p[m];
    const int blk = (int)blockIdx.x - (CAP == 1 ? 0 : ga.start[m]), gy = ga.aux[m];
    const int k1 = blk % ga.gx, ant = blk / (ga.gx * gy);
    const int q0 = p.q_begin + ((blk / ga.gx) % gy) * S::R2;
    const int M = p.M, Rv = min(S::R2, p.q_begin + p.q_count - q0);
    const int N1 = p.N1, H1 = N1 / 2, N = p.N, n = N / 2, S_ = p.S;
    const int tid = threadIdx.x, ps = tid / S::TPS, j = tid % S::TPS;
    const int pol = ps / S::NP, pr = ps % S::NP;
    const bool act = 2 * pr < Rv;
    const bool upper = (k1 != 0 && k1 != H1);
    // the gains of the first spectrum's set: before the wait where no kernel of the call selects it
    const unsigned char *gsel = p.gsel ? p.gsel + (long long)(ant * 2) * M + q0 : nullptr;
    auto load_gains = [&] {
        for (int e = tid; e < 2 * N2; e += S::THREADS) {
            const int ge = e / N2, k2 = e % N2, kc = k1 + N1 * k2, k = k2 >= N2 / 2 ? N - kc : kc;
            const int set = gsel ? gsel[(long long)ge * M] : 0;
            const float2 *g = p.gains + ((long long)(ant * 2 + ge) * p.n_gsets_max + set) * n;
            sm.gain[ge][k2] = k < n ? __ldg(g + k) : make_float2(0.f, 0.f);
        }
    };
    if (!gsel) load_gains();
    pdl_release();
    pdl_wait();

    // points j + SUB r of the pair, straight into registers
    cpair z[16];
    {
        const long long row = (long long)(ant * 2 + pol) * p.a_spectra + (q0 - p.q_begin) + 2 * pr;
        if constexpr (IN == kInPairs) {
            const float4 *a = reinterpret_cast<const float4 *>(p.A) + ((row >> 1) * (H1 + 1) + k1) * N2 + j;
#pragma unroll
            for (int r = 0; r < 16; r++) z[r] = as_cpair(act ? a[S::SUB * r] : make_float4(0.f, 0.f, 0.f, 0.f));
        } else {
            const long long o0 = (row * (H1 + 1) + k1) * N2 + j, o1 = o0 + (long long)(H1 + 1) * N2;
#pragma unroll
            for (int r = 0; r < 16; r++) {
                float2 u = make_float2(0.f, 0.f), v = u;
                if (act) {
                    if constexpr (IN == kInHalf) {
                        const uint32_t *h = reinterpret_cast<const uint32_t *>(p.A);
                        const uint32_t hu = h[o0 + S::SUB * r], hv = h[o1 + S::SUB * r];
                        u = __half22float2(*reinterpret_cast<const __half2 *>(&hu));
                        v = __half22float2(*reinterpret_cast<const __half2 *>(&hv));
                    } else {
                        u = p.A[o0 + S::SUB * r];
                        v = p.A[o1 + S::SUB * r];
                    }
                }
                z[r] = cpair{make_float2(u.x, v.x), make_float2(u.y, v.y)};
            }
        }
    }
    // rotation tables (angle/pi = phi/pi - 2 delta k / N, k = k1 + N1 (32 a + b)) and gains, under the loads
    const float inv = 2.0f / (float)N;
    for (int e = tid; e < S::NS * (S::HI + S::LO + 1); e += S::THREADS) {
        const int sq = e % S::NS, which = e / S::NS;
        const int q = min(q0 + 2 * (sq % S::NP), p.q_begin + p.q_count - 1), q1 = min(q + 1, p.q_begin + p.q_count - 1);
        const float2 *f = p.ftab + (long long)(ant * 2 + sq / S::NP) * M;   // (delta, phi / pi)
        const float2 f0 = f[q], f1 = f[q1];
        float s0, c0, s1, c1;
        if (which < S::HI) {
            const float kk = (float)(k1 + N1 * S::LO * which);
            sincospif(f0.y - f0.x * kk * inv, &s0, &c0);
            sincospif(f1.y - f1.x * kk * inv, &s1, &c1);
            const float us = IN == kInHalf ? p.tc_unscale : 1.0f;   // the inverse of the FP16 intermediate's scale
            sm.th[sq][which] = make_float4(c0 * us, c1 * us, s0 * us, s1 * us);
        } else if (which < S::HI + S::LO) {
            const int b = which - S::HI;
            sincospif(-f0.x * (float)(N1 * b) * inv, &s0, &c0);
            sincospif(-f1.x * (float)(N1 * b) * inv, &s1, &c1);
            sm.tl[sq][b] = make_float4(c0, c1, s0, s1);
        } else {   // upper class: Y = G exp(2 i phi - 2 pi i delta) conj(Z)
            sincospif(2.0f * f0.y - 2.0f * f0.x, &s0, &c0);
            sincospif(2.0f * f1.y - 2.0f * f1.x, &s1, &c1);
            sm.qu[sq] = make_float4(c0, c1, s0, s1);
        }
    }
    if (gsel) load_gains();

    // radix 16 over the span, the twiddle, the transpose (within the sequence's half or whole warp)
    float4 *x = sm.x[ps];
    p2_dft16(z);
#pragma unroll
    for (int k = 1; k < 16; k++) {
        const float2 w = __ldg(p.tw2 + k * j);
        z[k] = cmulp<false>(z[k], cpair{dup2(w.x), dup2(w.y)});
    }
#pragma unroll
    for (int k = 0; k < 16; k++) x[k * S::XR + j] = as_float4(z[k]);
    __syncwarp();
    // radix 16 within the blocks: N2 = 256: thread j has block j, F[j + 16 i] in z[i]. N2 = 512: threads
    // 2 b and 2 b + 1 have the even and odd points of block b, then the last radix 2 between them, after
    // which z[i] and z[8 + i] are F[k2] and F[k2 + 256] of k2 = b + 16 i (even) or b + 16 (i + 8) (odd thread)
    if constexpr (N2 == 256) {
#pragma unroll
        for (int r = 0; r < 16; r++) z[r] = as_cpair(x[j * S::XR + r]);
        p2_dft16(z);
    } else {
        const int b = j >> 1, o = j & 1;
#pragma unroll
        for (int r = 0; r < 16; r++) z[r] = as_cpair(x[b * S::XR + o + 2 * r]);
        p2_dft16(z);
#pragma unroll
        for (int k = 1; k < 16; k++) {
            const float2 w = __ldg(p.tw2 + 16 * k * o);
            z[k] = cmulp<false>(z[k], cpair{dup2(w.x), dup2(w.y)});
        }
        const float2 s = dup2(o ? -1.0f : 1.0f), ms = neg2(s);
#pragma unroll
        for (int i = 0; i < 8; i++) {
            float4 own = as_float4(z[i]), snd = as_float4(z[i + 8]);
            if (o) {
                const float4 t = own;
                own = snd;
                snd = t;
            }
            float4 got;
            got.x = __shfl_xor_sync(0xFFFFFFFFu, snd.x, 1);
            got.y = __shfl_xor_sync(0xFFFFFFFFu, snd.y, 1);
            got.z = __shfl_xor_sync(0xFFFFFFFFu, snd.z, 1);
            got.w = __shfl_xor_sync(0xFFFFFFFFu, snd.w, 1);
            const cpair u = as_cpair(own), v = as_cpair(got);
            z[i] = cpair{__fadd2_rn(u.x, v.x), __fadd2_rn(u.y, v.y)};
            // even minus odd (exact products by the sign)
            z[i + 8] = cpair{__ffma2_rn(u.x, s, __fmul2_rn(v.x, ms)), __ffma2_rn(u.y, s, __fmul2_rn(v.y, ms))};
        }
    }
    __syncthreads();   // tables and gains

    // rotate, gain, quantise; a word holds a slot's two spectra of one polarisation
    if (act) {
        const int q = q0 + 2 * pr;
        const bool two = 2 * pr + 1 < Rv;
        const long long st = ant * 2 + pol;
        int ga0 = 0, ga1 = 0, gb = 0;
        if (gsel) {
            gb = gsel[(long long)pol * M];
            ga0 = gsel[(long long)pol * M + 2 * pr];
            ga1 = two ? gsel[(long long)pol * M + 2 * pr + 1] : ga0;
        }
        const bool same = ga0 == gb && ga1 == gb;
        const float2 *g0 = p.gains + (st * p.n_gsets_max + ga0) * n, *g1 = p.gains + (st * p.n_gsets_max + ga1) * n;
        float2 *pre = p.prequant ? p.prequant + (st * M + q) * n : nullptr;
        unsigned *stg = sm.stg + (pol * S::NG + (pr >> 1)) * S::PITCH;
        const int kb = N2 == 256 ? j : (j >> 1) + 128 * (j & 1);   // the thread's first slot
        const cpair l0 = as_cpair(sm.tl[ps][kb % 16]), l1 = as_cpair(sm.tl[ps][kb % 16 + 16]);
        const cpair qu = as_cpair(sm.qu[ps]);
        const int pb = (pr & 1) ^ (N2 == 256 ? 0 : j & 1);
        auto slot = [&](auto ic, auto pc) {
            constexpr int i = decltype(ic)::value;
            constexpr bool up = i >= 8;
            const int k2 = kb + (N2 == 256 ? 16 * i : 16 * (i & 7) + (up ? 256 : 0));
            const int kc = k1 + N1 * k2, k = up ? N - kc : kc;
            const cpair r = cmulp<true>(as_cpair(sm.th[ps][k2 >> 5]), (i & 1) ? l1 : l0);
            const cpair v = cmulp<false>(r, z[i]);
            cpair g;
            if (same) {
                const float2 a = sm.gain[pol][k2];
                g = cpair{dup2(a.x), dup2(a.y)};
            } else {
                const float2 a = __ldg(g0 + k), b = __ldg(g1 + k);
                g = cpair{make_float2(a.x, b.x), make_float2(a.y, b.y)};
            }
            cpair y;
            if constexpr (up) y = cmulp_conj(cmulp<false>(g, qu), v);
            else y = cmulp<(decltype(pc)::value != 0)>(g, v);
            if (pre) {
                pre[k] = make_float2(y.x.x, y.y.x);
                if (two) pre[n + k] = make_float2(y.x.y, y.y.y);
            }
            stg[2 * k2 + pb] = quant8x4(make_float2(y.x.x, y.y.x), make_float2(y.x.y, y.y.y));
        };
        auto slots = [&](auto self, auto ic, auto ec, auto pc) {
            constexpr int i = decltype(ic)::value;
            if constexpr (i < decltype(ec)::value) {
                slot(ic, pc);
                self(self, P2Int<i + 1>{}, ec, pc);
            }
        };
        // (the two polarisations' products with the gain are rounded as k_phase2 rounds its y0 and y1)
        if (pol) slots(slots, P2Int<0>{}, P2Int<8>{}, P2Int<1>{});
        else slots(slots, P2Int<0>{}, P2Int<8>{}, P2Int<0>{});
        if (upper) slots(slots, P2Int<8>{}, P2Int<16>{}, P2Int<0>{});
    }
    __syncthreads();

    // corner turn: a slot's four spectra -> heap row of its channel, one 16-byte store (or two of 8 bytes)
    // where the four share a heap and the row is aligned
    const int g = tid % S::NG, qg = q0 + 4 * g, Rg = min(4, Rv - 4 * g);
    if (Rg <= 0) return;
    const int hp = qg / S_, hs = qg - hp * S_, Sh = min(S_, M - hp * S_);
    int8_t *out = p.out + (long long)ant * M * n * 4, *row0 = out + (long long)hp * S_ * n * 4 + hs * 4;
    const unsigned al = ((unsigned)(uintptr_t)row0 | (unsigned)(Sh * 4)) & 15u;
    const bool one = Rg == 4 && hs + 4 <= Sh;
    int8_t *rp[4];
    int rs[4];
    for (int r = 0, hr = hp, sr = hs; r < 4; r++) {
        rs[r] = min(S_, M - hr * S_) * 4;
        rp[r] = out + (long long)hr * S_ * n * 4 + sr * 4;
        if (++sr == S_) {
            sr = 0;
            hr++;
        }
    }
    const unsigned *w0 = sm.stg + g * S::PITCH, *w1 = w0 + S::NG * S::PITCH;
#pragma unroll 4
    for (int k2 = tid / S::NG; k2 < (upper ? N2 : N2 / 2); k2 += S::THREADS / S::NG) {
        const int kc = k1 + N1 * k2, k = k2 >= N2 / 2 ? N - kc : kc;
        uint2 a = *reinterpret_cast<const uint2 *>(w0 + 2 * k2), b = *reinterpret_cast<const uint2 *>(w1 + 2 * k2);
        if (N2 == 512 && (k2 & 128)) {
            a = make_uint2(a.y, a.x);
            b = make_uint2(b.y, b.x);
        }
        const uint4 v = make_uint4(__byte_perm(a.x, b.x, 0x5410u), __byte_perm(a.x, b.x, 0x7632u),
                                   __byte_perm(a.y, b.y, 0x5410u), __byte_perm(a.y, b.y, 0x7632u));
        if (one && al == 0u) {
            *reinterpret_cast<uint4 *>(row0 + (long long)k * Sh * 4) = v;
        } else if (one && (al & 7u) == 0u) {
            uint2 *o = reinterpret_cast<uint2 *>(row0 + (long long)k * Sh * 4);
            o[0] = make_uint2(v.x, v.y);
            o[1] = make_uint2(v.z, v.w);
        } else {
            const unsigned vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (r < Rg) *reinterpret_cast<unsigned *>(rp[r] + (long long)k * rs[r]) = vv[r];
        }
    }
}

size_t phase2_smem_bytes(int N2, int R2) {
    const int LD = N2 + N2 / 16 + 1;
    const int LO = N2 < 32 ? N2 : 32, HI = N2 / LO;
    return sizeof(float2) * ((size_t)2 * R2 * LD + 2 * R2 * ((HI + 1) + (LO + 1) + 1)) +
           (sizeof(long long) + sizeof(int)) * R2;
}

// the grid for N2 < 1024: (classes k1, tiles of R2 spectra, antennas)
int phase2_blocks(int N2, const Phase2Params &p, int n_ant, int *gx, int *gy) {
    (void)N2;
    *gx = p.N1 / 2 + 1;
    *gy = (p.q_count + p.R2 - 1) / p.R2;
    return *gx * *gy * n_ant;
}

// (g = nullptr: only the kernel's shared-memory size is set)
template <int N2, int IN, int CAP>
static cudaError_t launch_p2(const GroupArgs<Phase2Params, CAP> *g, cudaStream_t s, bool pdl) {
    constexpr int R2 = phase2_R2_for(N2);
    void (*kernel)(GroupArgs<Phase2Params, CAP>) = nullptr;
    size_t smem = 0;
    unsigned threads = 0;
    // On pairs from where it is the faster: N2 = 512 always (8 taps, one antenna: 16 spectra 11.8 against
    // 12.8 us, 16384 spectra 0.322 against 0.390 ms), N2 = 256 from two waves of its CTAs on (2048 spectra
    // 24.5 against 26.6 us, 16384 0.145 against 0.165 ms; 16 spectra 9.8 against 8.7 us, where half the
    // threads per spectrum make a CTA's chain longer and nothing else runs beside it)
    if constexpr (N2 >= 256) {
        kernel = k_phase2_pairs<N2, IN, CAP>;
        smem = sizeof(typename P2Pair<N2>::Smem);
        threads = P2Pair<N2>::THREADS;
        if (!g) {
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess || N2 == 512) return e;
        }
    }
    if constexpr (N2 != 512) {
        if (N2 < 256 || !g || g->start[g->n] < 8 * phase2w_wave()) {
            kernel = k_phase2<N2, IN, CAP>;
            smem = phase2_smem_bytes(N2, R2);
            threads = kP2Threads;
        }
        if (!g) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    for (int m = 0; m < g->n; m++)
        if (g->p[m].R2 != R2 || g->p[m].a_spectra % 2) return cudaErrorInvalidValue;
    if (g->n < 1 || g->start[g->n] < 1) return cudaSuccess;
    return launch_kernel(kernel, dim3((unsigned)g->start[g->n]), threads, smem, s, pdl, *g);
}

template <int N2, int CAP>
static cudaError_t launch_p2_in(int in, const GroupArgs<Phase2Params, CAP> *g, cudaStream_t s, bool pdl) {
    switch (in) {
        case kInPairs: return launch_p2<N2, kInPairs, CAP>(g, s, pdl);
        case kInHalf: return launch_p2<N2, kInHalf, CAP>(g, s, pdl);
        case kInHalfPairs: return cudaErrorInvalidValue;   // N2 = 1024 only
        default: return launch_p2<N2, kInFloat, CAP>(g, s, pdl);
    }
}

template <int CAP>
static cudaError_t launch_p2_n2(int N2, int in, const GroupArgs<Phase2Params, CAP> *g, cudaStream_t s, bool pdl) {
    switch (N2) {
        case 2: return launch_p2_in<2, CAP>(in, g, s, pdl);
        case 4: return launch_p2_in<4, CAP>(in, g, s, pdl);
        case 8: return launch_p2_in<8, CAP>(in, g, s, pdl);
        case 16: return launch_p2_in<16, CAP>(in, g, s, pdl);
        case 32: return launch_p2_in<32, CAP>(in, g, s, pdl);
        case 64: return launch_p2_in<64, CAP>(in, g, s, pdl);
        case 128: return launch_p2_in<128, CAP>(in, g, s, pdl);
        case 256: return launch_p2_in<256, CAP>(in, g, s, pdl);
        case 512: return launch_p2_in<512, CAP>(in, g, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t prepare_phase2(int N2, int in) {
    if (N2 == 1024) return prepare_phase2w(in);
    const cudaError_t e = launch_p2_n2<1>(N2, in, nullptr, nullptr, false);
    return e != cudaSuccess ? e : launch_p2_n2<kMaxGroup>(N2, in, nullptr, nullptr, false);
}

cudaError_t launch_phase2_group(int N2, int in, const Phase2Group &g, cudaStream_t s) {
    return N2 == 1024 ? launch_phase2w_group(in, g, s) : launch_p2_n2(N2, in, &g, s, false);
}

cudaError_t launch_phase2(int N2, const Phase2Params &p, int n_ant, cudaStream_t s, bool pdl) {
    if (N2 == 1024) return launch_phase2w(p, n_ant, s, pdl);   // one warp per pair of 1024-point sequences
    GroupArgs<Phase2Params, 1> g;
    g.p[0] = p;
    g.start[0] = 0;
    g.start[1] = phase2_blocks(N2, p, n_ant, &g.gx, &g.aux[0]);
    g.n = 1;
    return launch_p2_n2(N2, p.in, &g, s, pdl);
}

}  // namespace fe
