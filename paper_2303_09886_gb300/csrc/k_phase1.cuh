// Phase 1 of the fused F-engine: 10-bit unpack, coarse delay, PFB FIR
// (Eq. 1) and the first stage of the four-step real DFT.
//
// Four-step split of the N-point DFT of one spectrum's filtered samples g:
//   t = N2 t1 + t2, k = k1 + N1 k2,
//   X[k1 + N1 k2] = sum_t2 exp(-2 pi i k2 t2 / N2) * B[k1][t2],
//   B[k1][t2]     = exp(-2 pi i k1 t2 / N) * sum_t1 g[N2 t1 + t2] exp(-2 pi i k1 t1 / N1).
// g is real, so only k1 in [0, N1/2] is kept (the rest is the conjugate).
//
// One CTA owns p.rows consecutive output spectra (up to kP1Blocks blocks of
// 32) x C = N1 * W columns {N2 t1 + t2 : t1 < N1, t2 in [t2_0, t2_0 + W)} of
// one (antenna, pol) stream. Output row r is the FIR over input rows r ..
// r + T - 1 (input row i holds the samples of spectrum q0 + i; Eq. 1's
// w[t + N j] weights row r + j); every PFB window uses one coarse delay
// (Sec. 3.3), so consecutive blocks of one delay are filtered as one span,
// whose register ring of input rows runs on from block to block (the T - 1
// rows of lead-in are read and decoded once per span).
//
// Each thread owns two adjacent FIR columns. A warp copies the packed bytes
// of its own 64 columns into its own shared-memory ring (cp.async, a few
// groups of 8 rows ahead; only warp barriers in the FIR), and a thread
// decodes a row's two samples from two 32-bit words: one byte permute puts
// the four bytes holding both fields in bit order, and each field goes into
// the mantissa of a float in place. The FIR keeps T + 1 input rows in a
// register ring and emits output rows in pairs (packed FP32x2 FMAs). g goes
// to shared memory as pairs of output rows, and for each (row pair, t2) the
// real N1-point DFT over t1 of both rows runs in packed registers, is
// multiplied by the twiddle and stored as the second stage reads it: the two
// spectra of a pair side by side, (re, re, im, im). For N1 = 64 two threads
// share the transform (the pair would not fit in one's registers): 1024
// spectra of 32768 channels, 16 taps: 0.385 ms and 0.234 in the second stage,
// against 0.40 and 0.25 with one row per thread and spectra stored apart.
//
// What bounds it: the FP32 pipe (a packed instruction takes two of its
// cycles; 43 % active) and the dependent chains of 16 warps per SM, the
// occupancy that 128 registers allow. Measured on 4 antennas x 2 x 2^25
// samples, 8192 channels, 16 taps: 0.402 ms and 26 thread-instructions per
// sample, against 0.484 ms and 38 with a thread per pair of columns 256 apart
// (four byte loads per row), tiles of 32 rows and one row per DFT thread. The
// intermediate is stored with the streaming hint: plain stores take 0.50 ms,
// because the lines written push the packed rows out of L2.
// 32 taps, 8192 channels, 8.4 M samples: 0.074 ms against 0.176 (the second
// sweep's rows are decoded again; 32 to 96 bytes spill where one sweep of 32
// taps spilled 2 to 4 KB).
#pragma once
#include <algorithm>

#include "fe_device.cuh"
#include "fe_internal.cuh"

namespace fe {

template <int T, int N1, int W>
struct P1Shape {
    static constexpr int C = N1 * W;         // FIR columns per tile
    static constexpr int CW = C < 64 ? C : 64;      // columns of one warp
    static constexpr int NW = C / CW;        // warps that filter
    static constexpr int THREADS = p1_threads(C), CTAS = 512 / THREADS;   // resident per SM (128 registers each)
    static constexpr int NS = CW / W;        // segments (t1 values) of one warp
    // floats per row pair of g (N1 = 64: a warp of the DFT reads 4 row pairs at a time, half a warp on
    // 32 banks)
    static constexpr int GROW = 2 * C + (N1 == 64 ? 16 : 0);
    static constexpr int G_FLOATS = (kP1Block / 2) * GROW;
    // Staged input: the packed bytes of each (input row, t1 segment of W
    // columns) are copied into the ring from the segment's first byte rounded
    // down to ALIGN, SEG bytes (the W samples' bytes plus up to 15 in front
    // and the second byte of the last field), SG rows per commit group,
    // NGRING groups in the ring.
    static constexpr int SEG = (15 + (5 * (W - 1) + 3) / 4 + 2 + 15) / 16 * 16;
    static constexpr int SG = 8;
    static constexpr int NGRING = (N1 * SEG <= 1024) ? 4 : 2;
    static constexpr int RING = NGRING * SG;
    static constexpr unsigned ALIGN = C == 32 ? 8u : 16u;   // rows of N = 32 samples are 40 bytes apart
    static constexpr int ROWB = NS * SEG;    // staged bytes per row of one warp
    static constexpr int STAGE_BYTES = NW * RING * ROWB + 16;   // (a row's last 32-bit word may reach past it)
    static constexpr int TW_FLOATS = (N1 / 2 + 1) * W * 4;
    // T = 32 goes over a block in two sweeps of 16 taps, the second adding to g (the weights and the
    // window of 32 taps would not fit in registers; the sums are the two halves of T = 32 as it is)
    static constexpr int TT = T > 16 ? 16 : T;
    static constexpr int SWEEPS = T / TT;
    static constexpr int PRE = (TT - 1 + SG - 1) / SG * SG;  // lead-in rows in whole groups
    static constexpr int PAD = PRE - (TT - 1);               // rows of the first group that are not read
    // A span runs over several blocks where the ring holds a block's lead-in
    // (the last rows of the block before) next to two groups in flight; else
    // every block is a span.
    static constexpr bool CARRY = SWEEPS == 1 && RING == kP1Block && PRE + 2 * SG <= RING;
    static constexpr int AHEAD = CARRY ? 2 : NGRING - 1;     // groups in flight
    static constexpr size_t SMEM = sizeof(float) * (size_t)(G_FLOATS + TW_FLOATS) + STAGE_BYTES;
};

__device__ __forceinline__ void p1_cp_async16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void p1_cp_async4(unsigned dst, const void *src, unsigned bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void p1_cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void p1_cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The history and the chunk of a stream as one run of packed bytes: byte V
// counts from the first history byte. Sample s (from the first history
// sample; H is a multiple of 4) starts in byte 5 s / 4 at bit 2 (s mod 4).
__device__ __forceinline__ unsigned p1_byte(unsigned s) { return (s >> 2) * 5u + ((s & 3u) * 5u >> 2); }

// One warp's staged input: lane e of copy k of a group takes the 16 bytes
// e + 32 k of the group's 8 rows x ROWB bytes.
template <int T, int N1, int W>
struct P1Stage {
    using S = P1Shape<T, N1, W>;
    static constexpr int CPR = S::ROWB / 16;                    // copies per row
    static constexpr int PER = (S::SG * CPR + 31) / 32;         // copies per lane and group
    const uint8_t *chunk0;    // chunk - hist_bytes: byte V of the chunk part
    const uint8_t *hist;
    unsigned hb, total;       // history bytes, history + chunk bytes
    unsigned ring;            // the warp's ring (shared-memory address)
    unsigned RB;              // bytes between rows
    unsigned V[PER];          // source byte of each copy, in the next group
    int rows_left;            // rows not yet copied, counted from the next group's first row
    bool fast;                // every copy of the span lies in the chunk, 16-byte aligned

    // span of n rows (lead-in included) whose row 0, column 0 is sample rel0
    __device__ __forceinline__ void start(unsigned rel0, int N2, int warp, int n) {
        const int lane = threadIdx.x & 31;
        rows_left = n + S::PAD;
#pragma unroll
        for (int k = 0; k < PER; k++) {
            const int e = lane + 32 * k, row = e / CPR, seg = (e % CPR) / (S::SEG / 16), c16 = e % (S::SEG / 16);
            const unsigned b = p1_byte(rel0 + (unsigned)(N2 * (S::NS * warp + seg)));
            // rounded down relative to the chunk's first byte, whichever side of it
            V[k] = (((b - hb) & ~(S::ALIGN - 1u)) + hb) + RB * (unsigned)(row - S::PAD) + 16u * (unsigned)c16;
        }
        // 16-byte copies when the warp's first byte (row 0, segment 0) lies in the chunk and its last
        // copy (row n - 1, segment NS - 1) ends inside it
        const unsigned first = p1_byte(rel0 + (unsigned)(N2 * S::NS * warp));
        const unsigned last = p1_byte(rel0 + (unsigned)(N2 * (S::NS * warp + S::NS - 1)));
        const unsigned end = ((last - hb) & ~(S::ALIGN - 1u)) + hb + RB * (unsigned)(n - 1) + (unsigned)S::SEG;
        fast = S::ALIGN == 16u && ((uintptr_t)(chunk0 + hb) & 15u) == 0u && first >= hb && end <= total;
    }

    // Copies the next group into its ring slots (slot of its first row: v0 mod
    // RING) and commits it; rows before the first (PAD) or past the last are
    // left out. An empty group past the end keeps the group count in step.
    __device__ __forceinline__ void group(int v0, bool first) {
        const int lane = threadIdx.x & 31;
        const unsigned dst = ring + (unsigned)((v0 % S::RING) * S::ROWB);
        const int row_lo = first ? S::PAD : 0;
#pragma unroll
        for (int k = 0; k < PER; k++) {
            const int e = lane + 32 * k, row = e / CPR;
            const bool in = (S::SG * CPR % 32 == 0 || e < S::SG * CPR) && row >= row_lo && row < rows_left;
            if (fast) {
                if (in) p1_cp_async16(dst + 16u * (unsigned)e, chunk0 + V[k]);
            } else if constexpr (N1 == 64) {
                // word by word, the four words of a copy on adjacent lanes: segments of 32 bytes would have an
                // instruction's words on 32 lines (16 taps, 36 spectra of 32768 channels, whose first rows lie in
                // the history: 0.058 -> 0.033 ms; with the longer segments of N1 <= 32 the plain order is the faster)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int el = 8 * i + (lane >> 2), e4 = el + 32 * k, row4 = e4 / CPR;
                    const unsigned v = __shfl_sync(0xFFFFFFFFu, V[k], el) + 4u * (unsigned)(lane & 3);   // below 0 wraps past total
                    if ((S::SG * CPR % 32 == 0 || e4 < S::SG * CPR) && row4 >= row_lo && row4 < rows_left) {
                        const bool ok = v < total;
                        const uint8_t *src = ok && v >= hb ? chunk0 + v : hist + (ok ? v : 0u);
                        p1_cp_async4(dst + 16u * (unsigned)e4 + 4u * (unsigned)(lane & 3), src, ok ? 4u : 0u);
                    }
                }
            } else if (in) {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const unsigned v = V[k] + 4u * (unsigned)i;   // below 0 wraps past total
                    const bool ok = v < total;
                    const uint8_t *src = ok && v >= hb ? chunk0 + v : hist + (ok ? v : 0u);
                    p1_cp_async4(dst + 16u * (unsigned)e + 4u * (unsigned)i, src, ok ? 4u : 0u);
                }
            }
            V[k] += RB * (unsigned)S::SG;
        }
        p1_cp_async_commit();
        rows_left -= S::SG;
    }
};

// Exact float of the 10-bit two's-complement field in the low bits of x:
// (field ^ 512) is the offset-binary value in [0, 1024), placed in the
// mantissa of 2^23 and the bias 2^23 + 512 subtracted (both steps exact).
__device__ __forceinline__ float field10_to_float(unsigned x) {
    return __uint_as_float(((x & 0x3FFu) ^ 0x200u) | 0x4B000000u) - 8389120.0f;
}

// Two adjacent samples of a column pair: the four bytes from the first
// field's first byte on, in bit order, shifted so that the second field is in
// bits 0-9 and the first in bits 10-19.
__device__ __forceinline__ unsigned p1_fields(const uint8_t *s, unsigned sel, unsigned sh) {
    return __byte_perm(*reinterpret_cast<const unsigned *>(s), *reinterpret_cast<const unsigned *>(s + 4), sel) >> sh;
}
// Their values: each field goes into a mantissa in place (2^23 + 1024 f and
// 2^23 + f, f offset binary); one packed FMA takes out the scale and the
// bias, exactly (8192 + f - 8704 and 2^23 + f - 8389120).
__device__ __forceinline__ float2 p1_decode(unsigned v) {
    const float x0 = __uint_as_float((v & 0xFFC00u) ^ 0x4B080000u);
    const float x1 = __uint_as_float((v & 0x3FFu) ^ 0x4B000200u);
    return __ffma2_rn(make_float2(x0, x1), make_float2(0.0009765625f, 1.0f), make_float2(-8704.0f, -8389120.0f));
}

// Weights of two adjacent columns (volatile: not kept from an earlier read)
__device__ __forceinline__ float2 p1_weights(const float *w) {
    float2 r;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(r.x) : "l"(w));
    asm volatile("ld.global.nc.f32 %0, [%1 + 4];" : "=f"(r.y) : "l"(w));
    return r;
}

// Sample at index s (from the first history sample), or 0 past the received
// samples.
__device__ __forceinline__ float sample10_at(const uint8_t *hist, const uint8_t *chunk, unsigned s, unsigned H,
                                             unsigned HL) {
    if (s >= HL) return 0.0f;
    const bool h = s < H;
    const unsigned u = h ? s : s - H;
    const uint8_t *b = (h ? hist : chunk) + p1_byte(u);
    const unsigned v = __byte_perm((unsigned)__ldg(b), (unsigned)__ldg(b + 1), 0x0004u);   // b[0] << 8 | b[1]
    return field10_to_float(v >> (6u - 2u * (u & 3u)));
}

// Position in g of output row r, tile column c (an even column's pair is
// adjacent: two floats on in a row, or four in a row pair).
template <class S>
__device__ __forceinline__ int p1_gpos(int r, int c) {
    return (r >> 1) * S::GROW + 2 * c + (r & 1);
}

// Output rows (r, r + 1) of a column pair from the ring win of TT + 1 input
// rows (win[i % (TT + 1)] holds input row i), r even: packed FP32x2 FMAs in
// independent chains (each output row's taps in two halves, added at the
// end; a sweep of T = 32 is one half). g0: the thread's column pair in row 0.
// add: the second sweep of T = 32.
template <class S>
__device__ __forceinline__ void p1_fir_pair(int r, const float2 (&win)[S::TT + 1], const float2 (&w2)[S::TT], float *g0,
                                            bool add) {
    constexpr int T = S::TT, TH = (T >= 4 && S::SWEEPS == 1) ? T / 2 : T;
    float2 a0 = make_float2(0.0f, 0.0f), a1 = make_float2(0.0f, 0.0f);
    float2 b0 = make_float2(0.0f, 0.0f), b1 = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < TH; j++) {
        a0 = __ffma2_rn(w2[j], win[(r + j) % (T + 1)], a0);
        a1 = __ffma2_rn(w2[j], win[(r + 1 + j) % (T + 1)], a1);
    }
#pragma unroll
    for (int j = TH; j < T; j++) {
        b0 = __ffma2_rn(w2[j], win[(r + j) % (T + 1)], b0);
        b1 = __ffma2_rn(w2[j], win[(r + 1 + j) % (T + 1)], b1);
    }
    float4 o = make_float4(a0.x, a1.x, a0.y, a1.y);
    float4 *g = reinterpret_cast<float4 *>(g0 + (r >> 1) * S::GROW);
    if constexpr (TH < T) {   // scalar sums, straight into the order of the row pair
        o = make_float4(__fadd_rn(a0.x, b0.x), __fadd_rn(a1.x, b1.x), __fadd_rn(a0.y, b0.y),
                        __fadd_rn(a1.y, b1.y));
    } else if (S::SWEEPS > 1 && add) {
        const float4 u = *g;
        o = make_float4(__fadd_rn(u.x, o.x), __fadd_rn(u.y, o.y), __fadd_rn(u.z, o.z), __fadd_rn(u.w, o.w));
    }
    *g = o;
}

// General case of the FIR: a run of output rows [ra, rb) of a block with a
// delay step, or with the window tap wanted; samples checked one by one
// (history / chunk / past the received samples), one row of loads at a time.
// The window tap of output row r is its first input row, i = r. Kept out of
// line so that its registers do not weigh on the common path.
template <int T, class S>
__device__ __noinline__ void p1_fir_general(const Phase1Params &p, const uint8_t *hist, const uint8_t *chunk,
                                            unsigned s0, int ra, int rb, float *g, int c, int stream, int q0,
                                            int t2_0, int t) {
    const int N = p.N;
    const unsigned H = (unsigned)p.H, HL = (unsigned)(p.H + p.L);
    float2 w2[T];
#pragma unroll
    for (int j = 0; j < T; j++)
        w2[j] = make_float2(__ldg(p.w + t2_0 + t + (long long)N * j), __ldg(p.w + t2_0 + t + 1 + (long long)N * j));
    unsigned dep = 0u;
    float2 win[T];
#pragma unroll 1
    for (int row = ra; row < rb + T - 1; row++) {
        const float xa = sample10_at(hist, chunk, s0 + (unsigned)(row * N) + dep, H, HL);
        const float xb = sample10_at(hist, chunk, s0 + 1u + (unsigned)(row * N) + dep, H, HL);
        asm volatile("" : "+r"(dep) : "f"(xa), "f"(xb));
        // shift the window: win[j] holds input row (row - T + 1 + j)
#pragma unroll
        for (int j = 0; j < T - 1; j++) win[j] = win[j + 1];
        win[T - 1] = make_float2(xa, xb);
        if (p.window_tap && row < rb) {
            int *tap = p.window_tap + ((long long)stream * p.M + q0 + row) * N + t2_0;
            tap[t] = (int)xa;
            tap[t + 1] = (int)xb;
        }
        const int r = row - (T - 1);
        if (r >= ra) {
            // the taps' two halves in separate chains, added at the end: the
            // summation order of p1_fir_pair, so that a window gives the same
            // bits whichever path filters it
            constexpr int TH = T >= 4 ? T / 2 : T;
            float2 a = make_float2(0.0f, 0.0f), b = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int j = 0; j < TH; j++) a = __ffma2_rn(w2[j], win[j], a);
#pragma unroll
            for (int j = TH; j < T; j++) b = __ffma2_rn(w2[j], win[j], b);
            if constexpr (TH < T) a = __fadd2_rn(a, b);
            g[p1_gpos<S>(r, c)] = a.x;
            g[p1_gpos<S>(r, c + 1)] = a.y;
        }
    }
}

// X[k1] of a row pair times its twiddle, into the intermediate.
template <int N1, int K1>
__device__ __forceinline__ void p1_store(const cpair &X, const float4 *tp, float4 *out, long long N2, int W) {
    const float4 t = tp[K1 * W];   // (re, re, im, im)
    const cpair tc{make_float2(t.x, t.y), make_float2(t.z, t.w)};
    cpair b;
    if constexpr (K1 == 0 || K1 == N1 / 2) {   // real
        b.x = __fmul2_rn(X.x, tc.x);
        b.y = __fmul2_rn(X.x, tc.y);
    } else {
        b = cmulp<(K1 < N1 / 4)>(X, tc);
    }
    __stcs(out + K1 * N2, make_float4(b.x.x, b.x.y, b.y.x, b.y.y));
}
template <int N1, int W, int K1, int KE>
__device__ __forceinline__ void p1_store_all(const cpair (&X)[N1 / 2 + 1], const float4 *tp, float4 *out, long long N2) {
    if constexpr (K1 <= KE) {
        p1_store<N1, K1>(X[K1], tp, out, N2, W);
        p1_store_all<N1, W, K1 + 1, KE>(X, tp, out, N2);
    }
}

// Bins K .. KE (<= 15) and 32 - K of the 64-point real DFT from the 32-point ones of the even and odd
// samples (rdit_combine2), stored.
template <int W, int K, int KE>
__device__ __forceinline__ void p1_combine64(const cpair *E, const cpair *O, const float4 *tp, float4 *out, long long N2) {
    if constexpr (K <= KE) {
        const cpair t = cmulp_w64<K, (K < 8)>(O[K]), e = E[K];
        cpair X;
        X.x = __fadd2_rn(e.x, t.x);
        X.y = __fadd2_rn(e.y, t.y);
        p1_store<64, K>(X, tp, out, N2, W);
        X.x = sub2(e.x, t.x);
        X.y = sub2(t.y, e.y);
        p1_store<64, 32 - K>(X, tp, out, N2, W);
        p1_combine64<W, K + 1, KE>(E, O, tp, out, N2);
    }
}

// Half of a 64-point real DFT of a row pair: one thread transforms the even samples (H = 0), one in
// another warp the odd ones; they exchange the bins that the other finishes through the slots of g that
// each has read (own: slot of its first sample), and finish K = 0 .. 8 and 9 .. 16 (bins K and 32 - K).
template <int W, int H>
__device__ __forceinline__ void p1_half64(float2 *g, bool act, int bar, const float4 *tp, float4 *out, long long N2) {
    // (a thread without a pair goes along up to its stores: its slots are its own, and their values unused)
    cpair Z[17];
    {
        float2 x[32];
#pragma unroll
        for (int i = 0; i < 32; i++) x[i] = g[(2 * i + H) * W];
        rdft_reg2<32>(x, Z);
    }
    constexpr int S0 = H ? 0 : 9;
#pragma unroll
    for (int i = 0; i < (H ? 9 : 8); i++) {
        g[(4 * i + H) * W] = Z[S0 + i].x;
        if (S0 + i != 0 && S0 + i != 16) g[(4 * i + 2 + H) * W] = Z[S0 + i].y;
    }
    asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
    if (!act) return;
    constexpr int K0 = H ? 9 : 0, R = 1 - H;
    cpair Y[17];   // the other half's
#pragma unroll
    for (int i = 0; i < (H ? 8 : 9); i++) {
        Y[K0 + i].x = g[(4 * i + R) * W];
        if (K0 + i != 0 && K0 + i != 16) Y[K0 + i].y = g[(4 * i + 2 + R) * W];
    }
    cpair X;
    if constexpr (H == 0) {
        X.x = __fadd2_rn(Z[0].x, Y[0].x);
        p1_store<64, 0>(X, tp, out, N2, W);
        X.x = sub2(Z[0].x, Y[0].x);
        p1_store<64, 32>(X, tp, out, N2, W);
        p1_combine64<W, 1, 8>(Z, Y, tp, out, N2);
    } else {
        p1_combine64<W, 9, 15>(Y, Z, tp, out, N2);
        X.x = Y[16].x;
        X.y = neg2(Z[16].x);
        p1_store<64, 16>(X, tp, out, N2, W);
    }
}

// The real N1-point DFT over t1 of the rows of a block in g, the twiddle and
// the store of B[k1][t2]. qa: the block's first row in the intermediate.
template <int N1, int W, class S>
__device__ __forceinline__ void p1_dft(const Phase1Params &p, float *g, const float *tw, int rows, int stream, int qa,
                                       int t2_0) {
    constexpr int H1 = N1 / 2;
    const int N2 = p.N2;
    const long long pair0 = (long long)stream * (p.a_spectra >> 1) + (qa >> 1);
    if constexpr (N1 == 64) {
        // two warps per 32 (row pair, t2): a thread with both halves would need 256 registers
        static_assert((kP1Block / 2) * W * 2 == S::THREADS, "one pass");
        const int wq = (threadIdx.x >> 5) & 3, e = 32 * wq + (threadIdx.x & 31), rp = e / W, w = e % W;
        const int n = ((rows + 1) >> 1) * W;
        if (32 * wq >= n) return;
        float2 *gp = reinterpret_cast<float2 *>(g + rp * S::GROW) + w;
        float4 *out = reinterpret_cast<float4 *>(p.A) + (pair0 + rp) * (H1 + 1) * N2 + t2_0 + w;
        const float4 *tp = reinterpret_cast<const float4 *>(tw) + w;
        if (threadIdx.x < S::THREADS / 2) p1_half64<W, 0>(gp, e < n, 1 + wq, tp, out, N2);
        else p1_half64<W, 1>(gp, e < n, 1 + wq, tp, out, N2);
    } else {
#pragma unroll 1
        for (int e = threadIdx.x; e < ((rows + 1) >> 1) * W; e += S::THREADS) {
            const int rp = e / W, w = e % W;
            const float2 *gp = reinterpret_cast<const float2 *>(g + rp * S::GROW) + w;
            float2 x[N1];
#pragma unroll
            for (int t1 = 0; t1 < N1; t1++) x[t1] = gp[t1 * W];
            cpair X[H1 + 1];
            rdft_reg2<N1>(x, X);
            p1_store_all<N1, W, 0, H1>(X, reinterpret_cast<const float4 *>(tw) + w,
                                       reinterpret_cast<float4 *>(p.A) + (pair0 + rp) * (H1 + 1) * N2 + t2_0 + w, N2);
        }
    }
}

// One tile per CTA; the tiles of one plan's launch (CAP = 1) or of several
// plans' (same T, N1, W) in one grid: member m owns the blocks [start[m],
// start[m + 1]), decomposed into the (t2 block, spectrum tile, stream) of its
// own launch.
template <int T, int N1, int W, int CAP>
__global__ void __launch_bounds__(P1Shape<T, N1, W>::THREADS, P1Shape<T, N1, W>::CTAS) k_phase1(const __grid_constant__ GroupArgs<Phase1Params, CAP> ga) {
    using S = P1Shape<T, N1, W>;
    extern __shared__ __align__(16) float gs[];   // g, the twiddles, the staged input
    __shared__ int c_sm[kP1Block];
    float *tw = gs + S::G_FLOATS;
    uint8_t *stg = reinterpret_cast<uint8_t *>(tw + S::TW_FLOATS);

    const int m = CAP == 1 ? 0 : group_member(ga, (int)blockIdx.x);
    const Phase1Params &p = ga.p[m];
    const int blk = (int)blockIdx.x - (CAP == 1 ? 0 : ga.start[m]), gy = ga.aux[m];
    const int t2_0 = (blk % ga.gx) * W, tile = (blk / ga.gx) % gy, stream = blk / (ga.gx * gy);
    const int N = p.N, N2 = p.N2;
    const int q0 = p.q_begin + tile * p.rows;
    const int Rv = min(p.rows, p.q_begin + p.q_count - q0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint8_t *chunk = p.chunk + (long long)stream * p.chunk_bytes;
    const uint8_t *hist = p.hist + (long long)stream * p.hist_bytes;
    // sample (from the first history sample) of input row 0, column t = 0, before the delay
    const long long rel_base = (long long)N * (p.m0 + q0) - (p.t_in - p.H) + t2_0;

    // this tile's twiddles exp(-2 pi i k1 t2 / N) (read after the first block's barrier)
    for (int i = threadIdx.x; i < (N1 / 2 + 1) * W; i += S::THREADS) {
        const float2 v = __ldg(p.tw1 + (long long)(i / W) * N2 + t2_0 + i % W);
        reinterpret_cast<float4 *>(tw)[i] = make_float4(v.x, v.x, v.y, v.y);
    }
    pdl_release();
    pdl_wait();

    // the coarse delay of each block (lane i: output row i), and whether its rows share it
    const int nblk = (Rv + kP1Block - 1) / kP1Block;
    int cdl[kP1Blocks];
#pragma unroll
    for (int b = 0; b < kP1Blocks; b++) {
        const int r = b * kP1Block + lane;
        cdl[b] = r < Rv ? ld_dep(p.ctab + (long long)stream * p.M + q0 + r) : 0;
    }

    // this thread's FIR columns (c, c + 1)
    const int c = 2 * threadIdx.x;
    const bool filt = c < S::C, fwarp = warp < S::NW;   // (a tile of 32 columns fills half a warp)
    const int t = N2 * (c / W) + (c % W);   // column offset in a row
    const float *wcol = p.w + t2_0 + (filt ? t : 0);
    P1Stage<T, N1, W> st;
    st.chunk0 = chunk - p.hist_bytes;
    st.hist = hist;
    st.hb = (unsigned)p.hist_bytes;
    st.total = (unsigned)(p.hist_bytes + p.chunk_bytes);
    st.RB = (unsigned)N / 4u * 5u;
    uint8_t *ring = stg + warp * (S::RING * S::ROWB);
    st.ring = (unsigned)__cvta_generic_to_shared(ring);

    int b = 0;
    while (b < nblk) {
        // blocks [b, be) of one delay
        int cd = 0, be = b;
#pragma unroll
        for (int i = 0; i < kP1Blocks; i++) {
            if (i < b || i >= nblk || be != i) continue;
            const int c0 = __shfl_sync(0xffffffffu, cdl[i], 0);
            const bool one = __all_sync(0xffffffffu, i * kP1Block + lane >= Rv || cdl[i] == c0);
            if (i == b) cd = c0;
            if (one && c0 == cd && !p.window_tap && (S::CARRY || i == b)) be = i + 1;
        }
        if (be == b) {
            // a delay step inside the block (or the window tap): run by run, sample by sample
            int cb = 0;
#pragma unroll
            for (int i = 0; i < kP1Blocks; i++)
                if (i == b) cb = cdl[i];
            const int rows = min(kP1Block, Rv - b * kP1Block);
            __syncthreads();   // g and c_sm of the block before have been read
            if (warp == 0) c_sm[lane] = cb;
            __syncthreads();
            const long long rb0 = rel_base + (long long)N * b * kP1Block + t;
            for (int ra = 0; ra < rows;) {
                int rb = ra + 1;
                while (rb < rows && c_sm[rb] == c_sm[ra]) rb++;
                if (filt)
                    p1_fir_general<T, S>(p, hist, chunk, (unsigned)(rb0 - c_sm[ra]), ra, rb, gs, c, stream,
                                         q0 + b * kP1Block, t2_0, t);
                ra = rb;
            }
            __syncthreads();
            p1_dft<N1, W, S>(p, gs, tw, rows, stream, q0 - p.q_begin + b * kP1Block, t2_0);
            b++;
            continue;
        }
        const unsigned rel_b = (unsigned)(rel_base + (long long)N * b * kP1Block - cd);
        const int n_out = min(be * kP1Block, Rv) - b * kP1Block;
        // the thread's bytes in a staged row: two words from the one holding its first byte (a row is a
        // multiple of 4 samples and of ALIGN bytes, so that they are the same in every row and sweep)
        const unsigned sa = rel_b + (unsigned)t, ba = p1_byte(sa);
        const unsigned seg0 = p1_byte(rel_b + (unsigned)(N2 * (c / W)));
        const unsigned o = (unsigned)((c / W) % S::NS) * S::SEG + (ba - (((seg0 - st.hb) & ~(S::ALIGN - 1u)) + st.hb));
        const unsigned sel = 0x0123u + 0x1111u * (o & 3u), sh = 12u - 2u * (sa & 3u);
        const uint8_t *my = ring + (o & ~3u);
        auto row_at = [&](int v) -> unsigned {   // fields of staged row v of the span (its slot is the same in every block)
            return p1_fields(my + (v % S::RING) * S::ROWB, sel, sh);
        };
        // the span's first copies, of the sweep from tap j0 on
        auto begin = [&](int j0, int n) {
            __syncwarp();   // the ring's slots of the span or sweep before have been read
            st.start(rel_b + (unsigned)N * (unsigned)j0, N2, warp, n + S::TT - 1);
            constexpr int FIRST = S::AHEAD + (S::CARRY ? S::PRE / S::SG : 0);
#pragma unroll
            for (int gi = 0; gi < FIRST; gi++) st.group(gi * S::SG, gi == 0);
            if constexpr (S::CARRY) {   // the lead-in
                p1_cp_async_wait<S::AHEAD>();
                __syncwarp();
            }
        };
        if (fwarp && S::CARRY) begin(0, n_out);
        for (; b < be; b++) {
            const int rows = min(kP1Block, Rv - b * kP1Block);
#pragma unroll 1
            for (int j0 = 0; j0 < T; j0 += S::TT) {
                if (fwarp && !S::CARRY) begin(j0, rows);
                // the columns' weights, read again for every block: over a DFT stage they would take 2 T of the
                // registers that it needs
                float2 w2[S::TT];
                if (fwarp) {
#pragma unroll
                    for (int j = 0; j < S::TT; j++) w2[j] = p1_weights(wcol + (long long)N * (j0 + j));
                }
                if (j0 == 0) __syncthreads();   // g of the block before has been read
                if (fwarp) {
                    float2 win[S::TT + 1];
                    // rows 0 .. T - 2: still in the ring from the block before (CARRY), or on their way
                    if constexpr (S::CARRY) {
#pragma unroll
                        for (int i = 0; i < S::TT - 1; i++) win[i] = p1_decode(row_at(S::PAD + i));
                    } else {
#pragma unroll
                        for (int gi = 0; gi < S::PRE / S::SG; gi++) {
                            p1_cp_async_wait<S::AHEAD - 1>();
                            __syncwarp();
                            st.group((gi + S::AHEAD) * S::SG, false);
#pragma unroll
                            for (int i = 0; i < S::SG; i++) {
                                const int v = gi * S::SG + i;
                                if (v >= S::PAD) win[v - S::PAD] = p1_decode(row_at(v));
                            }
                        }
                    }
#pragma unroll
                    for (int gi = 0; gi < kP1Block / S::SG; gi++) {
                        if (gi * S::SG >= rows) break;
                        p1_cp_async_wait<S::AHEAD - 1>();
                        __syncwarp();
                        st.group(S::PRE + (gi + S::AHEAD) * S::SG, false);
#pragma unroll
                        for (int i = 0; i < S::SG; i++) {
                            const int v = S::PRE + gi * S::SG + i, row = v - S::PAD;
                            win[row % (S::TT + 1)] = p1_decode(row_at(v));
                            const int r = gi * S::SG + i - 1;   // the pair (r, r + 1) has its rows r .. r + T
                            if ((i & 1) && (S::C >= 64 || filt))
                                p1_fir_pair<S>(r, win, w2, gs + 2 * c, j0 > 0);
                        }
                    }
                }
            }
            __syncthreads();
            p1_dft<N1, W, S>(p, gs, tw, rows, stream, q0 - p.q_begin + b * kP1Block, t2_0);
        }
        p1_cp_async_wait<0>();
    }
}

// (g = nullptr: only the kernel's shared-memory size is set)
template <int T, int N1, int W, int CAP>
cudaError_t launch_phase1_tw(const GroupArgs<Phase1Params, CAP> *g, cudaStream_t s, bool pdl) {
    using S = P1Shape<T, N1, W>;
    static_assert(kP1Block % S::RING == 0, "a row's ring slot is the same in every block");
    if (!g)
        return cudaFuncSetAttribute(k_phase1<T, N1, W, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    for (int m = 0; m < g->n; m++)
        if (g->p[m].W != W || g->p[m].N2 % W || g->p[m].rows < 1 || g->p[m].rows > kP1Blocks * kP1Block ||
            (g->p[m].rows & 1))
            return cudaErrorInvalidValue;
    if (g->n < 1 || g->start[g->n] < 1) return cudaSuccess;
    return launch_kernel(k_phase1<T, N1, W, CAP>, dim3((unsigned)g->start[g->n]), (unsigned)S::THREADS, S::SMEM, s, pdl, *g);
}

template <int T, int CAP>
cudaError_t launch_phase1_n1(int N1, int W, const GroupArgs<Phase1Params, CAP> *g, cudaStream_t s, bool pdl) {
    switch (N1 * 1000 + W) {
        case 8064: return launch_phase1_tw<T, 8, 64, CAP>(g, s, pdl);
        case 16032: return launch_phase1_tw<T, 16, 32, CAP>(g, s, pdl);
        case 32016: return launch_phase1_tw<T, 32, 16, CAP>(g, s, pdl);
        case 64008: return launch_phase1_tw<T, 64, 8, CAP>(g, s, pdl);
        case 8032: return launch_phase1_tw<T, 8, 32, CAP>(g, s, pdl);
        case 8016: return launch_phase1_tw<T, 8, 16, CAP>(g, s, pdl);
        case 8008: return launch_phase1_tw<T, 8, 8, CAP>(g, s, pdl);
        case 8004: return launch_phase1_tw<T, 8, 4, CAP>(g, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fe
