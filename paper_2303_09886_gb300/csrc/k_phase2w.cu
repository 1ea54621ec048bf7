// Phase 2 for N2 = 1024: one warp computes the 1024-point FFTs of one
// polarisation of two consecutive spectra in registers, then the fine-delay
// rotation, gain, requantisation and corner turn (Sec. 2.1 steps 4-6,
// Sec. 2.2, Sec. 3.6).
//
// With t2 = 32 a + b and k2 = c + 32 d (a, b, c, d in [0, 32)):
//   Y[c][b]     = sum_a exp(-2 pi i c a / 32) B[32 a + b]
//   Y'[c][b]    = exp(-2 pi i c b / 1024) Y[c][b]
//   F[c + 32 d] = sum_b Y'[c][b] exp(-2 pi i d b / 32).
// The pair's sequences arrive in the warp's shared-memory buffer by bulk copy
// (as (re, re, im, im) per point where phase 1 writes pairs); lane b reads
// B[32 a + b] for every a, does the first 32-point DFT in registers, applies
// the twiddle, and writes Y'[.][b] back into the buffer (rows of 33); after
// that transpose lane c holds Y'[c][.] and does the second 32-point DFT in
// registers, leaving F[c + 32 d] for every d. One shared-memory round trip
// per point instead of one per radix pass, and every arithmetic instruction
// is packed FP32x2 over the two spectra.
//
// A work item is one first-stage class k1 and 4 consecutive spectra of one
// antenna, done by one of the CTA's two groups of four warps: warp w of a
// group takes spectra 2 (w / 2), 2 (w / 2) + 1 and polarisation w % 2. The
// groups take turns over the CTA's contiguous range of items and synchronise
// apart from each other (named barriers), so that one group's staging and
// corner turn run under the other's transforms. A warp's next pair is asked
// for as soon as its buffer has been read, and arrives under the second DFT,
// the epilogue and the corner turn.
//
// What bounds it: latency at 8 warps per SM (a warp holds 128 registers of
// data), 33 % of the issue slots, FP32 pipe 35 % active; memory is not the
// limit (the same time per spectrum with the intermediate in L2). Measured on
// 4 antennas x 2 x 2048 spectra of 8192 channels: 0.449 ms and 25.6 M warp
// instructions per 33.5 M samples, against 0.559 ms and 44.9 M for one warp
// per sequence at 16 warps per SM. Two warps per pair with 16 points per
// thread (16 warps per SM, the input straight into registers) took 0.63 ms:
// the transform's halves then meet in shared memory twice.
//
// Slot k2 is channel k1 + N1 k2 for
// k2 < 512, and for k2 >= 512 (classes k1 = 1 .. N1/2 - 1 only) the conjugate
// of channel N - (k1 + N1 k2).
#include <algorithm>

#include <cuda_fp16.h>

#include "fe_device.cuh"
#include "fe_internal.cuh"
#include "fe_waits.cuh"

namespace fe {

namespace {

constexpr int kWGroups = 2;
constexpr int kWGroupThreads = 128;
constexpr int kWThreads = kWGroupThreads * kWGroups;
constexpr int kWWarps = kWThreads / 32;
constexpr int kWR = 4;        // spectra per work item
constexpr int kWN2 = 1024;
constexpr long long kWaitCycles = 2000000000LL;   // about a second: a bulk copy that has not come by then has failed

// Word (two 16-bit cells: the item's spectra 2 pr, 2 pr + 1) of slot k2 of one
// polarisation in a group's staging buffer: the two words of a slot change
// places with bit 4 of k2, so that the 32 lanes of a store (consecutive k2)
// hit 32 banks.
__device__ __forceinline__ int stg_word(int k2, int pr) { return k2 * 2 + (pr ^ ((k2 >> 4) & 1)); }

__device__ __forceinline__ uint32_t sm_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void group_sync(int grp) {
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kWGroupThreads) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

// A work item is (antenna, class k1, group of kWR consecutive spectra), in
// that order; item -> its fields.
struct WItem {
    int ant, k1, q0;
};
__device__ __forceinline__ WItem witem(const Phase2Params &p, int it, int H1, int G) {
    const int per_ant = (H1 + 1) * G;
    WItem w;
    w.ant = it / per_ant;
    const int rem = it - w.ant * per_ant;
    w.k1 = rem / G;
    w.q0 = p.q_begin + (rem - w.k1 * G) * kWR;
    return w;
}

// (re, re, im, im) of two spectra throughout
struct WSmem {
    float4 buf[kWWarps][32][33];          // per warp: its pair of sequences, then the transpose tile
    float4 tw[32][32];                    // exp(-2 pi i c b / 1024), [c][b]
    float4 gain[2][kWN2];                 // gains of the slots, [pol][k2]
    unsigned stg[kWGroups][2][kWN2 * 2];  // output staging, [group][pol][slot, pair]
    float4 q[kWWarps][32];                // per warp: Q[d]
    unsigned long long full[kWWarps];     // per warp: its pair has arrived
    int seg_end;
    int gave_up;                          // a warp's wait has: the others do not wait to their limits
};

}  // namespace

// Persistent: one CTA per SM (a thread holds 32 points of two spectra: 128
// registers of data), a contiguous range of work items of equal work per CTA.
// The CTAs of one (CAP = 1) or several plans' second stages in one grid:
// member m owns CTAs [start[m], start[m + 1]) and aux[m] antennas. kPre: the
// spectra before quantisation are written as well, by a kernel of its own
// (512 spectra, 2 polarisations of 8192 channels: 125 us, and 173 where the
// one kernel did it in a loop over slots with the points in local memory; with
// the stores in a second copy of the epilogue the plain one took 490 us
// instead of 453 on the workload above).
template <int IN, int CAP, bool kPre>
__global__ void __launch_bounds__(kWThreads, 1) k_phase2w(const __grid_constant__ GroupArgs<Phase2Params, CAP> ga) {
    constexpr bool kPaired = IN == kInPairs || IN == kInHalfPairs, kHalf = IN == kInHalf || IN == kInHalfPairs;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    WSmem &sm = *reinterpret_cast<WSmem *>(smem_raw);
    const int mem = CAP == 1 ? 0 : group_member(ga, (int)blockIdx.x);
    const Phase2Params &p = ga.p[mem];
    const int n_ant = ga.aux[mem];
    const long long cta_b = (int)blockIdx.x - ga.start[mem], cta_nb = ga.start[mem + 1] - ga.start[mem];

    const int M = p.M, N1 = p.N1, H1 = N1 / 2, N = p.N, n = N / 2, S_ = p.S;
    const int G = (p.q_count + kWR - 1) / kWR;
    const int n_items = n_ant * (H1 + 1) * G;
    // Contiguous ranges of equal work: classes k1 = 0 and N1/2 keep only the
    // lower half of their slots (half the epilogue and corner turn), so their
    // items count 4 units against 5 for the others; CTA b takes the items
    // whose work starts in [b W / nb, (b + 1) W / nb) (b = cta_b of nb = cta_nb).
    constexpr int wL = 4, wF = 5;
    const int Wa = G * (2 * wL + (H1 - 1) * wF);   // work of one antenna
    auto first_item = [&](long long x) {          // first item whose work starts at >= x
        const int ant = (int)(x / Wa);
        const int y = (int)(x - (long long)ant * Wa);
        int k1, g;
        if (y < wL * G) {
            k1 = 0;
            g = (y + wL - 1) / wL;
        } else if (y < (wL + (H1 - 1) * wF) * G) {
            const int y1 = y - wL * G;
            k1 = 1 + y1 / (wF * G);
            g = (y1 - (k1 - 1) * wF * G + wF - 1) / wF;
        } else {
            k1 = H1;
            g = (y - (wL + (H1 - 1) * wF) * G + wL - 1) / wL;
        }
        return min(n_items, ant * (H1 + 1) * G + k1 * G + g);
    };
    const long long Wt = (long long)n_ant * Wa;
    const int it0 = first_item(Wt * cta_b / cta_nb), it1 = first_item(Wt * (cta_b + 1) / cta_nb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp >> 2, pr = (warp >> 1) & 1, pol = warp & 1;
    float4(*tile)[33] = sm.buf[warp];
    const uint32_t mbar = sm_addr(&sm.full[warp]);
    if (threadIdx.x == 0) sm.gave_up = 0;   // (read after the first segment's barriers)
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();

    // the fields of the items this group goes through, kept without divisions
    WItem nx = witem(p, it0 + grp, H1, G);
    auto advance = [&](WItem &w) {
        w.q0 += kWGroups * kWR;
        while (w.q0 >= p.q_begin + G * kWR) {
            w.q0 -= G * kWR;
            if (++w.k1 > H1) {
                w.k1 = 0;
                w.ant++;
            }
        }
    };
    // this warp's pair of sequences in item w: their first point, in the units of the layout. The
    // intermediate holds an even number of spectra, so that a pair's second one is there even past the last.
    auto pair_at = [&](const WItem &w) -> long long {
        const long long row = (long long)(w.ant * 2 + pol) * p.a_spectra + (w.q0 - p.q_begin) + 2 * pr;
        return ((kPaired ? row >> 1 : row) * (H1 + 1) + w.k1) * kWN2;
    };
    auto active_in = [&](const WItem &w) { return w.q0 + 2 * pr < p.q_begin + p.q_count; };
    // into its buffer (one lane): one run where phase 1 wrote pairs, else the two sequences behind
    // each other
    auto fetch = [&](const WItem &w) {
        constexpr uint32_t EB = IN == kInPairs ? 16 : IN == kInHalf ? 4 : 8;
        constexpr uint32_t bytes = (kPaired ? 1u : 2u) * EB * kWN2;
        asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(mbar),
                     "r"(bytes)
                     : "memory");
        const char *a = reinterpret_cast<const char *>(p.A) + pair_at(w) * EB;
        bulk_copy(sm_addr(tile), a, EB * kWN2, mbar);
        if constexpr (!kPaired)
            bulk_copy(sm_addr(tile) + EB * kWN2, a + (long long)(H1 + 1) * kWN2 * EB, EB * kWN2, mbar);
    };
    // (delta, phi / pi) of the warp's two spectra, and their gain sets (set 0 without timed gains). The tables'
    // addresses go through the wait below, so that these loads cannot be moved above it; as plain loads they
    // could not be moved past the epilogue's stores either (4 antennas, 8192 channels: 455 - 456 against 451 - 452 us
    // over six alternating runs)
    const float2 *ftab = p.ftab;
    const unsigned char *gtab = p.gsel;
    float2 f0 = make_float2(0.f, 0.f), f1 = f0;
    int gsel = 0;
    auto model = [&](const WItem &w) {
        const long long sq = (long long)(w.ant * 2 + pol) * M;
        const int q = w.q0 + 2 * pr, q1 = min(q + 1, p.q_begin + p.q_count - 1);
        f0 = __ldg(ftab + sq + q);
        f1 = __ldg(ftab + sq + q1);
        if (gtab) gsel = (int)__ldg(gtab + sq + q) | (int)__ldg(gtab + sq + q1) << 8;
    };
    for (int e = threadIdx.x; e < 32 * 32; e += kWThreads) {
        const float2 t = __ldg(p.tw2 + (((e >> 5) * (e & 31)) & (kWN2 - 1)));
        (&sm.tw[0][0])[e] = make_float4(t.x, t.x, t.y, t.y);
    }
    pdl_release();
    pdl_wait();   // phase 1's results, and the delay table's
    asm volatile("" : "+l"(ftab), "+l"(gtab)::"memory");
    // the warp's waits, the same in all its lanes (bounded: fengine_device_status reports one that gave up)
    CopyWait cw;
    long long t0 = 0;   // of the first failed try
    auto here = [&](unsigned parity) -> bool {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity), "r"(20000u)
            : "memory");
        return __all_sync(0xFFFFFFFFu, ok != 0) != 0;
    };
    auto late = [&]() -> bool {
        if (t0 == 0) t0 = clock64();
        return __any_sync(0xFFFFFFFFu, clock64() - t0 > kWaitCycles) != 0;
    };
    auto over = [&]() -> bool {
        if (__any_sync(0xFFFFFFFFu, *(volatile int *)&sm.gave_up != 0)) return true;
        if (!late()) return false;
        if (lane == 0) {
            *(volatile int *)&sm.gave_up = 1;
            if (p.err) atomicExch(p.err, 2);
        }
        return true;
    };
    if (it0 + grp < it1 && active_in(nx)) {
        cw.ask([&] {
            if (lane == 0) fetch(nx);
        });
        model(nx);
    }

    for (int seg = it0; seg < it1;) {
        // [seg, se): items of one class and antenna whose first spectra use the same gain sets
        const WItem ws = witem(p, seg, H1, G);
        const int ant = ws.ant, k1 = ws.k1;
        const int class_end = min(it1, (ant * (H1 + 1) + k1 + 1) * G);
        __syncthreads();   // the gains of the segment before have been read
        if (threadIdx.x == 0) sm.seg_end = class_end;
        int gs0 = 0, gs1 = 0;
        if (p.gsel) {
            const unsigned char *g0 = p.gsel + (long long)(ant * 2) * M, *g1 = g0 + M;
            gs0 = ld_dep(g0 + ws.q0);
            gs1 = ld_dep(g1 + ws.q0);
            __syncthreads();
            for (int i = seg + 1 + threadIdx.x; i < class_end; i += kWThreads) {
                const int q = ws.q0 + (i - seg) * kWR;
                if (ld_dep(g0 + q) != gs0 || ld_dep(g1 + q) != gs1) {
                    atomicMin(&sm.seg_end, i);
                    break;
                }
            }
        }
        for (int e = threadIdx.x; e < 2 * kWN2; e += kWThreads) {
            const int ps = e / kWN2, k2 = e % kWN2;
            const int kc = k1 + N1 * k2;
            const int k = k2 >= kWN2 / 2 ? N - kc : kc;
            const float2 *g = p.gains + ((long long)(ant * 2 + ps) * p.n_gsets_max + (ps ? gs1 : gs0)) * n;
            const float2 v = (k >= 0 && k < n) ? __ldg(g + k) : make_float2(0.f, 0.f);
            sm.gain[ps][k2] = make_float4(v.x, v.x, v.y, v.y);
        }
        __syncthreads();
        const int se = sm.seg_end;
        const bool upper = (k1 != 0 && k1 != H1);
        const int stream = ant * 2 + pol;

        const int first = seg + (grp + kWGroups - (seg - it0) % kWGroups) % kWGroups;
        const int q_first = p.q_begin + (first - (ant * (H1 + 1) + k1) * G) * kWR;
        int hp = q_first / S_, hs = q_first - hp * S_;   // heap and position in it of the item's first spectrum
        for (int it = first; it < se; it += kWGroups) {
            const int q0 = q_first + (it - first) * kWR;
            const int Rv = min(kWR, p.q_begin + p.q_count - q0);
            bool active = 2 * pr < Rv;
            advance(nx);   // the group's next item
            const bool more = it + kWGroups < it1 && active_in(nx);

            // rotation factors of the warp's two sequences, angles over pi:
            //   P[c] = exp(i pi (phi/pi - 2 delta (k1 + N1 c) / N))        (lane c)
            //   Q[d] = exp(-i pi 2 delta 32 N1 d / N),  qu = exp(i pi (2 phi/pi - 2 delta)),
            // so that channel k1 + N1 k2 (k2 = c + 32 d) is P[c] Q[d] F[k2] and the
            // upper-half channel N - (k1 + N1 k2) is qu conj(P[c] Q[d] F[k2]).
            cpair P, Pu;
            {
                const float inv = 2.0f / (float)N;
                // P carries the inverse of the FP16 intermediate's scale (a power of two)
                const float u = kHalf ? p.tc_unscale : 1.0f;
                float s0, c0, s1, c1;
                sincospif(f0.y - f0.x * (float)(k1 + N1 * lane) * inv, &s0, &c0);
                sincospif(f1.y - f1.x * (float)(k1 + N1 * lane) * inv, &s1, &c1);
                P = cpair{make_float2(c0 * u, c1 * u), make_float2(s0 * u, s1 * u)};
                sincospif(-f0.x * (float)(32 * N1 * lane) * inv, &s0, &c0);
                sincospif(-f1.x * (float)(32 * N1 * lane) * inv, &s1, &c1);
                sm.q[warp][lane] = make_float4(c0, c1, s0, s1);
                sincospif(2.0f * f0.y - 2.0f * f0.x, &s0, &c0);
                sincospif(2.0f * f1.y - 2.0f * f1.x, &s1, &c1);
                Pu = cmulp_conj(cpair{make_float2(c0, c1), make_float2(s0, s1)}, P);
            }
            cpair z[32];
            if (active) {   // the pair has arrived
                t0 = 0;
                active = cw.arrived(here, over);
            }
            if (active) {
                const float4 *lin = &tile[0][0];
                if constexpr (IN == kInPairs) {
#pragma unroll
                    for (int a = 0; a < 32; a++) z[a] = as_cpair(lin[32 * a + lane]);
                } else if constexpr (IN == kInHalfPairs) {
                    const uint2 *hp2 = reinterpret_cast<const uint2 *>(lin);
#pragma unroll
                    for (int a = 0; a < 32; a++) {
                        const uint2 v = hp2[32 * a + lane];
                        z[a] = cpair{__half22float2(*reinterpret_cast<const __half2 *>(&v.x)),
                                     __half22float2(*reinterpret_cast<const __half2 *>(&v.y))};
                    }
                } else if constexpr (IN == kInHalf) {
                    const __half2 *hb = reinterpret_cast<const __half2 *>(lin);
#pragma unroll
                    for (int a = 0; a < 32; a++) {
                        const float2 u = __half22float2(hb[32 * a + lane]), v = __half22float2(hb[kWN2 + 32 * a + lane]);
                        z[a] = cpair{make_float2(u.x, v.x), make_float2(u.y, v.y)};
                    }
                } else {
                    const float2 *fb = reinterpret_cast<const float2 *>(lin);
#pragma unroll
                    for (int a = 0; a < 32; a++) {
                        const float2 u = fb[32 * a + lane], v = fb[kWN2 + 32 * a + lane];
                        z[a] = cpair{make_float2(u.x, v.x), make_float2(u.y, v.y)};
                    }
                }
                __syncwarp();
                fft_regc2<32>(z);                                 // z[c] = Y[c][lane]
#pragma unroll
                for (int c = 1; c < 32; c++) z[c] = cmulp<true>(z[c], as_cpair(sm.tw[c][lane]));
#pragma unroll
                for (int c = 0; c < 32; c++) tile[c][lane] = as_float4(z[c]);
                __syncwarp();
#pragma unroll
                for (int b = 0; b < 32; b++) z[b] = as_cpair(tile[lane][b]);
                // the buffer is free again: this warp's accesses before the bulk copy's writes
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            const int gcur = gsel;
            if (more) {
                cw.ask([&] {
                    if (lane == 0) fetch(nx);
                });
                model(nx);
            }
            if (active) fft_regc2<32>(z);                         // z[d] = F[lane + 32 d]
            group_sync(grp);   // the group's corner turn of the item before has read the staging buffer
            if (active) {
                const float4 *qs = sm.q[warp], *gp = sm.gain[pol] + lane;
                unsigned *stg = sm.stg[grp][pol];
                const int q = q0 + 2 * pr, gst = pol ? gs1 : gs0;
                float2 *pre = kPre ? p.prequant + ((long long)stream * M + q) * n : nullptr;
                const bool two = 2 * pr + 1 < Rv;
                auto put = [&](int k2, int k, const cpair &y) {
                    if constexpr (kPre) {
                        pre[k] = make_float2(y.x.x, y.y.x);
                        if (two) pre[n + k] = make_float2(y.x.y, y.y.y);
                    }
                    stg[stg_word(k2, pr)] = quant8x4(make_float2(y.x.x, y.y.x), make_float2(y.x.y, y.y.y));
                };
                if (gcur == (gst | gst << 8)) {
#pragma unroll
                    for (int d = 0; d < 16; d++) {   // channel k1 + N1 k2
                        const int k2 = lane + 32 * d;
                        const cpair r = cmulp<true>(P, as_cpair(qs[d]));
                        put(k2, k1 + N1 * k2, cmulp<false>(as_cpair(gp[32 * d]), cmulp<false>(r, z[d])));
                    }
                    if (upper) {
#pragma unroll
                        for (int d = 16; d < 32; d++) {   // channel N - (k1 + N1 k2)
                            const int k2 = lane + 32 * d;
                            const cpair r = cmulp_conj(Pu, as_cpair(qs[d]));
                            put(k2, N - (k1 + N1 * k2), cmulp<false>(as_cpair(gp[32 * d]), cmulp_conj(r, z[d])));
                        }
                    }
                } else {
                    // the same with the gains of a spectrum whose set is not the segment's (a gain update inside
                    // the item)
                    const float2 *gd0 = p.gains + ((long long)stream * p.n_gsets_max + (gcur & 0xFF)) * n;
                    const float2 *gd1 = p.gains + ((long long)stream * p.n_gsets_max + (gcur >> 8)) * n;
                    cpair zl[32];
#pragma unroll
                    for (int d = 0; d < 32; d++) zl[d] = z[d];
#pragma unroll 1
                    for (int d = 0; d < (upper ? 32 : 16); d++) {
                        const bool up = d >= 16;
                        const int k2 = lane + 32 * d, kc = k1 + N1 * k2, k = up ? N - kc : kc;
                        const cpair qd = as_cpair(qs[d]);
                        const cpair v = up ? cmulp_conj(cmulp_conj(Pu, qd), zl[d]) : cmulp<false>(cmulp<true>(P, qd), zl[d]);
                        const float2 a = __ldg(gd0 + k), b = __ldg(gd1 + k);
                        const cpair y = cmulp<false>(cpair{make_float2(a.x, b.x), make_float2(a.y, b.y)}, v);
                        put(k2, k, y);
                    }
                }
            }
            group_sync(grp);

            // corner turn: slot k2's four spectra -> heap row of its channel, one 16-byte store
            // (or two of 8 bytes) where the four share a heap and the row is aligned
            const int tid = threadIdx.x % kWGroupThreads;
            int8_t *out = p.out + (long long)ant * M * n * 4;
            while (hs >= S_) {
                hs -= S_;
                hp++;
            }
            const int s = hs, Sh = min(S_, M - hp * S_);
            int8_t *row0 = out + (long long)hp * S_ * n * 4 + s * 4;
            const unsigned al = ((unsigned)(uintptr_t)row0 | (unsigned)(Sh * 4)) & 15u;   // low bits of every cell's address
            const bool one = Rv == kWR && s + kWR <= Sh;                                  // all in one heap
            auto corner = [&](auto &&put) {
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if (u >= 2 && !upper) break;
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const int k2 = (tid & 15) | (i << 4) | ((tid >> 4) << 5) | (u << 8);
                        const int kc = k1 + N1 * k2, k = u >= 2 ? N - kc : kc;
                        const uint2 a = *reinterpret_cast<const uint2 *>(&sm.stg[grp][0][2 * k2]);
                        const uint2 b = *reinterpret_cast<const uint2 *>(&sm.stg[grp][1][2 * k2]);
                        const unsigned a0 = i ? a.y : a.x, a1 = i ? a.x : a.y, b0 = i ? b.y : b.x, b1 = i ? b.x : b.y;
                        put(k, make_uint4(__byte_perm(a0, b0, 0x5410u), __byte_perm(a0, b0, 0x7632u),
                                          __byte_perm(a1, b1, 0x5410u), __byte_perm(a1, b1, 0x7632u)));
                    }
                }
            };
            if (one && al == 0u) {
                corner([&](int k, uint4 v) { *reinterpret_cast<uint4 *>(row0 + (long long)k * Sh * 4) = v; });
            } else if (one && (al & 7u) == 0u) {
                corner([&](int k, uint4 v) {
                    uint2 *o = reinterpret_cast<uint2 *>(row0 + (long long)k * Sh * 4);
                    o[0] = make_uint2(v.x, v.y);
                    o[1] = make_uint2(v.z, v.w);
                });
            } else {
                int8_t *rp[kWR];
                int rs[kWR];
                for (int r = 0, hr = hp, sr = s; r < kWR; r++) {
                    rs[r] = min(S_, M - hr * S_) * 4;
                    rp[r] = out + (long long)hr * S_ * n * 4 + sr * 4;
                    if (++sr == S_) {
                        sr = 0;
                        hr++;
                    }
                }
                corner([&](int k, uint4 v) {
                    const unsigned vv[kWR] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int r = 0; r < kWR; r++)
                        if (r < Rv) *reinterpret_cast<unsigned *>(rp[r] + (long long)k * rs[r]) = vv[r];
                });
            }
            hs += kWGroups * kWR;
        }
        seg = se;
    }
    t0 = 0;
    cw.leave(here, late);
}

long long phase2w_items(const Phase2Params &p, int n_ant) {
    return (long long)n_ant * (p.N1 / 2 + 1) * ((p.q_count + kWR - 1) / kWR);
}

int phase2w_wave() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

// (g = nullptr: only the kernel's shared-memory size is set)
template <int IN, int CAP>
static cudaError_t launch_w(const GroupArgs<Phase2Params, CAP> *g, cudaStream_t s, bool pdl) {
    void (*kernel)(GroupArgs<Phase2Params, CAP>) = k_phase2w<IN, CAP, false>;
    if (!g) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WSmem));
        if constexpr (CAP == 1) {
            if (e == cudaSuccess)
                return cudaFuncSetAttribute(k_phase2w<IN, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sizeof(WSmem));
        }
        return e;
    }
    for (int m = 0; m < g->n; m++)
        if (g->p[m].N / g->p[m].N1 != kWN2 || g->p[m].a_spectra % 2 || (CAP > 1 && g->p[m].prequant))
            return cudaErrorInvalidValue;
    if (g->n < 1 || g->start[g->n] < 1) return cudaSuccess;
    if constexpr (CAP == 1) {
        if (g->p[0].prequant) kernel = k_phase2w<IN, 1, true>;
    }
    return launch_kernel(kernel, dim3((unsigned)g->start[g->n]), (unsigned)kWThreads, sizeof(WSmem), s, pdl, *g);
}

template <int CAP>
static cudaError_t launch_w_in(int in, const GroupArgs<Phase2Params, CAP> *g, cudaStream_t s, bool pdl) {
    switch (in) {
        case kInPairs: return launch_w<kInPairs, CAP>(g, s, pdl);
        case kInHalf: return launch_w<kInHalf, CAP>(g, s, pdl);
        case kInHalfPairs: return launch_w<kInHalfPairs, CAP>(g, s, pdl);
        default: return launch_w<kInFloat, CAP>(g, s, pdl);
    }
}

cudaError_t prepare_phase2w(int in) {
    const cudaError_t e = launch_w_in<1>(in, nullptr, nullptr, false);
    return e != cudaSuccess ? e : launch_w_in<kMaxGroup>(in, nullptr, nullptr, false);
}

cudaError_t launch_phase2w_group(int in, const Phase2Group &g, cudaStream_t s) { return launch_w_in(in, &g, s, false); }

cudaError_t launch_phase2w(const Phase2Params &p, int n_ant, cudaStream_t s, bool pdl) {
    const long long items = phase2w_items(p, n_ant);
    if (items <= 0) return cudaSuccess;
    const int wave = phase2w_wave();
    if (wave < 1) return cudaErrorUnknown;
    GroupArgs<Phase2Params, 1> g;
    g.p[0] = p;
    g.start[0] = 0;
    g.start[1] = (int)std::min<long long>(items, wave);
    g.aux[0] = n_ant;
    g.gx = 1;
    g.n = 1;
    return launch_w_in(p.in, &g, s, pdl);
}

}  // namespace fe
