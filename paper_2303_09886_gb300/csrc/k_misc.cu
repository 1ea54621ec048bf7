// The call's first kernel (FP64 delay/phase table, lost-data flags, history
// tail) and the phase-1 dispatch over tap counts.
#include "fe_device.cuh"
#include "fe_internal.cuh"

namespace fe {

template <int T, int CAP>
cudaError_t launch_phase1_n1(int N1, int W, const GroupArgs<Phase1Params, CAP> *g, cudaStream_t s, bool pdl);

// g = nullptr: only the kernel's shared-memory size is set
template <int CAP>
static cudaError_t launch_phase1_t(int T, int N1, int W, const GroupArgs<Phase1Params, CAP> *g, cudaStream_t s,
                                   bool pdl) {
    switch (T) {
        case 1: return launch_phase1_n1<1, CAP>(N1, W, g, s, pdl);
        case 2: return launch_phase1_n1<2, CAP>(N1, W, g, s, pdl);
        case 4: return launch_phase1_n1<4, CAP>(N1, W, g, s, pdl);
        case 8: return launch_phase1_n1<8, CAP>(N1, W, g, s, pdl);
        case 16: return launch_phase1_n1<16, CAP>(N1, W, g, s, pdl);
        case 32: return launch_phase1_n1<32, CAP>(N1, W, g, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_phase1_group(int T, int N1, const Phase1Group &g, cudaStream_t s) {
    return launch_phase1_t<kMaxGroup>(T, N1, g.p[0].W, &g, s, false);
}

cudaError_t prepare_phase1(int T, int N1, int W) {
    const cudaError_t e = launch_phase1_t<1>(T, N1, W, nullptr, nullptr, false);
    return e != cudaSuccess ? e : launch_phase1_t<kMaxGroup>(T, N1, W, nullptr, nullptr, false);
}

// blocks of a launch: (t2 blocks, tiles of p.rows spectra, streams)
int phase1_blocks(int N1, const Phase1Params &p, int n_streams, int *gx, int *gy) {
    (void)N1;
    *gx = p.N2 / p.W;
    *gy = (p.q_count + p.rows - 1) / p.rows;
    return *gx * *gy * n_streams;
}

cudaError_t launch_phase1(int T, int N1, const Phase1Params &p, int n_streams, cudaStream_t s, bool pdl) {
    GroupArgs<Phase1Params, 1> g;
    g.p[0] = p;
    g.start[0] = 0;
    g.start[1] = phase1_blocks(N1, p, n_streams, &g.gx, &g.aux[0]);
    g.n = 1;
    return launch_phase1_t<1>(T, N1, p.W, &g, s, pdl);
}

// Spectra per phase-1 CTA. More rows share the T - 1 lead-in rows, the weights
// and the twiddles; fewer give more CTAs. Costs in rows: a filtered row 1, a
// lead-in row about 0.3 of it, a CTA's start-up and DFT latency about 8; the
// launch takes ceil(CTAs / resident CTAs) rounds of that.
int phase1_rows(int T, int N1, int N2, int q_count, int n_streams) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        sms = 148;
    const int W = phase1_W(N1, N2);
    const long long slots = 512LL / p1_threads(N1 * W) * sms, cols = (long long)(N2 / W) * n_streams;
    int best = kP1Block;
    double best_cost = -1.0;
    for (int rows : {128, 64, 32, 16, 8}) {
        const long long ctas = cols * ((q_count + rows - 1) / rows);
        const int used = rows < q_count ? rows : q_count;
        const double cost = (double)((ctas + slots - 1) / slots) * (used + 0.3 * (T - 1) + 8.0);
        if (best_cost < 0.0 || cost < best_cost) {
            best = rows;
            best_cost = cost;
        }
    }
    return best;
}

// Delay model of a stream (Sec. 2.1 steps 2 and 4, Sec. 3.3) at the spectrum
// with timestamp t0 = N m, with the last segment whose t_apply <= t0 (segment
// 0 before all of them):
//   d = d0 + rate (t0 - t_ref),  c = floor(d + 1/2),  delta = d - c.
// FP64 with explicit round-to-nearest operations (no contraction), so the
// host-side range check in the API computes the very same c.
struct DelayAt {
    long long c;   // clamped into [min_delay, max_delay]
    bool clamped;
    double delta, dt;
    int seg;
};
__device__ __forceinline__ DelayAt delay_at(const DelayTableParams &p, int st, long long t0) {
    const DelaySeg *sg = p.seg + (long long)st * kMaxSeg;
    const int ns = p.nseg[st];
    DelayAt r;
    r.seg = 0;
    for (int k = 1; k < ns; k++)
        if (sg[k].t_apply <= t0) r.seg = k;
    r.dt = (double)(t0 - sg[r.seg].t_ref);
    const double d = __dadd_rn(sg[r.seg].d0, __dmul_rn(sg[r.seg].rate, r.dt));
    const double c = floor(__dadd_rn(d, 0.5));
    r.delta = __dadd_rn(d, -c);
    r.c = (long long)c;
    r.clamped = r.c < p.min_delay || r.c > p.max_delay;   // unreachable after the host check
    if (r.clamped) r.c = r.c < p.min_delay ? p.min_delay : p.max_delay;
    return r;
}

// Entry e of the delay table: c, delta and phi = phi0 + phi_rate (t0 - t_ref),
// reduced to phi/pi in [-1, 1] before the single rounding to FP32.
__device__ __forceinline__ void delay_entry(const DelayTableParams &p, long long e) {
    if (e >= (long long)p.n_streams * p.M) return;
    const int st = (int)(e / p.M), q = (int)(e % p.M);
    const long long t0 = (long long)p.N * (p.m0 + q);
    const DelayAt a = delay_at(p, st, t0);
    const DelaySeg &sg = p.seg[(long long)st * kMaxSeg + a.seg];
    const double phi = __dadd_rn(sg.phi0, __dmul_rn(sg.phi_rate, a.dt));
    const double u = phi * 0.31830988618379067154;       // phi / pi
    const double red = u - 2.0 * rint(0.5 * u);          // in [-1, 1]
    if (a.clamped) atomicExch(p.err, 1);
    p.ctab[e] = (int)a.c;
    p.ftab[e] = make_float2((float)a.delta, (float)red);
    // the previous spectrum's coarse delay, recomputed the same way
    if (p.cchg) p.cchg[e] = (unsigned char)(q > 0 && delay_at(p, st, t0 - p.N).c != a.c);
    if (p.g_tapply) {
        const long long *ta = p.g_tapply + (long long)st * kMaxGainSeg;
        int g = 0;
        for (int k = 0; k < p.n_gsets[st]; k++)
            if (ta[k] <= t0) g = k;
        p.gsel[e] = (unsigned char)g;
    }
}

// History tail: word w of the new history (32-bit words; every stream's bytes
// are a multiple of 4 and 4-byte aligned): the last tail_bytes bytes of [old
// history | chunk] of every stream (the chunk-overlap region of Sec. 3.1, kept
// resident on the device instead of copying the next chunk's prefix). The
// words of a history fit 32 bits; those of a chunk do not (the down-converter
// takes up to 2^34 samples, 5.4e9 words of a stream).
__device__ __forceinline__ void tail_words(const uint8_t *hist_in, const uint8_t *chunk, uint8_t *hist_out,
                                           long long tail_bytes, long long chunk_bytes, int n_streams, int block,
                                           int n_blocks) {
    const unsigned tw = (unsigned)(tail_bytes >> 2);
    const long long cw = chunk_bytes >> 2;
    const uint32_t *hi = reinterpret_cast<const uint32_t *>(hist_in), *ch = reinterpret_cast<const uint32_t *>(chunk);
    uint32_t *ho = reinterpret_cast<uint32_t *>(hist_out);
    for (int st = 0; st < n_streams; st++) {
        // word w comes from word w + cw of [history | chunk]: history words below keep, chunk words from it on
        const unsigned keep = cw < (long long)tw ? tw - (unsigned)cw : 0u;
        const uint32_t *h = hi + (long long)st * tw + (keep ? cw : 0), *c = ch + (long long)st * cw + (cw - (long long)tw);
        uint32_t *o = ho + (long long)st * tw;
        for (unsigned w = (unsigned)block * blockDim.x + threadIdx.x; w < tw; w += (unsigned)n_blocks * blockDim.x)
            o[w] = w < keep ? h[w] : c[w];
    }
}

// Lost data (Sec. 3.7). Block x < n_ant * n_heaps_out: output heap h of
// antenna a; its threads check the spectra of the heap in both polarisations:
// spectrum m (coarse delay c) reads [N m - c, N m - c + N T), usable iff every
// heap that window touches was received (history heaps from hv_in, chunk
// heaps from valid). The heap is transmitted (flag 1) iff all are usable.
// The last block writes the received flags of the HV heaps before the end
// of this chunk, for the next call.
__device__ __forceinline__ void lost_block(const LostDataParams &p, const DelayTableParams &d, int block) {
    const int n_out = (p.M + p.S - 1) / p.S;
    const long long hist_first = p.heap0 - p.HV;   // heap of hv_in[0]
    auto received = [&](int stream, long long h) -> bool {
        if (h >= p.heap0) {
            const long long i = h - p.heap0;
            if (i >= p.chunk_heaps) return false;
            return p.valid ? p.valid[(long long)stream * p.chunk_heaps + i] != 0 : true;
        }
        const long long i = h - hist_first;
        return i >= 0 && p.hv_in[(long long)stream * p.HV + i] != 0;
    };
    if (block < p.n_ant * n_out) {
        if (!p.heap_flags) return;
        const int a = block / n_out, h = block % n_out;
        const int q0 = h * p.S, cnt = min(p.S, p.M - q0);
        int ok = 1;
        for (int e = threadIdx.x; e < 2 * cnt; e += blockDim.x) {
            const int pol = e / cnt, q = q0 + e % cnt, stream = 2 * a + pol;
            const long long start = (long long)p.N * (p.m0 + q) - delay_at(d, stream, (long long)p.N * (p.m0 + q)).c;
            const long long end = start + (long long)p.N * p.T - 1;
            const long long h0 = start >= 0 ? start / kHeapSamples : -((-start + kHeapSamples - 1) / kHeapSamples);
            const long long h1 = end >= 0 ? end / kHeapSamples : -((-end + kHeapSamples - 1) / kHeapSamples);
            for (long long hh = h0; hh <= h1 && ok; hh++)
                if (!received(stream, hh)) ok = 0;
        }
        ok = __syncthreads_and(ok);
        if (threadIdx.x == 0) p.heap_flags[(long long)a * n_out + h] = (unsigned char)ok;
        return;
    }
    // history heaps of the next call: heap (heap0 + chunk_heaps) - HV + i
    for (int e = threadIdx.x; e < 2 * p.n_ant * p.HV; e += blockDim.x) {
        const int stream = e / p.HV, i = e % p.HV;
        const long long hh = p.heap0 + p.chunk_heaps - p.HV + i;
        p.hv_out[(long long)stream * p.HV + i] = received(stream, hh) ? 1 : 0;
    }
}

// One call's (CAP = 1) or those of a batch's members in one grid.
template <int CAP>
__global__ void __launch_bounds__(256) k_prologue(const __grid_constant__ GroupArgs<PrologueParams, CAP> ga) {
    pdl_release();
    const int m = CAP == 1 ? 0 : group_member(ga, (int)blockIdx.x);
    const PrologueParams &p = ga.p[m];
    const int b = (int)blockIdx.x - (CAP == 1 ? 0 : ga.start[m]);
    if (b < p.b_delay) {
        delay_entry(p.d, (long long)b * 256 + threadIdx.x);
    } else if (b < p.b_delay + p.b_lost) {
        lost_block(p.l, p.d, b - p.b_delay);
    } else {
        tail_words(p.hist_in, p.chunk, p.hist_out, p.tail_bytes, p.chunk_bytes, p.n_streams, b - p.b_delay - p.b_lost,
                   p.b_tail);
    }
}

// blocks of a history tail: about 8 words per thread over all streams, at most 4 blocks per SM
static int tail_blocks(long long tail_bytes, int n_streams) {
    const long long per = (tail_bytes / 4 + 255) / 256, want = (per * n_streams + 7) / 8;
    return (int)(want < 1 ? 1 : want > per ? (per < 608 ? per : 608) : want > 608 ? 608 : want);
}

template <int CAP>
static cudaError_t launch_prologue_n(GroupArgs<PrologueParams, CAP> &g, cudaStream_t s) {
    int total = 0;
    for (int m = 0; m < g.n; m++) {
        PrologueParams &p = g.p[m];
        p.b_delay = (int)(((long long)p.d.n_streams * p.d.M + 255) / 256);
        p.b_lost = p.lost ? p.l.n_ant * ((p.l.M + p.l.S - 1) / p.l.S) + 1 : 0;
        p.b_tail = p.tail_bytes > 0 ? tail_blocks(p.tail_bytes, p.n_streams) : 0;
        g.start[m] = total;
        total += p.b_delay + p.b_lost + p.b_tail;
    }
    g.start[g.n] = total;
    return total ? launch_kernel(k_prologue<CAP>, dim3((unsigned)total), 256u, 0, s, false, g) : cudaSuccess;
}

cudaError_t launch_prologue(const PrologueParams &p, cudaStream_t s) {
    GroupArgs<PrologueParams, 1> g;
    g.p[0] = p;
    g.n = 1;
    return launch_prologue_n(g, s);
}

cudaError_t launch_prologue_group(PrologueGroup &g, cudaStream_t s) { return launch_prologue_n(g, s); }

// The history tail by itself (the down-converter's).
__global__ void __launch_bounds__(256) k_tail_update(const uint8_t *hist_in, const uint8_t *chunk, uint8_t *hist_out,
                                                     long long tail_bytes, long long chunk_bytes, int n_streams) {
    tail_words(hist_in, chunk, hist_out, tail_bytes, chunk_bytes, n_streams, (int)blockIdx.x, (int)gridDim.x);
}

cudaError_t launch_tail_update(const uint8_t *hist_in, const uint8_t *chunk, uint8_t *hist_out, long long hist_bytes,
                               long long chunk_bytes, int n_streams, cudaStream_t s) {
    return launch_kernel(k_tail_update, dim3((unsigned)tail_blocks(hist_bytes, n_streams)), 256u, 0, s, false, hist_in, chunk,
                         hist_out, hist_bytes, chunk_bytes, n_streams);
}

}  // namespace fe
