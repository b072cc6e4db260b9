// Entropy/importance misalignment counts (the diagnostic behind Fig. 1b): per prompt,
// the k = floor(pct * T / 100) tokens with the largest and the smallest entropy H and
// importance S, and how many of the high-entropy tokens are among the low-importance
// ones (and the reverse).
//
// CTA b handles prompt b.  A value's key is its order-preserving unsigned image; equal
// values are ordered by index (the lower first).  The four thresholds (the k-th largest and
// k-th smallest of H and of S) are selected together: every pass keeps, for each selection, a
// key interval [lo, lo + 2^shift bins) that holds its threshold, counts the keys of the
// interval in 1024 equal bins (shared-memory histogram), and narrows it to the bin that the
// wanted rank falls into.  The first interval is the span of the prompt's own keys, so
// neighbouring values spread over the bins (a fixed top digit, sign and exponent, would put
// most of a prompt on two or three counters), and a 27-bit span is done in three passes.  When
// only some of the tokens equal to a threshold belong to its group, further passes select the
// index below which they do, in the same way.  A last pass counts the two intersections.
// Integer counts: the result is exact.
//
// What bounds it is latency: each pass is one look at the prompt's keys (those of its first 2048
// tokens in registers, the rest from L1), four barriers and a scan.  While the two intervals of a
// value agree, which they do in the first pass, one histogram serves both: half of the shared
// atomics.  256 prompts of 128 to 4096 tokens: 144 us for 32 passes of 8-bit digits, one selection
// at a time, each scanned by one thread; 23.0 for the passes above with every key re-read and four
// histograms; 17.0 now.  Four prompts of 32768: 234, 127 and 65 us.
#include "estp_internal.cuh"

namespace estp {
namespace {

constexpr int kThreads = 512;
constexpr int kSel = 4;               // top of H, bottom of H, top of S, bottom of S
constexpr int kBins = 1024;
constexpr int kBinBits = 10;
constexpr int kGroup = kThreads / kSel;   // threads that scan one selection's histogram
constexpr int kPerThread = kBins / kGroup;
// Tokens a thread keeps in registers.  256 prompts of up to 4096 tokens 18.8 / 17.0 / 16.6 us and 16
// short ones 10.9 / 8.5 / 9.9 with 1 / 4 / 8.
constexpr int kCached = 4;

// monotone map float -> uint32 (larger float, larger image); inputs are finite, and
// -0 maps with +0 (they are equal values, so their order falls to the index)
__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t u = f == 0.f ? 0u : __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Bits by which an interval of `span` + 1 keys is shifted to fall into kBins bins.
__device__ __forceinline__ int shift_for(uint32_t span) {
    const int bits = 32 - __clz(span);
    return bits > kBinBits ? bits - kBinBits : 0;
}

struct Select {       // one selection's interval and the wanted rank inside it
    uint32_t lo;      // first key of the interval: bins are (key - lo) >> shift
    int shift;
    int rank;         // 1-based, ascending, among the keys of the interval
    int equal;        // keys in the interval (once shift is 0: keys equal to lo)
};

struct Shared {
    uint32_t hist[kSel][kBins];
    int warp_total[kThreads / 32];
    uint32_t lo4[kThreads / 32], hi4[kThreads / 32], lo5[kThreads / 32], hi5[kThreads / 32];
    Select sel[kSel];
    int n_hl, n_lh;
};

// Narrows every selection (those with rank > 0) to a single key.  each(f) calls f(i, kh, ks) for
// this thread's tokens with the keys of H and S; key(s, i, kh, ks) is a token's key in selection
// s, and in(s, i, kh, ks) whether it takes part.  kTwins: the two selections of one value see the
// same keys, so that while their intervals agree one histogram serves both.  All threads call;
// sh.sel is read and written between barriers.
template <bool kTwins, typename Each, typename Key, typename In>
__device__ __forceinline__ void narrow(Shared& sh, Each each, Key key, In in) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = threadIdx.x / kGroup;  // the selection this thread scans
    int shift[kSel];  // -1: done (every round takes kBinBits off, so at most four follow)
#pragma unroll
    for (int s = 0; s < kSel; ++s) shift[s] = sh.sel[s].rank > 0 ? sh.sel[s].shift : -1;
    while ((shift[0] & shift[1] & shift[2] & shift[3]) >= 0) {
        for (int i = threadIdx.x; i < kSel * kBins; i += kThreads) (&sh.hist[0][0])[i] = 0;
        uint32_t lo[kSel];
#pragma unroll
        for (int s = 0; s < kSel; ++s) lo[s] = sh.sel[s].lo;
        const Select mine = sh.sel[grp];
        const bool twin[2] = {kTwins && lo[0] == lo[1] && shift[0] == shift[1],
                              kTwins && lo[2] == lo[3] && shift[2] == shift[3]};
        const int hist_of = twin[grp >> 1] ? grp & ~1 : grp;
        __syncthreads();
        each([&](int i, uint32_t kh, uint32_t ks) {
#pragma unroll
            for (int s = 0; s < kSel; ++s)
                if (shift[s] >= 0 && !((s & 1) && twin[s >> 1]) && in(s, i, kh, ks)) {
                    const uint32_t x = key(s, i, kh, ks), bin = (x - lo[s]) >> shift[s];
                    if (x >= lo[s] && bin < (uint32_t)kBins) atomicAdd(&sh.hist[s][bin], 1u);
                }
        });
        __syncthreads();
        // scan of the selection's bins: kPerThread a thread, its warp, its group's warps
        int cnt[kPerThread], sum = 0;
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            cnt[j] = (int)sh.hist[hist_of][(threadIdx.x % kGroup) * kPerThread + j];
            sum += cnt[j];
        }
        int inc = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += v;
        }
        if (lane == 31) sh.warp_total[warp] = inc;
        __syncthreads();
        int before = inc - sum;
        for (int w = grp * (kGroup / 32); w < warp; ++w) before += sh.warp_total[w];
        // (a closed selection's histogram is empty, so nothing is found for it)
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            if (before < mine.rank && mine.rank <= before + cnt[j]) {
                Select n;
                n.lo = mine.lo + ((uint32_t)((threadIdx.x % kGroup) * kPerThread + j) << mine.shift);
                n.shift = mine.shift > kBinBits ? mine.shift - kBinBits : 0;
                n.rank = mine.rank - before;
                n.equal = cnt[j];
                sh.sel[grp] = n;
            }
            before += cnt[j];
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < kSel; ++s)
            shift[s] = shift[s] > kBinBits ? shift[s] - kBinBits : shift[s] > 0 ? 0 : -1;
    }
}

__global__ void __launch_bounds__(kThreads, 2) misalign_kernel(const float* __restrict__ H,
                                                            const float* __restrict__ S,
                                                            const int32_t* __restrict__ cu, int B,
                                                            int64_t sumT, int pct,
                                                            int32_t* __restrict__ counts,
                                                            int* status) {
    __shared__ Shared sh;
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // cu_seqlens is checked by every CTA the same way; CTA 0 reports
    int bad = 0;
    if (threadIdx.x == 0) bad = cu[0] != 0 || (int64_t)cu[B] != sumT;
    for (int q = threadIdx.x; q < B; q += blockDim.x) bad |= cu[q + 1] < cu[q];
    if (__syncthreads_or(bad)) {
        if (b == 0 && threadIdx.x == 0) report(status, ESTP_ERR_INVALID_ARG);
        return;
    }
    const int64_t t0 = cu[b];
    const int T = cu[b + 1] - cu[b];
    const int k = (int)((int64_t)pct * T / 100);
    if (k == 0) {
        if (threadIdx.x == 0) {
            counts[3 * b] = 0;
            counts[3 * b + 1] = 0;
            counts[3 * b + 2] = 0;
        }
        return;
    }
    const float* h = H + t0;
    const float* s = S + t0;
    // a thread's tokens: the keys of the first kCached stay in registers
    uint32_t ch[kCached], cs[kCached];
#pragma unroll
    for (int j = 0; j < kCached; ++j) {
        const int i = threadIdx.x + j * kThreads;
        ch[j] = i < T ? ordered(h[i]) : 0u;
        cs[j] = i < T ? ordered(s[i]) : 0u;
    }
    auto each = [&](auto f) {
#pragma unroll
        for (int j = 0; j < kCached; ++j) {
            const int i = threadIdx.x + j * kThreads;
            if (i < T) f(i, ch[j], cs[j]);
        }
        for (int i = threadIdx.x + kCached * kThreads; i < T; i += kThreads) f(i, ordered(h[i]), ordered(s[i]));
    };
    auto val = [](int sel, int, uint32_t kh, uint32_t ks) { return sel < 2 ? kh : ks; };
    // the spans of the prompt's keys
    uint32_t lo_h = 0xFFFFFFFFu, hi_h = 0, lo_s = 0xFFFFFFFFu, hi_s = 0;
    each([&](int, uint32_t kh, uint32_t ks) {
        lo_h = min(lo_h, kh);
        hi_h = max(hi_h, kh);
        lo_s = min(lo_s, ks);
        hi_s = max(hi_s, ks);
    });
    lo_h = __reduce_min_sync(0xffffffffu, lo_h);
    hi_h = __reduce_max_sync(0xffffffffu, hi_h);
    lo_s = __reduce_min_sync(0xffffffffu, lo_s);
    hi_s = __reduce_max_sync(0xffffffffu, hi_s);
    if (lane == 0) {
        sh.lo4[warp] = lo_h;
        sh.hi4[warp] = hi_h;
        sh.lo5[warp] = lo_s;
        sh.hi5[warp] = hi_s;
    }
    __syncthreads();
    if (threadIdx.x < kSel) {
        const uint32_t* lo4 = threadIdx.x < 2 ? sh.lo4 : sh.lo5;
        const uint32_t* hi4 = threadIdx.x < 2 ? sh.hi4 : sh.hi5;
        uint32_t lo = lo4[0], hi = hi4[0];
        for (int w = 1; w < kThreads / 32; ++w) {
            lo = min(lo, lo4[w]);
            hi = max(hi, hi4[w]);
        }
        // the k-th largest is the (T - k + 1)-th smallest
        sh.sel[threadIdx.x] = Select{lo, shift_for(hi - lo), (threadIdx.x & 1) ? k : T - k + 1, 0};
    }
    __syncthreads();
    narrow<true>(sh, each, val, [](int, int, uint32_t, uint32_t) { return true; });
    // Ties with a threshold: of its `equal` tokens the first n_take by index belong to the
    // group.  (Selected among the tied tokens' indices when that is not all of them.)
    uint32_t v[kSel];
    int cut[kSel];
#pragma unroll
    for (int q = 0; q < kSel; ++q) v[q] = sh.sel[q].lo;
    __syncthreads();
    if (threadIdx.x < kSel) {
        const Select r = sh.sel[threadIdx.x];
        const int take = (threadIdx.x & 1) ? r.rank : r.equal - r.rank + 1;
        sh.sel[threadIdx.x] = Select{0, shift_for((uint32_t)T), take < r.equal ? take : 0, 0};
    }
    __syncthreads();
    narrow<false>(sh, each, [](int, int i, uint32_t, uint32_t) { return (uint32_t)i; },
                  [&](int q, int i, uint32_t kh, uint32_t ks) { return val(q, i, kh, ks) == v[q]; });
#pragma unroll
    for (int q = 0; q < kSel; ++q) cut[q] = sh.sel[q].rank > 0 ? (int)sh.sel[q].lo : T;
    if (threadIdx.x == 0) sh.n_hl = sh.n_lh = 0;
    __syncthreads();
    int hl = 0, lh = 0;
    each([&](int i, uint32_t kh, uint32_t ks) {
        const bool th = kh > v[0] || (kh == v[0] && i <= cut[0]), bh = kh < v[1] || (kh == v[1] && i <= cut[1]);
        const bool ts = ks > v[2] || (ks == v[2] && i <= cut[2]), bs = ks < v[3] || (ks == v[3] && i <= cut[3]);
        hl += th && bs;
        lh += bh && ts;
    });
    hl = __reduce_add_sync(0xffffffffu, hl);
    lh = __reduce_add_sync(0xffffffffu, lh);
    if (lane == 0) {
        atomicAdd(&sh.n_hl, hl);
        atomicAdd(&sh.n_lh, lh);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        counts[3 * b] = k;
        counts[3 * b + 1] = sh.n_hl;
        counts[3 * b + 2] = sh.n_lh;
    }
}

}  // namespace

estp_status launch_misalignment(estp_ctx* ctx, const float* H, const float* S, const int32_t* cu,
                                int B, int64_t sumT, int pct, int32_t* counts, cudaStream_t st) {
    misalign_kernel<<<B, kThreads, 0, st>>>(H, S, cu, B, sumT, pct, counts, ctx->status);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "misalignment launch");
}

}  // namespace estp
