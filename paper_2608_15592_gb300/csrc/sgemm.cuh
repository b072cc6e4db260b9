// fp32 matrix tiles on the FMA pipe, for contractions whose inputs are fp32 and whose result
// has to keep fp32 accuracy (the tensor cores take no fp32 operands).
//
// A block of 256 threads (16 x 16) forms a BM x BN tile of C[m, n] = sum_k A(m, k) B(n, k),
// BM = 16 TM, BN = 16 TN, from slices of BK values of k that are staged in shared memory as
// [k][m] and [k][n], double-buffered: the next slice's global loads are in flight while this
// one is multiplied.  Each thread holds TM x TN sums as packed pairs (fma.rn.f32x2: two FMAs
// per issue slot, which leaves the other slots to the shared loads).  The sums of every 64
// values of k are formed on their own and then added to the running ones, so that a sum over
// k has chains of 64 and k / 64 additions and not one of k.  (kChains = false leaves that out, for short sums of at
// most 128 terms: half the registers.)
#pragma once
#include "estp_internal.cuh"

namespace estp {

// Operand of a tile: rows 0 .. rows-1 along the tile's side, `ld` floats apart when a row's k
// values are contiguous (element (r, k) at p[r ld + k]), or k rows `ld` apart with the tile's
// side contiguous (element (r, k) at p[k ld + r]).  vec: 16-byte loads (base and ld aligned).
struct GemmSide {
    const float* p;
    int64_t ld;
    int64_t rows;
    int vec;
};

template <int TM, int TN, int BK, bool kAlongA, bool kAlongB, bool kChains = true>
struct SgemmTile {
    static constexpr int kThreads = 256;
    static constexpr int BM = 16 * TM, BN = 16 * TN;
    static constexpr int SA = BM + 4, SB = BN + 4;  // floats between k rows in shared memory
    static constexpr int kSlice = BK * (SA + SB);
    static constexpr int kSmemFloats = 2 * kSlice;
    static constexpr int kQA = BM * BK / 4 / kThreads, kQB = BN * BK / 4 / kThreads;  // loads a thread
    static_assert(BM * BK % (4 * kThreads) == 0 && BN * BK % (4 * kThreads) == 0, "slice size");
    static_assert(BK % 16 == 0 && 64 % BK == 0, "slice depth");

    // sums of this thread: C[row(i)][col(2 j), col(2 j + 1)]
    float2 c[TM][TN / 2];

    static __device__ __forceinline__ int ty() { return threadIdx.x >> 4; }
    static __device__ __forceinline__ int tx() { return threadIdx.x & 15; }
    // side index of a thread's i-th value: two groups of four for an 8-wide side
    static __device__ __forceinline__ int place(int t, int i, int width) {
        return width == 8 ? (i >> 2) * 64 + t * 4 + (i & 3) : t * width + i;
    }
    static __device__ __forceinline__ int row(int i) { return place(ty(), i, TM); }
    static __device__ __forceinline__ int col(int j) { return place(tx(), j, TN); }

    // (side index, k) of this thread's q-th load of a slice of `side` rows
    template <bool kAlong>
    static __device__ __forceinline__ void where(int q, int side, int& r, int& k) {
        const int w = (threadIdx.x >> 5) + q * (kThreads / 32), lane = threadIdx.x & 31;
        if (kAlong) {  // a warp takes 8 rows x 16 k: 64-byte runs, two-way store conflicts
            const int per = side / 8;
            r = (w % per) * 8 + (lane >> 2);
            k = (w / per) * 16 + (lane & 3) * 4;
        } else {
            const int i = w * 32 + lane, per = side / 4;
            r = (i % per) * 4;
            k = i / per;
        }
    }

    template <bool kAlong>
    static __device__ __forceinline__ float4 fetch(const GemmSide& s, int64_t r, int64_t k, int64_t k1) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kAlong) {
            if (r < s.rows && k < k1) {
                const float* p = s.p + r * s.ld + k;
                if (s.vec && k + 4 <= k1) return *reinterpret_cast<const float4*>(p);
                v.x = p[0];
                if (k + 1 < k1) v.y = p[1];
                if (k + 2 < k1) v.z = p[2];
                if (k + 3 < k1) v.w = p[3];
            }
        } else if (k < k1 && r < s.rows) {
            const float* p = s.p + k * s.ld + r;
            if (s.vec && r + 4 <= s.rows) return *reinterpret_cast<const float4*>(p);
            v.x = p[0];
            if (r + 1 < s.rows) v.y = p[1];
            if (r + 2 < s.rows) v.z = p[2];
            if (r + 3 < s.rows) v.w = p[3];
        }
        return v;
    }

    template <bool kAlong>
    static __device__ __forceinline__ void stage(float* sm, int stride, int r, int k, const float4& v) {
        if (kAlong) {
            sm[(k + 0) * stride + r] = v.x;
            sm[(k + 1) * stride + r] = v.y;
            sm[(k + 2) * stride + r] = v.z;
            sm[(k + 3) * stride + r] = v.w;
        } else {
            *reinterpret_cast<float4*>(sm + k * stride + r) = v;
        }
    }

    template <int W>
    static __device__ __forceinline__ void frag(const float* sm, int t, float* v) {
        if constexpr (W == 8 || W == 4) {
#pragma unroll
            for (int g = 0; g < W / 4; ++g) {
                const float4 x = *reinterpret_cast<const float4*>(sm + g * 64 + t * 4);
                v[4 * g] = x.x; v[4 * g + 1] = x.y; v[4 * g + 2] = x.z; v[4 * g + 3] = x.w;
            }
        } else if constexpr (W == 2) {
            const float2 x = *reinterpret_cast<const float2*>(sm + t * 2);
            v[0] = x.x; v[1] = x.y;
        } else {
            v[0] = sm[t];
        }
    }

    // Rows m0.. of A and n0.. of B over k in [k0, k1); sm: kSmemFloats floats, 16-byte aligned.
    // kSumA: thread t < BM also returns in *sum_a the sum over k of A(m0 + t, k).
    // Ends with a barrier (sm may be reused).
    template <bool kSumA = false>
    __device__ __forceinline__ void run(float* sm, const GemmSide& A, int64_t m0, const GemmSide& B,
                                        int64_t n0, int64_t k0, int64_t k1, float* sum_a = nullptr) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) c[i][j] = make_float2(0.f, 0.f);
        if (kSumA) *sum_a = 0.f;
        if (k0 >= k1) return;
        float4 ra[kQA], rb[kQB];
        auto load = [&](int64_t k) {
#pragma unroll
            for (int q = 0; q < kQA; ++q) {
                int r, kk;
                where<kAlongA>(q, BM, r, kk);
                ra[q] = fetch<kAlongA>(A, m0 + r, k + kk, k1);
            }
#pragma unroll
            for (int q = 0; q < kQB; ++q) {
                int r, kk;
                where<kAlongB>(q, BN, r, kk);
                rb[q] = fetch<kAlongB>(B, n0 + r, k + kk, k1);
            }
        };
        auto put = [&](int buf) {
            float* as = sm + buf * kSlice;
            float* bs = as + BK * SA;
#pragma unroll
            for (int q = 0; q < kQA; ++q) {
                int r, kk;
                where<kAlongA>(q, BM, r, kk);
                stage<kAlongA>(as, SA, r, kk, ra[q]);
            }
#pragma unroll
            for (int q = 0; q < kQB; ++q) {
                int r, kk;
                where<kAlongB>(q, BN, r, kk);
                stage<kAlongB>(bs, SB, r, kk, rb[q]);
            }
        };
        load(k0);
        put(0);
        __syncthreads();
        float2 p[kChains ? TM : 1][TN / 2];
        int buf = 0, slices = 0;
        float part_a = 0.f;
        for (int64_t k = k0; k < k1; k += BK) {
            const bool more = k + BK < k1;
            if (more) load(k + BK);
            if (slices == 0) {
                if constexpr (kChains) {
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < TN / 2; ++j) p[i][j] = make_float2(0.f, 0.f);
                }
                part_a = 0.f;
            }
            const float* as = sm + buf * kSlice;
            const float* bs = as + BK * SA;
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                float av[TM], bv[TN];
                frag<TM>(as + kk * SA, ty(), av);
                frag<TN>(bs + kk * SB, tx(), bv);
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN / 2; ++j) {
                        float2& sum = kChains ? p[kChains ? i : 0][j] : c[i][j];
                        sum = __ffma2_rn(make_float2(av[i], av[i]), make_float2(bv[2 * j], bv[2 * j + 1]), sum);
                    }
                if (kSumA && threadIdx.x < BM) part_a += as[kk * SA + threadIdx.x];
            }
            if (++slices == 64 / BK || !more) {
                slices = 0;
                if constexpr (kChains) {
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < TN / 2; ++j) c[i][j] = __fadd2_rn(c[i][j], p[i][j]);
                }
                if (kSumA) *sum_a += part_a;
            }
            if (more) put(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
};

}  // namespace estp
