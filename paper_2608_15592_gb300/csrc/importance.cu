// Attention importance (Eq. 2-0, Sec. 3.1): row log-normalisers, causal column sums
// of the softmax attention, the deterministic partial reduce and the final scaling.
//
// This file holds the device plan, the CUDA-core kernels for fp32 inputs (bf16 inputs go to the
// tensor cores at both head sizes) and the launchers that pick a path.
//
// Column sums are formed in the transposed orientation: a CTA owns a tile of KEYS
// and streams the query tiles that may attend to it, so the sum over queries of
// A_ij = 2^(s_ij log2e - lse_i log2e) stays in the thread that owns key j.  Each
// item writes its keys' partial sums to its own slot of a partial buffer; the reduce
// kernel adds the slots of every key in a fixed order (no float atomics).
#include <type_traits>

#include "importance_plan.cuh"
#include "importance_tc.cuh"
#include "sgemm.cuh"

namespace estp {

// One plan, computed by all 1024 threads of the calling block.
static __device__ void plan_body(const int32_t* cu, int B, int64_t sumT, int max_seqlen, int tile,
                                 int qc, int mult, int kind, bool sorted, int32_t* base,
                                 PlanInfo* info, int* status) {
    // thread t owns prompts [t*per, (t+1)*per); one read of cu, warp-shuffle scans
    __shared__ int64_t warp_sum[32];
    __shared__ int bad;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) bad = 0;
    __syncthreads();
    if (tid == 0 && (cu[0] != 0 || (int64_t)cu[B] != sumT)) bad = 1;
    // a sorted plan's prompts by rank of length (equal lengths as they come)
    __shared__ int16_t order[kMaxSorted];
    if (sorted && tid < B) {
        const int32_t len = cu[tid + 1] - cu[tid];
        int rank = 0;
        for (int b = 0; b < B; ++b) {
            const int32_t other = cu[b + 1] - cu[b];
            rank += other > len || (other == len && b < tid);
        }
        order[rank] = info->order[rank] = (int16_t)tid;
    }
    if (sorted) __syncthreads();
    const int per = (B + 1023) / 1024;
    const int b0 = min(B, tid * per), b1 = min(B, b0 + per);
    int64_t local = 0;
    for (int i = b0; i < b1; ++i) {
        const int b = sorted ? order[i] : i;
        const int32_t len = cu[b + 1] - cu[b];
        if (len < 0 || len > max_seqlen) { bad = 1; continue; }
        const int nt = (len + tile - 1) / tile;
        local += (int64_t)mult * plan_count(nt, qc, kind);
    }
    int64_t inc = local;  // inclusive scan within the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t v = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += v;
    }
    if (lane == 31) warp_sum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int64_t w = warp_sum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t v = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += v;
        }
        warp_sum[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    const int64_t total = warp_sum[31];
    const bool ok = !bad && total < INT32_MAX / 2;  // item indices stay 32-bit
    int64_t run = inc - local + (wid > 0 ? warp_sum[wid - 1] : 0);
    for (int i = b0; i < b1; ++i) {
        base[i] = ok ? (int32_t)run : 0;
        const int b = sorted ? order[i] : i;
        const int32_t len = cu[b + 1] - cu[b];
        const int nt = (len + tile - 1) / tile;
        if (len >= 0) run += (int64_t)mult * plan_count(nt, qc, kind);
    }
    if (tid == 1023) {
        base[B] = ok ? (int32_t)total : 0;
        info->ok = ok ? 1 : 0;
        info->total = ok ? (int32_t)total : 0;
        info->next = 0;
        info->sorted = sorted ? 1 : 0;
    }
    if (tid == 0 && !ok) report(status, ESTP_ERR_INVALID_ARG);
}

__global__ void __launch_bounds__(1024) attn_plan_kernel(const int32_t* cu, int B, int64_t sumT,
                                                         int max_seqlen,
                                                         const __grid_constant__ PlanSet plans,
                                                         int* status) {
    // the tensor-core kernel that consumes the plan may launch now and run its prologue;
    // it waits for this grid before its first read of the plan
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const PlanReq p = plans.plan[blockIdx.x];
    plan_body(cu, B, sumT, max_seqlen, p.tile, p.qc, p.mult, p.kind, p.sorted != 0, p.base, p.info, status);
}

namespace {

// ----------------------------------------------------------- CUDA-core kernels
// fp32 inputs: the scores are formed on the FMA pipe (the tensor cores take no fp32 operands)
// in the register tiles of sgemm.cuh.  An item's fixed side is kRows = 16 TM rows (128, or 64
// where 128 would leave SMs idle), its streamed side comes in tiles of 128, and whatever of a
// tile is wholly masked (above the diagonal, past the prompt) is left out in units of 64.
// The bound is the FMA pipe (54 packed FMAs a clock and SM): a 128 x 128 tile takes 32 packed
// FMAs a thread for four 16-byte shared loads.  Items come from a counter, the longest prompt's
// first and its longest first: with prompts in batch order the long items of a late prompt ended
// alone (row normalisers 174 -> 158 us on 4 prompts, column sums 504 -> 369 on 32).  4 prompts of 300
// to 1500 tokens, 16 heads, d 128, against 64 x 64 tiles of scalar FMAs (4 x 4 a thread): row
// normalisers 485 -> 158 us, column sums 857 -> 162.
constexpr int kFThreads = 256;
constexpr int kFCols = 128;          // rows of a streamed tile
template <int TM, int TN>
using ScoreTile = SgemmTile<TM, TN, 16, true, true, false>;
constexpr int kFSmem = ScoreTile<8, 8>::kSmemFloats;

struct F32Args {
    const float* Q;
    const float* K;
    const float* lse;          // column sums: [Hq, sumT] natural log
    const int32_t* cu;
    const int32_t* base;
    PlanInfo* info;
    int B, Hq, Hkv, d;
    int64_t sumT;
    float scale_log2;          // softmax_scale * log2(e)
    ImpHeads hs;
    int exclude_self;
    int sms;                   // SMs of the device (a block of each wave on every one)
    int qc;                    // column sums: query tiles per item
    float* part;               // column sums: [c_max][n_groups][sumT]
    float* lse_out;            // row normalisers: [Hq, sumT]
    int c_max;                 // chunk slots of part (bounds checks of debug builds)
    int* status;
};

// First item of a block.  Items get shorter, so the second block of each SM takes them in the
// reverse order: the SM with the longest first item gets the shortest second one.
__device__ __forceinline__ int first_item(int sms) {
    const int wave = blockIdx.x / sms, r = blockIdx.x - wave * sms;
    return wave * sms + ((wave & 1) ? sms - 1 - r : r);
}

// The items after it come from the plan's counter.
__device__ __forceinline__ int next_item(PlanInfo* info, int* slot) {
    __syncthreads();
    if (threadIdx.x == 0) *slot = (int)gridDim.x + atomicAdd(&info->next, 1);
    __syncthreads();
    return *slot;
}

// Row log-normalisers: rows = queries of one tile, streamed over the keys up to its diagonal.
template <int TM>
__global__ void __launch_bounds__(kFThreads, TM == 8 ? 1 : 2) lse_f32_kernel(const F32Args a) {
    __shared__ __align__(16) float sm[kFSmem];
    __shared__ int slot;
    constexpr int kRows = 16 * TM;
    const int total = a.info->total;
    const int rep = a.Hq / a.Hkv;
    for (int item = first_item(a.sms); item < total; item = next_item(a.info, &slot)) {
        const int at = upper_slot(a.base, a.B, item);
        const LseItem it = decode_lse_item_at(item, at, prompt_of(a.info, at), a.base, a.cu, kRows, a.hs.n_heads);
        const int h = a.hs.head_list[it.hslot];
        const int q0 = it.qt * kRows;
        const GemmSide qs{a.Q + (it.t0 * a.Hq + h) * a.d, (int64_t)a.Hq * a.d, it.T, 1};
        const GemmSide ks{a.K + (it.t0 * a.Hkv + h / rep) * a.d, (int64_t)a.Hkv * a.d, it.T, 1};
        float m[TM], s[TM];
#pragma unroll
        for (int r = 0; r < TM; ++r) { m[r] = -1e30f; s[r] = 0.f; }
        // rows q0 + r0 .. of R x 16 rows against C x 16 keys from k0
        auto tile = [&](auto R, auto C, auto r0c, int k0) {
            constexpr int kR = decltype(R)::value, kC = decltype(C)::value, r0 = decltype(r0c)::value;
            using Tile = ScoreTile<kR, kC>;
            Tile t;
            t.run(sm, qs, q0 + r0, ks, k0, 0, a.d);
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                const int i = q0 + r0 + Tile::row(r);
                float v[kC];
                float mx = -1e30f;
#pragma unroll
                for (int c = 0; c < kC; ++c) {
                    const int j = k0 + Tile::col(c);
                    const float x = c & 1 ? t.c[r][c >> 1].y : t.c[r][c >> 1].x;
                    v[c] = j <= i && j < it.T ? x * a.scale_log2 : -1e30f;
                    mx = fmaxf(mx, v[c]);
                }
                float& mr = m[r0 / 16 + r];
                float& sr = s[r0 / 16 + r];
                const float nm = fmaxf(mr, mx);
                sr *= ex2(mr - nm);
                mr = nm;
#pragma unroll
                for (int c = 0; c < kC; ++c) sr += ex2(v[c] - nm);
            }
        };
        using std::integral_constant;
        constexpr integral_constant<int, 8> c8{};
        constexpr integral_constant<int, 4> c4{};
        constexpr integral_constant<int, 0> z{};
        if (TM == 8 && it.T - q0 > 64) {
            constexpr integral_constant<int, TM> full{};
            for (int k0 = 0; k0 < q0; k0 += kFCols) tile(full, c8, z, k0);
            tile(full, c4, z, q0);  // diagonal: 64 keys for all rows, the next 64 for the lower half
            if constexpr (TM == 8) tile(c4, c4, integral_constant<int, 64>{}, q0 + 64);
        } else {  // 64 rows
            int k0 = 0;
            for (; k0 + kFCols <= q0; k0 += kFCols) tile(c4, c8, z, k0);
            for (; k0 <= q0; k0 += 64) tile(c4, c4, z, k0);
        }
#pragma unroll
        for (int r = 0; r < TM; ++r) {
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) {
                const float m2 = __shfl_xor_sync(0xffffffffu, m[r], off);
                const float s2 = __shfl_xor_sync(0xffffffffu, s[r], off);
                const float nm = fmaxf(m[r], m2);
                s[r] = s[r] * ex2(m[r] - nm) + s2 * ex2(m2 - nm);
                m[r] = nm;
            }
            const int i = q0 + ScoreTile<TM, 4>::row(r);
            if ((threadIdx.x & 15) == 0 && i < it.T)
                a.lse_out[(int64_t)h * a.sumT + it.t0 + i] = (m[r] + lg2(s[r])) * kLn2;
        }
    }
}

// Column sums: rows = keys of one tile, streamed over the item's queries and heads.
template <int TM>
__global__ void __launch_bounds__(kFThreads, 2) imp_f32_kernel(const F32Args a) {
    __shared__ __align__(16) float sm[kFSmem];
    __shared__ int slot;
    constexpr int kRows = 16 * TM;
    const int total = a.info->total;
    for (int item = first_item(a.sms); item < total; item = next_item(a.info, &slot)) {
        const int at = upper_slot(a.base, a.B, item);
        const ImpItem it = decode_imp_item_at(item, at, prompt_of(a.info, at), a.base, a.cu, kRows, a.qc);
        const int k0 = it.kt * kRows;
        const int i_end = min(it.T, it.qt1 * kRows);  // queries of the item
        const GemmSide ks{a.K + (it.t0 * a.Hkv + a.hs.group[it.g]) * a.d, (int64_t)a.Hkv * a.d, it.T, 1};
        float col[TM];
#pragma unroll
        for (int r = 0; r < TM; ++r) col[r] = 0.f;
        for (int hi = a.hs.begin[it.g]; hi < a.hs.begin[it.g + 1]; ++hi) {
            const int h = a.hs.head_list[hi];
            const GemmSide qs{a.Q + (it.t0 * a.Hq + h) * a.d, (int64_t)a.Hq * a.d, it.T, 1};
            const float* lse = a.lse + (int64_t)h * a.sumT + it.t0;
            // keys k0 .. of R x 16 keys against C x 16 queries from i0
            auto tile = [&](auto R, auto C, int i0) {
                constexpr int kR = decltype(R)::value, kC = decltype(C)::value;
                using Tile = ScoreTile<kR, kC>;
                Tile t;
                t.run(sm, ks, k0, qs, i0, 0, a.d);
                float nl[kC];  // -lse log2e
#pragma unroll
                for (int c = 0; c < kC; ++c) {
                    const int i = i0 + Tile::col(c);
                    nl[c] = i < it.T ? -lse[i] * kLog2e : -INFINITY;
                }
#pragma unroll
                for (int r = 0; r < kR; ++r) {
                    const int j = k0 + Tile::row(r);
                    float v = 0.f;
#pragma unroll
                    for (int c = 0; c < kC; ++c) {
                        const int i = i0 + Tile::col(c);
                        const float x = c & 1 ? t.c[r][c >> 1].y : t.c[r][c >> 1].x;
                        const bool ok = i >= j + a.exclude_self && i < it.T;
                        v += ok ? ex2(fmaf(x, a.scale_log2, nl[c])) : 0.f;
                    }
                    col[r] += v;
                }
            };
            constexpr std::integral_constant<int, 8> c8{};
            constexpr std::integral_constant<int, 4> c4{};
            int i0 = it.qt0 * kRows;
            if (TM == 8 && it.T - k0 > 64) {
                constexpr std::integral_constant<int, TM> full{};
                if (i0 == k0) {  // diagonal: the first 64 queries see the first 64 keys only
                    tile(c4, c4, i0);
                    tile(full, c4, i0 + 64);
                    i0 += 128;
                }
                for (; i0 + 64 < i_end; i0 += kFCols) tile(full, c8, i0);
                if (i0 < i_end) tile(full, c4, i0);
            } else {  // 64 keys
                for (; i0 + 64 < i_end; i0 += kFCols) tile(c4, c8, i0);
                if (i0 < i_end) tile(c4, c4, i0);
            }
        }
        const int c_slot = (it.qt0 - it.kt) / a.qc;
        if (!in_bounds(c_slot >= 0 && c_slot < a.c_max, a.status)) continue;
        float* out = a.part + ((int64_t)c_slot * a.hs.n_groups + it.g) * a.sumT + it.t0;
#pragma unroll
        for (int r = 0; r < TM; ++r) {
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) col[r] += __shfl_xor_sync(0xffffffffu, col[r], off);
            const int j = k0 + ScoreTile<TM, 4>::row(r);
            if ((threadIdx.x & 15) == 0 && j < it.T) out[j] = col[r];
        }
    }
}

// acc[j] (+)= sum over chunk slots c and group slots g of part, in a fixed order.
// Largest b with cu[b] <= j: cu staged in shared memory when it fits (kCuStage entries).
constexpr int kCuStage = 2048;

__device__ __forceinline__ const int32_t* stage_cu(const int32_t* cu, int B, int32_t* cu_s) {
    if (B + 1 > kCuStage) return cu;
    for (int i = threadIdx.x; i <= B; i += blockDim.x) cu_s[i] = cu[i];
    __syncthreads();
    return cu_s;
}

__global__ void imp_reduce_kernel(const float* part, const PlanInfo* info, const int32_t* cu,
                                  int B, int64_t sumT, int n_groups, int tile, int qc,
                                  int accumulate, float* acc, int c_max, int* status) {
    __shared__ int32_t cu_s[kCuStage];
    const int32_t* cuv = stage_cu(cu, B, cu_s);
    // the partials are complete past this point (launched as a programmatic dependent
    // of the column-sum kernel; a no-op after an ordinary launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= sumT) return;
    float v = 0.f;
    if (info->ok) {
        const int b = upper_slot(cuv, B, j);
        const int T = cuv[b + 1] - cuv[b];
        const int nt = (T + tile - 1) / tile;
        const int kt = (int)((j - cuv[b]) / tile);
        int n = chunks_of(nt, kt, qc) * n_groups;  // partials (c, g), c-major
        if (!in_bounds(n <= c_max * n_groups && b >= 0 && b < B, status)) n = 0;
        // up to 16 partials are loaded before any is added (independent loads in flight), then
        // added as a tree, so that a sum of n partials has chains of n / 16 additions
        constexpr int kBatch = 16;
        for (int i0 = 0; i0 < n; i0 += kBatch) {
            float p[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i) p[i] = i0 + i < n ? part[(int64_t)(i0 + i) * sumT + j] : 0.f;
#pragma unroll
            for (int w = kBatch / 2; w > 0; w >>= 1)
#pragma unroll
                for (int i = 0; i < w; ++i) p[i] += p[i + w];
            v += p[0];
        }
    }
    acc[j] = accumulate ? acc[j] + v : v;
}

// S_j = C_j / (n_j * layers * heads): n_j = N_b (Eq. 2-0), the causal count of the
// queries whose terms enter C_j (div 1: N_b - j, one fewer without the diagonal;
// S_j = 0 where it is 0), or 1 (div 2).
__global__ void imp_finalize_kernel(const float* acc, const int32_t* cu, int B, int64_t sumT,
                                    float inv_lh, int div, int exclude_self, float* out) {
    __shared__ int32_t cu_s[kCuStage];
    const int32_t* cuv = stage_cu(cu, B, cu_s);
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= sumT) return;
    const int b = upper_slot(cuv, B, j);
    if (!in_bounds(b >= 0 && b < B, nullptr)) return;
    int64_t n = cuv[b + 1] - cuv[b];
    if (div == 1) n = (int64_t)cuv[b + 1] - j - (exclude_self ? 1 : 0);
    else if (div == 2) n = 1;
    out[j] = n > 0 ? acc[j] * inv_lh / (float)n : 0.f;
}

// Whether a plan sorts its prompts: where some items wait for others to end.  (Below that the
// sorting and the look-up cost ~2 us and give nothing.)
int f32_sorted(int B, int64_t items, int64_t blocks) { return B > 1 && B <= kMaxSorted && items > blocks; }

// A group of its own for every head.
ImpHeads heads_apart(const ImpHeads& hs, int rep) {
    ImpHeads o = hs;
    o.n_groups = hs.n_heads;
    for (int i = 0; i < hs.n_heads; ++i) {
        o.group[i] = (int16_t)(hs.head_list[i] / rep);
        o.begin[i] = (int16_t)i;
    }
    o.begin[hs.n_heads] = (int16_t)hs.n_heads;
    return o;
}

template <class Kernel>
cudaError_t launch_f32(estp_ctx* ctx, Kernel kernel, F32Args& a, cudaStream_t st) {
    a.sms = ctx->num_sms;
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kFThreads, 0);
    if (e != cudaSuccess) return e;
    kernel<<<ctx->num_sms * (occ > 0 ? occ : 1), kFThreads, 0, st>>>(a);
    return cudaGetLastError();
}

PlanReq lse_plan_f32(const ImpHeads& hs, int B, int64_t sumT, int num_sms, int32_t* base,
                     PlanInfo* info) {
    const int rows = f32_rows(B, sumT, hs.n_heads, num_sms);
    return {rows, 1, hs.n_heads, 1, base, info,
            f32_sorted(B, (int64_t)B * hs.n_heads * mean_tiles(B, sumT, rows), rows == 128 ? num_sms : 2 * num_sms)};
}

// Row normalisers of the selected heads (fp32).
estp_status launch_lse_f32(estp_ctx* ctx, const void* Q, const void* K, int Hq, int Hkv, int d,
                           float scale, const ImpHeads& hs, const int32_t* cu, int B, int64_t sumT,
                           float* lse, const PlanReq& plan, cudaStream_t st) {
    F32Args a{};
    a.Q = static_cast<const float*>(Q); a.K = static_cast<const float*>(K);
    a.cu = cu; a.B = B; a.Hq = Hq; a.Hkv = Hkv; a.d = d; a.sumT = sumT;
    a.info = plan.info;
    a.base = plan.base;
    a.scale_log2 = scale * kLog2e;
    a.hs = hs;
    a.lse_out = lse;
    const cudaError_t e = plan.tile == 128 ? launch_f32(ctx, lse_f32_kernel<8>, a, st)
                                           : launch_f32(ctx, lse_f32_kernel<4>, a, st);
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "lse launch");
}

PlanReq lse_plan(bool tc, estp_ctx* ctx, const ImpHeads& hs, int B, int64_t sumT, char* ws) {
    int32_t* base = plan_base(ws);
    PlanInfo* info = plan_info(ws, B);
    return tc ? lse_plan_tc(hs, base, info) : lse_plan_f32(hs, B, sumT, ctx->num_sms, base, info);
}

}  // namespace

estp_status launch_lse(estp_ctx* ctx, const void* Q, const void* K, estp_dtype dtype, int Hq,
                       int Hkv, int d, float scale, const ImpHeads& hs, const int32_t* cu,
                       int B, int64_t sumT, int max_seqlen, float* lse, cudaStream_t st) {
    estp_status s = ws_reserve(ctx, plan_bytes(B));
    if (s != ESTP_OK) return s;
    const bool tc = tc_supported(dtype, d);
    const PlanReq plan = lse_plan(tc, ctx, hs, B, sumT, static_cast<char*>(ctx->ws));
    launch_plans(ctx, cu, B, sumT, max_seqlen, st, plan);
    return tc ? launch_lse_tc(ctx, Q, K, Hq, Hkv, d, scale, hs, cu, B, sumT, lse, plan, st)
              : launch_lse_f32(ctx, Q, K, Hq, Hkv, d, scale, hs, cu, B, sumT, lse, plan, st);
}

estp_status launch_importance(estp_ctx* ctx, const void* Q, const void* K, estp_dtype dtype,
                              const float* lse, int Hq, int Hkv, int d, float scale,
                              const ImpHeads& heads, const int32_t* cu, int B, int64_t sumT,
                              int max_seqlen, bool accumulate, uint32_t flags, float* acc,
                              cudaStream_t st) {
    const bool tc = tc_supported(dtype, d);
    const F32Split split = f32_split(B, sumT, max_seqlen, heads.n_heads, heads.n_groups, ctx->num_sms);
    const bool apart = !tc && split.per_head;
    const ImpHeads hs = apart ? heads_apart(heads, Hq / Hkv) : heads;
    const int tile = tc ? tc_tile() : split.rows;
    const int qc = tc ? tc_qc(B, sumT, hs.n_groups, ctx->num_sms) : split.qc;
    const int c_max = chunk_slots(max_seqlen, tile, qc);
    // workspace: [own lse][plan of the lse][plan][partials]
    const size_t lse_bytes = lse ? 0 : align_up(sizeof(float) * (size_t)Hq * (size_t)sumT, 256);
    const size_t off_lse_plan = lse_bytes;
    const size_t off_plan = off_lse_plan + plan_bytes(B);
    const size_t off_part = off_plan + plan_bytes(B);
    const size_t part_bytes = sizeof(float) * (size_t)c_max * (size_t)hs.n_groups * (size_t)sumT;
    estp_status s = ws_reserve(ctx, off_part + part_bytes);
    if (s != ESTP_OK) return s;
    char* ws = static_cast<char*>(ctx->ws);
    int32_t* base = plan_base(ws + off_plan);
    PlanInfo* info = plan_info(ws + off_plan, B);
    float* part = reinterpret_cast<float*>(ws + off_part);
    const PlanReq plan{tile, qc, hs.n_groups, 0, base, info,
                       tc ? 0 : f32_sorted(B, (int64_t)B * hs.n_groups * items_f(mean_tiles(B, sumT, tile), qc),
                                           2 * ctx->num_sms)};
    float* lse_use = const_cast<float*>(lse);
    if (lse) {
        launch_plans(ctx, cu, B, sumT, max_seqlen, st, plan);
    } else {  // the rows of the selected heads first; both plans in one launch
        lse_use = reinterpret_cast<float*>(ws);
        const PlanReq lp = lse_plan(tc, ctx, heads, B, sumT, ws + off_lse_plan);
        launch_plans(ctx, cu, B, sumT, max_seqlen, st, lp, plan);
        s = tc ? launch_lse_tc(ctx, Q, K, Hq, Hkv, d, scale, heads, cu, B, sumT, lse_use, lp, st)
               : launch_lse_f32(ctx, Q, K, Hq, Hkv, d, scale, heads, cu, B, sumT, lse_use, lp, st);
        if (s != ESTP_OK) return s;
    }
    if (tc) {
        s = launch_imp_tc(ctx, Q, K, lse_use, Hq, Hkv, d, scale, hs, cu, B, sumT,
                          (flags & ESTP_IMP_EXCLUDE_SELF) != 0, base, info, part, c_max, qc, st);
        if (s != ESTP_OK) return s;
    } else {
        F32Args a{};
        a.Q = static_cast<const float*>(Q); a.K = static_cast<const float*>(K);
        a.lse = lse_use; a.cu = cu; a.base = base; a.info = info; a.B = B;
        a.Hq = Hq; a.Hkv = Hkv; a.d = d; a.sumT = sumT; a.scale_log2 = scale * kLog2e;
        a.hs = hs; a.exclude_self = (flags & ESTP_IMP_EXCLUDE_SELF) ? 1 : 0; a.qc = qc;
        a.part = part; a.c_max = c_max; a.status = ctx->status;
        const cudaError_t e = tile == 128 ? launch_f32(ctx, imp_f32_kernel<8>, a, st)
                                          : launch_f32(ctx, imp_f32_kernel<4>, a, st);
        if (e != cudaSuccess) return cuda_fail(e, "importance launch");
    }
    {  // a programmatic dependent of the column-sum kernel: it waits on it on the device
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((sumT + 255) / 256));
        cfg.blockDim = dim3(256);
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = cudaLaunchKernelEx(&cfg, imp_reduce_kernel, (const float*)part,
                                           (const PlanInfo*)info, cu, B, sumT, hs.n_groups, tile,
                                           qc, accumulate ? 1 : 0, acc, c_max, ctx->status);
        if (e != cudaSuccess) return cuda_fail(e, "importance reduce launch");
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "importance launch");
}

estp_status launch_importance_finalize(estp_ctx* ctx, const float* acc, const int32_t* cu, int B,
                                       int64_t sumT, int n_layers, int n_heads, uint32_t flags,
                                       float* out, cudaStream_t st) {
    (void)ctx;
    const float inv_lh = 1.f / ((float)n_layers * (float)n_heads);
    const int div = (flags & ESTP_IMP_DIV_CAUSAL) ? 1 : (flags & ESTP_IMP_DIV_NONE) ? 2 : 0;
    imp_finalize_kernel<<<(unsigned)((sumT + 255) / 256), 256, 0, st>>>(
        acc, cu, B, sumT, inv_lh, div, (flags & ESTP_IMP_EXCLUDE_SELF) ? 1 : 0, out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "finalize launch");
}

}  // namespace estp
