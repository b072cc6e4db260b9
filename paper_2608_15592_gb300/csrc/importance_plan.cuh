// Work plans for the attention kernels (shared by the CUDA-core and tcgen05 paths).
//
// Importance items.  A prompt of T tokens has nt = ceil(T / tile) key tiles.  Key
// tile kt receives mass only from query tiles kt .. nt-1 (causal), which are cut
// into chunks of qc query tiles:  item (group slot g, key tile kt, chunk c) covers
// query tiles kt + c*qc .. min(nt, kt + (c+1)*qc) - 1.  Items of one prompt are
// numbered g-major, then kt, then c.  The number of items of one group is
//   f(nt) = sum_{m=1..nt} ceil(m / qc) = qc*a*(a+1)/2 + r*(a+1),  nt = a*qc + r,
// and key tile kt starts at item F(kt) = f(nt) - f(nt - kt).
//
// LSE items: (query tile, head slot), numbered from the last query tile (longest
// rows, most key tiles) to the first, so that a dynamic scheduler hands out the
// largest items of a prompt first.
#pragma once
#include "estp_internal.cuh"
#include "split_rules.cuh"

namespace estp {

constexpr int kMaxSorted = 64;  // prompts of a plan in order of length

struct PlanInfo {
    int32_t ok;      // 1 when cu_seqlens passed the device checks
    int32_t total;   // total items
    int32_t next;    // dynamic work counter of the persistent kernels (zeroed by the plan)
    int32_t sorted;  // 1: items run over the prompts order[0], order[1], .. (longest first)
    int16_t order[kMaxSorted];
};

// Per-prompt count of a plan of kind 0: importance items f(nt); kind 1: one per tile, nt;
// kind 2: one per pair of tiles (query tile, key tile <= query tile), nt (nt + 1) / 2.
__host__ __device__ __forceinline__ int64_t plan_count(int64_t nt, int qc, int kind) {
    return kind == 0 ? items_f(nt, qc) : kind == 1 ? nt : nt * (nt + 1) / 2;
}

// One plan: each prompt counts mult * plan_count(ceil(length / tile), qc, kind) items.  sorted (at
// most kMaxSorted prompts): the prompts run from the longest to the shortest.
struct PlanReq {
    int tile, qc, mult, kind;
    int32_t* base;   // [B + 1] prefix of the counts, in the order of the prompts
    PlanInfo* info;
    int sorted;
};
constexpr int kMaxPlans = 3;
struct PlanSet {
    PlanReq plan[kMaxPlans];
};

// The plans a call's kernels need and the validation of cu_seqlens, in one launch of a block
// of 1024 threads each.  The plans are read where they were passed (__grid_constant__): a block
// that picks its own out of a parameter passed by value copies all of them to its stack first
// (5.5 against 3.4 us a launch, which every call waits for).
__global__ void __launch_bounds__(1024) attn_plan_kernel(const int32_t* cu, int B, int64_t sumT,
                                                         int max_seqlen,
                                                         const __grid_constant__ PlanSet plans,
                                                         int* status);
template <class... Plans>
void launch_plans(estp_ctx* ctx, const int32_t* cu, int B, int64_t sumT, int max_seqlen,
                  cudaStream_t st, const Plans&... plans) {
    static_assert(sizeof...(plans) <= kMaxPlans, "plans of one call");
    attn_plan_kernel<<<sizeof...(plans), 1024, 0, st>>>(cu, B, sumT, max_seqlen, PlanSet{{plans...}},
                                                        ctx->status);
}

// Workspace bytes of a plan, and its two parts.
static_assert(sizeof(PlanInfo) <= 256, "the info part of a plan");
inline size_t plan_bytes(int B) { return align_up(sizeof(int32_t) * (size_t)(B + 1), 256) + 256; }
inline int32_t* plan_base(char* ws) { return reinterpret_cast<int32_t*>(ws); }
inline PlanInfo* plan_info(char* ws, int B) {
    return reinterpret_cast<PlanInfo*>(ws + plan_bytes(B) - 256);
}

struct ImpItem {
    int b, g, kt, qt0, qt1;
    int64_t t0;
    int T;
};

// The prompt whose items start at base[slot], slot = upper_slot(base, B, item).
__device__ __forceinline__ int prompt_of(const PlanInfo* info, int slot) {
    return info->sorted ? info->order[slot] : slot;
}

// Item `item` of prompt b, whose items start at base[slot].
__device__ __forceinline__ ImpItem decode_imp_item_at(int item, int slot, int b, const int32_t* base,
                                                      const int32_t* cu, int tile, int qc) {
    ImpItem it;
    it.b = b;
    it.t0 = cu[it.b];
    it.T = cu[it.b + 1] - cu[it.b];
    const int nt = (it.T + tile - 1) / tile;
    // a plan holds fewer than 2^30 items, so 32 bits do (a 64-bit division costs ~100 instructions)
    auto f = [qc](uint32_t n) {
        const uint32_t a = n / (uint32_t)qc, r = n % (uint32_t)qc;
        return (uint32_t)qc * (a * (a + 1) / 2) + r * (a + 1);
    };
    const uint32_t per_group = f((uint32_t)nt);
    const uint32_t local = (uint32_t)(item - base[slot]);
    it.g = (int)(local / per_group);
    const uint32_t rem = local - (uint32_t)it.g * per_group;
    int lo = 0, hi = nt - 1;  // largest kt with F(kt) <= rem
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (per_group - f((uint32_t)(nt - mid)) <= rem) lo = mid; else hi = mid - 1;
    }
    it.kt = lo;
    const int c = (int)(rem - (per_group - f((uint32_t)(nt - lo))));
    it.qt0 = lo + c * qc;
    it.qt1 = min(nt, it.qt0 + qc);
    return it;
}

__device__ __forceinline__ ImpItem decode_imp_item_at(int item, int b, const int32_t* base,
                                                      const int32_t* cu, int tile, int qc) {
    return decode_imp_item_at(item, b, b, base, cu, tile, qc);
}

struct LseItem {
    int b, hslot, qt;
    int64_t t0;
    int T;
};

__device__ __forceinline__ LseItem decode_lse_item_at(int item, int slot, int b, const int32_t* base,
                                                      const int32_t* cu, int tile, int n_heads) {
    LseItem it;
    it.b = b;
    it.t0 = cu[it.b];
    it.T = cu[it.b + 1] - cu[it.b];
    const int nt = (it.T + tile - 1) / tile;
    const int local = item - base[slot];
    const int rank = local / n_heads;
    it.hslot = local - rank * n_heads;
    it.qt = nt - 1 - rank;
    return it;
}

__device__ __forceinline__ LseItem decode_lse_item_at(int item, int b, const int32_t* base,
                                                      const int32_t* cu, int tile, int n_heads) {
    return decode_lse_item_at(item, b, b, base, cu, tile, n_heads);
}

__device__ __forceinline__ LseItem decode_lse_item(int item, const int32_t* base, int B,
                                                   const int32_t* cu, int tile, int n_heads) {
    return decode_lse_item_at(item, upper_slot(base, B, item), base, cu, tile, n_heads);
}

}  // namespace estp
