// tcgen05 (tensor-core) path of the attention kernels for bf16 inputs.
#pragma once
#include "importance_plan.cuh"

namespace estp {

bool tc_supported(estp_dtype dtype, int d);
int tc_tile();  // keys (and queries) per tile
// pairs of query tiles per column-sum item for a call over B prompts, sumT tokens and
// n_groups KV groups on num_sms SMs
int tc_qc(int B, int64_t sumT, int n_groups, int num_sms);

// The row normalisers' plan, and the kernel that consumes it.  The kernel is a programmatic
// dependent of the launch before it (the plan); so is the column sums' kernel, which may follow
// it directly.
PlanReq lse_plan_tc(const ImpHeads& hs, int32_t* base, PlanInfo* info);
estp_status launch_lse_tc(estp_ctx* ctx, const void* Q, const void* K, int Hq, int Hkv, int d,
                          float scale, const ImpHeads& hs, const int32_t* cu, int B, int64_t sumT,
                          float* lse, const PlanReq& plan, cudaStream_t st);

estp_status launch_imp_tc(estp_ctx* ctx, const void* Q, const void* K, const float* lse, int Hq,
                          int Hkv, int d, float scale, const ImpHeads& hs, const int32_t* cu,
                          int B, int64_t sumT, bool exclude_self, const int32_t* base,
                          const PlanInfo* info, float* part, int c_max, int qc, cudaStream_t st);

}  // namespace estp
