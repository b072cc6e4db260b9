// Entropy of the next-token distribution with the logits formed on the tensor cores
// (Eq. 2-1 of z = h W^T, where W is the model's output projection): the [rows, V] logits
// are never written to memory.
//
// lm_head_kernel: one persistent CTA per SM.  A work item is (row block rb of 128 tokens,
// vocabulary split sp); items run split-fastest, so the CTAs working at one time share a
// few row blocks (kept in L2) and stream W.  For every 256-entry vocabulary tile of its
// split (the last one shorter, in units of 32 entries) the CTA forms the 128 x 256 logit tile in TMEM,
//   D = sum over 64-wide chunks c of the hidden size of A_c B_c^T,
// with A_c = hidden[rows of rb, c] and B_c = W[entries of the tile, c] staged by TMA in a
// 4-stage ring (128B-swizzled, 48 KB per stage), 4 tcgen05.mma (M = 128, N = 256, K = 16)
// per stage, and two accumulators of 256 fp32 columns (all 512 TMEM columns), so that the
// epilogue of one tile overlaps the MMAs of the next.
//   warp 0      TMA producer
//   warp 1      MMA issuer (one thread)
//   warps 2-5   epilogue: warp w reads TMEM lanes 32 (w % 4) .. (one token each) in
//               32-column chunks and folds them into the token's running
//               m = max y, s = sum 2^(y - m), t = sum 2^(y - m) (y - m), y = z log2(e)
// At the end of an item each token's (m, s, t) for the split goes to a partial buffer;
// lm_head_merge_kernel combines the splits in a fixed order,
//   M = max m_k, S = sum 2^(m_k - M) s_k, T = sum 2^(m_k - M) (t_k + s_k (m_k - M)),
// and writes H = ln 2 (log2 S - T / S) (nats).
//
// Every mbarrier wait is bounded (a test may lower the limit of the abortable waits
// through estp_set_wait_limit); on expiry the CTA records ESTP_ERR_TIMEOUT in the status
// word, drains its own copies and MMAs and frees its TMEM.
#include "split_rules.cuh"
#include "tcgen05.cuh"

namespace estp {
namespace {

constexpr int kM = 128;                       // tokens per tile (TMEM lanes)
constexpr int kN = 256;                       // vocabulary entries per tile (MMA N)
constexpr int kUnit = 32;                     // granularity of a tile that is not full
constexpr int kKc = 64;                       // hidden-size chunk per stage (one swizzle atom)
constexpr int kStages = 4;
constexpr int kABytes = kM * kKc * 2;         // 16 KB
constexpr int kBBytes = kN * kKc * 2;         // 32 KB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kAccBufs = 2;                   // 2 x 256 TMEM columns
constexpr int kEpiWarp0 = 2;
constexpr int kEpiWarps = 4;
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
// dynamic shared memory (offsets from a 1024-aligned base)
constexpr int kBarOff = kStages * kStageBytes;
constexpr int kNumBars = 2 * kStages + 2 * kAccBufs + 1;  // full, empty, acc_full, acc_empty, drain
constexpr int kMiscOff = kBarOff + kNumBars * 8;           // tmem address, abort flag
constexpr int kSmemBytes = kMiscOff + 16 + 1024;           // + alignment slack
static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");

struct LmArgs {
    int64_t n_rows;
    int64_t V;
    int nk;            // hidden-size chunks (D / 64)
    int n_unit;        // vocabulary units of kUnit entries
    int S;             // vocabulary splits
    int gran;          // units a split is cut in (1, or a whole tile)
    int a_bytes;       // bytes of a stage's A box: 128 rows, or the rows of a single smaller block
    int64_t n_items;   // row blocks x splits
    float* part;       // [3][S][n_rows]: m, s, t (log2 units)
    int* status;
    long long wait_cycles;  // limit of the abortable waits (kWaitCycles unless a test lowers it)
};

// Vocabulary units [u0, u1) of split sp: lm_split says when splits end inside a tile.
__device__ __forceinline__ void split_range(const LmArgs& a, int sp, int& u0, int& u1) {
    const int64_t n = (a.n_unit + a.gran - 1) / a.gran;
    u0 = (int)(sp * n / a.S) * a.gran;
    u1 = min(a.n_unit, (int)((sp + 1) * n / a.S) * a.gran);
}
constexpr int kTileUnits = kN / kUnit;
static_assert(kTileUnits == kLmTileUnits, "units of a tile");

// D (TMEM) = A B^T (+ D when acc != 0) with N = n columns.
__device__ __forceinline__ void mma_n(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t n, uint32_t acc) {
    const uint32_t idesc = idesc_bf16(kM, 0) | ((n >> 3) << 17);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Fold 32 logits z (one chunk of this token's row) into (m, s, t), log2 units.  Columns
// at or past `valid` are outside the vocabulary.
__device__ __forceinline__ void fold_chunk(float* v, int valid, float& m, float& s, float& t) {
    if (valid < 32) {
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c >= valid) v[c] = -1e30f;  // 2^(y - m) = 0 and 0 * (y - m) = 0 (finite)
    }
    float mk[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float* w8 = v + 8 * k;
        mk[k] = fmaxf(fmax3(fmax3(w8[0], w8[1], w8[2]), w8[3], w8[4]), fmax3(w8[5], w8[6], w8[7]));
    }
    const float my = fmaxf(fmax3(mk[0], mk[1], mk[2]), mk[3]) * kLog2e;
    if (my > m) {  // rescale (s, t) to the new max: t' = f (t + s (m - m')), s' = f s
        if (m == -INFINITY) {
            s = 0.f;
            t = 0.f;
        } else {
            const float dm = m - my, f = ex2(dm);
            t = f * fmaf(s, dm, t);
            s *= f;
        }
        m = my;
    }
    const float2 l2 = make_float2(kLog2e, kLog2e), nm = make_float2(-m, -m);
    float2 s2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float2 t2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        const float2 d = __ffma2_rn(make_float2(v[c], v[c + 1]), l2, nm);  // y - m
        const float2 e = make_float2(ex2(d.x), ex2(d.y));
        const int j = (c >> 1) & 1;
        s2[j] = __fadd2_rn(s2[j], e);
        t2[j] = __ffma2_rn(e, d, t2[j]);
    }
    const float2 ss = __fadd2_rn(s2[0], s2[1]), tt = __fadd2_rn(t2[0], t2[1]);
    s += ss.x + ss.y;
    t += tt.x + tt.y;
}

__global__ void __launch_bounds__(kThreads, 1)
    lm_head_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                   const __grid_constant__ CUtensorMap tm_bu, const LmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    // an offset, not a rounded address: the compiler then knows the pointer as shared memory
    uint8_t* sm = smem_raw + (-smem_u32(smem_raw) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + kBarOff);
    uint64_t* full = bars;                       // [kStages]
    uint64_t* empty = full + kStages;            // [kStages]
    uint64_t* acc_full = empty + kStages;        // [kAccBufs]
    uint64_t* acc_empty = acc_full + kAccBufs;   // [kAccBufs]
    uint64_t* drain = acc_empty + kAccBufs;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + kMiscOff);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + kMiscOff + 4);

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the merge may be scheduled
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < kAccBufs; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], kEpiWarps);  // one arrival per epilogue warp
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) {  // TMEM: kAccBufs x 256 columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kAccBufs * kN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_a)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_b)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_bu)) : "memory");
            uint32_t step = 0;
            bool ok = true;
            for (int64_t item = blockIdx.x; ok && item < a.n_items; item += gridDim.x) {
                const int sp = (int)(item % a.S), rb = (int)(item / a.S);
                int u0, u1;
                split_range(a, sp, u0, u1);
                for (int ut = u0; ok && ut < u1; ut += kTileUnits) {
                    const int n_u = u1 - ut < kTileUnits ? u1 - ut : kTileUnits;
                    for (int kc = 0; kc < a.nk; ++kc, ++step) {
                        const int stage = (int)(step % kStages);
                        const uint32_t u = step / kStages;
                        if (u >= 1 && !wait_bar(&empty[stage], (u - 1) & 1, abort_flag, a.status, a.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        uint8_t* st = sm + stage * kStageBytes;
                        // a tile of a split of whole tiles is one box, past the vocabulary zero-filled; another
                        // one's last tile is a box for each of its units
                        const int boxed = n_u == kTileUnits || a.gran == kTileUnits ? kTileUnits : n_u;
                        mbar_expect_tx(&full[stage], a.a_bytes + boxed * (kBBytes / kTileUnits));
                        tma_load_2d(st, &tm_a, kc * kKc, rb * kM, &full[stage]);
                        if (boxed == kTileUnits) {
                            tma_load_2d(st + kABytes, &tm_b, kc * kKc, ut * kUnit, &full[stage]);
                        } else {
                            for (int j = 0; j < n_u; ++j)
                                tma_load_2d(st + kABytes + j * (kBBytes / kTileUnits), &tm_bu, kc * kKc,
                                            (ut + j) * kUnit, &full[stage]);
                        }
                    }
                }
            }
            // every copy this thread issued has landed before the CTA can exit
            for (uint32_t i = 0; i < (uint32_t)kStages && i < step; ++i)
                drain_wait(&full[(step - 1 - i) % kStages], ((step - 1 - i) / kStages) & 1, a.status);
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        if (lane == 0) {
            uint32_t step = 0, tile = 0;
            bool ok = true, issued = false;
            for (int64_t item = blockIdx.x; ok && item < a.n_items; item += gridDim.x) {
                const int sp = (int)(item % a.S);
                int u0, u1;
                split_range(a, sp, u0, u1);
                for (int ut = u0; ok && ut < u1; ut += kTileUnits, ++tile) {
                    const uint32_t n = (uint32_t)((u1 - ut < kTileUnits ? u1 - ut : kTileUnits) * kUnit);
                    const int ab = (int)(tile % kAccBufs);
                    const uint32_t ua = tile / kAccBufs;
                    if (ua >= 1 && !wait_bar(&acc_empty[ab], (ua - 1) & 1, abort_flag, a.status, a.wait_cycles)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(ab * kN);
                    for (int kc = 0; kc < a.nk; ++kc, ++step) {
                        const int stage = (int)(step % kStages);
                        if (!wait_bar(&full[stage], (step / kStages) & 1, abort_flag, a.status, a.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        issued = true;
                        const uint32_t sa = smem_u32(sm + stage * kStageBytes);
#pragma unroll
                        for (int kk = 0; kk < kKc / 16; ++kk)
                            mma_n(d, sw128_desc(sa + kk * 32), sw128_desc(sa + kABytes + kk * 32), n,
                                  (kc > 0 || kk > 0) ? 1u : 0u);
                        mma_commit(&empty[stage]);
                    }
                    if (ok) mma_commit(&acc_full[ab]);
                }
            }
            if (issued) {  // every MMA done before the TMEM is released
                mma_commit(drain);
                drain_wait(drain, 0, a.status);
            }
        }
    } else {
        // ------------------------------------------------------------- epilogue
        const int q = warp & 3;               // TMEM lane quarter
        const int row_l = q * 32 + lane;      // token of the tile owned by this thread
        uint32_t tile = 0;
        bool ok = true;
        for (int64_t item = blockIdx.x; ok && item < a.n_items; item += gridDim.x) {
            const int sp = (int)(item % a.S), rb = (int)(item / a.S);
            int u0, u1;
            split_range(a, sp, u0, u1);
            float m = -INFINITY, s = 0.f, t = 0.f;
            for (int ut = u0; ut < u1; ut += kTileUnits, ++tile) {
                const int n_u = u1 - ut < kTileUnits ? u1 - ut : kTileUnits;
                const int ab = (int)(tile % kAccBufs);
                if (!warp_wait(&acc_full[ab], (tile / kAccBufs) & 1, abort_flag, a.status, a.wait_cycles)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * kN);
                const int64_t v0 = (int64_t)ut * kUnit;
#pragma unroll 1
                for (int ch = 0; ch < n_u; ++ch) {  // a unit is one 32-column load
                    float v[32];
                    tmem_ld32(taddr + ch * 32, v);
                    tmem_wait_ld();
                    if (ch == n_u - 1) {  // the whole tile is in registers: release it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty[ab]);
                    }
                    const int64_t left = a.V - (v0 + ch * 32);
                    fold_chunk(v, left < 32 ? (int)left : 32, m, s, t);
                }
            }
            if (!ok) break;
            const int64_t row = (int64_t)rb * kM + row_l;
            if (row < a.n_rows) {
                const int64_t plane = (int64_t)a.S * a.n_rows;
                float* p = a.part + (int64_t)sp * a.n_rows + row;
                p[0] = m;
                p[plane] = s;
                p[2 * plane] = t;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kAccBufs * kN));
    }
}

// Per token: the splits' (m, s, t) combined, H in nats.  A block takes 32 tokens; its warp y the
// splits y, y + Y, .. of each in order, and the Y results are combined in warp order (a fixed
// order, whatever the launch).  A single row block has a split per SM (152).  One thread a token,
// which read its splits one after another, took 198 us with the 594 whole-tile splits that 37
// tokens of a 152064-entry vocabulary had then (the call 342 us, against 176 now).  Launched as a
// programmatic dependent of lm_head_kernel.
constexpr int kMergeWarps = 32;
__device__ __forceinline__ void merge_split(float& M, float& S, float& T, float m, float s, float t) {
    const float mm = fmaxf(M, m);
    if (mm == -INFINITY) return;  // splits without vocabulary entries
    const float da = M - mm, db = m - mm;
    // an empty side (-inf) has S = T = 0 and a weight of 0
    const float fa = M == -INFINITY ? 0.f : ex2(da), fb = m == -INFINITY ? 0.f : ex2(db);
    T = (M == -INFINITY ? 0.f : fa * fmaf(S, da, T)) + (m == -INFINITY ? 0.f : fb * fmaf(s, db, t));
    S = fa * S + fb * s;
    M = mm;
}

__global__ void __launch_bounds__(32 * kMergeWarps) lm_head_merge_kernel(const float* part, int64_t n_rows, int S,
                                                                          float* __restrict__ H) {
    __shared__ float3 red[kMergeWarps][32];
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the partials are complete
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int64_t r = (int64_t)blockIdx.x * 32 + lane;
    const int64_t plane = (int64_t)S * n_rows;
    float M = -INFINITY, Sx = 0.f, Tx = 0.f;
    if (r < n_rows) {
        constexpr int kBatch = 4;  // splits whose loads are in flight at once
        for (int k0 = warp; k0 < S; k0 += kBatch * n_warps) {
            float m[kBatch], s[kBatch], t[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int k = k0 + j * n_warps;
                const float* p = part + (int64_t)k * n_rows + r;
                m[j] = k < S ? p[0] : -INFINITY;
                s[j] = k < S ? p[plane] : 0.f;
                t[j] = k < S ? p[2 * plane] : 0.f;
            }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) merge_split(M, Sx, Tx, m[j], s[j], t[j]);
        }
    }
    red[warp][lane] = make_float3(M, Sx, Tx);
    __syncthreads();
    if (warp != 0 || r >= n_rows) return;
    for (int w = 1; w < n_warps; ++w) {
        const float3 o = red[w][lane];
        merge_split(M, Sx, Tx, o.x, o.y, o.z);
    }
    H[r] = kLn2 * (lg2(Sx) - Tx / Sx);
}


// [rows, ld] bf16 row-major viewed as a 2-D tensor (D, rows); box 64 x box_rows, 128B
// swizzle; rows past the end read as zero.
estp_status make_map_2d(CUtensorMap* m, const void* base, int64_t D, int64_t rows, int64_t ld,
                        int box_rows) {
    auto fn = tensor_map_encoder();
    if (!fn) return fail(ESTP_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)kKc, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                    box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ESTP_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return ESTP_OK;
}

}  // namespace

estp_status launch_lm_head_entropy(estp_ctx* ctx, const void* hidden, int64_t ldh, const void* W,
                                   int64_t ldw, int64_t n_rows, int64_t D, int64_t V, float* H,
                                   cudaStream_t st) {
    CUtensorMap tma, tmb, tmbu;
    // a batch of fewer rows than a tile loads only those (in groups of 8): what the other rows of
    // the shared tile hold goes to logits that no one reads.  (A box of 128 rows around one row of a
    // 4096-wide hidden state: the call 220 us against 173.)
    const int a_rows = n_rows < kM ? (int)(n_rows + 7) / 8 * 8 : kM;
    estp_status s = make_map_2d(&tma, hidden, D, n_rows, ldh, a_rows);
    if (s != ESTP_OK) return s;
    s = make_map_2d(&tmb, W, D, V, ldw, kN);
    if (s != ESTP_OK) return s;
    s = make_map_2d(&tmbu, W, D, V, ldw, kUnit);
    if (s != ESTP_OK) return s;
    LmArgs a{};
    a.n_rows = n_rows;
    a.V = V;
    a.nk = (int)(D / kKc);
    a.n_unit = (int)((V + kUnit - 1) / kUnit);
    const int64_t n_rb = (n_rows + kM - 1) / kM;
    // vocabulary splits: at least as many that the row blocks in flight at once (G / S of them,
    // 256 D bytes each) fit in ~48 MB of L2 beside the W tiles streaming through
    const int64_t G = ctx->num_sms;
    const int64_t l2_budget = 48ll << 20, rb_bytes = (int64_t)kM * D * 2;
    const int64_t s_l2 = (G * rb_bytes + l2_budget - 1) / l2_budget;
    const LmSplit cut = lm_split(n_rb, a.n_unit, s_l2, G);
    const int64_t S = cut.S;
    a.S = (int)S;
    a.gran = cut.gran;
    a.a_bytes = a_rows * kKc * 2;
    a.n_items = n_rb * S;
    s = ws_reserve(ctx, sizeof(float) * 3 * (size_t)S * (size_t)n_rows);
    if (s != ESTP_OK) return s;
    a.part = static_cast<float*>(ctx->ws);
    a.status = ctx->status;
    a.wait_cycles = ctx->wait_cycles;
    cudaError_t e = cudaFuncSetAttribute(lm_head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmemBytes);
    if (e != cudaSuccess) return cuda_fail(e, "lm-head kernel smem attribute");
    const int64_t grid = a.n_items < ctx->num_sms ? a.n_items : ctx->num_sms;
    lm_head_kernel<<<(unsigned)grid, kThreads, kSmemBytes, st>>>(tma, tmb, tmbu, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "lm-head kernel launch");
    // a warp per four splits (the merge's batch), at most kMergeWarps
    const int mw = a.S >= 4 * kMergeWarps ? kMergeWarps : (a.S + 3) / 4;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n_rows + 31) / 32));
    cfg.blockDim = dim3((unsigned)(32 * mw));
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, lm_head_merge_kernel, (const float*)a.part, n_rows, a.S, H);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "lm-head merge launch");
}

}  // namespace estp
