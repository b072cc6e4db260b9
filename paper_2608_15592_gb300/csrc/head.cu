// Training loss of the length head (Sec. 3.3): the soft label of Eq. 3-1, the linear
// head of Eq. 3-2 and the loss of Eq. 3-3 averaged over the prompts, with its gradients;
// and the MLP predictor of Sec. 3.3 / Fig. 2 (one hidden layer of F ReLU units in front
// of the K-bin softmax projection), its prediction and its loss.
//
// Everything is fp32: the contractions run on the FMA pipe through the tiles of sgemm.cuh.
// A layer y = W x (x [B, D], W [K, D]) with its loss takes three launches:
//   logit_part_kernel: z = W x cut into 32 x 32 tiles and, so that a small batch still fills
//     the GPU, into splits of D; each split's sums go to its own slot of a partial buffer.
//   head_loss_kernel: CTA b adds prompt b's slots in order, p_hat = softmax(z),
//     y_hat = sum p_hat_k c_k (relative to the centre of the largest logit), the soft label
//     around the bin nearest to y_b, the prompt's CE and squared error, and dL/dz_b (with the
//     batch mean's 1/B).
//   layer_grad_kernel: tiles of dL/dW = sum_b dz_b x_b^T and of dL/dx_b = W^T dz_b, with
//     dL/dbias = sum_b dz_b along the first column of tiles, and one block for the loss.
// The MLP adds wide_gemm_kernel, u = max(W1 h + b1, 0) and dL/dh = W1^T g, cut along its
// contraction over a cluster whose CTAs add their tiles through distributed shared memory
// (hidden_rows_kernel forms u for at most 8 prompts), and outer_kernel, dL/dW1 = g^T h with dL/db1; g = dL/du where u > 0 (the ReLU's
// derivative), formed by layer_grad_kernel.  Every sum runs in a fixed order.
//
// Measured, 256 prompts, D = 4096, K = 32 (GB300, device times with cold caches):
//   linear head: 7.5 + 5.6 + 14.4 us against 51 + 48 us for one block a prompt forming its K dot
//   products one after another (one load in flight a lane) and one thread an output of the
//   gradients (256 dependent loads); the call 59 -> 26 us.
//   MLP, F = 1024: hidden 60 us (36 TFLOP/s fp32), dL/dW1 55, dL/dh 64, against 489, 600 and 151
//   for kernels that read an operand from L2 for every few FMAs; the call 1016 -> 198 us.
#include <cooperative_groups.h>

#include <type_traits>

#include "estp_internal.cuh"
#include "sgemm.cuh"
#include "split_rules.cuh"

namespace estp {
namespace {

namespace cg = cooperative_groups;

constexpr int kMaxK = 1024;
constexpr int kLossThreads = 128;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Each kernel below may be launched as a programmatic dependent of the launch before it: it
// lets its own dependent start, then waits for the launch before it to complete.
__device__ __forceinline__ void chain_launches() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Partial logits: part[s][b][k] = sum over split s of D of x[b, :] W[k, :].
// Block (b tile of 32, k tile of 32, split).
using LogitTile = SgemmTile<2, 2, 64, true, true>;
__global__ void __launch_bounds__(256) logit_part_kernel(GemmSide x, GemmSide w, int64_t D, int split,
                                                         float* __restrict__ part) {
    __shared__ __align__(16) float sm[LogitTile::kSmemFloats];
    chain_launches();
    const int64_t b0 = (int64_t)blockIdx.x * LogitTile::BM, k0 = (int64_t)blockIdx.y * LogitTile::BN;
    const int64_t d0 = (int64_t)blockIdx.z * split;
    LogitTile t;
    t.run(sm, x, b0, w, k0, d0, d0 + split < D ? d0 + split : D);
    float* out = part + (int64_t)blockIdx.z * x.rows * w.rows;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int64_t b = b0 + t.row(i), k = k0 + t.col(0);
        if (b < x.rows && k < w.rows) out[b * w.rows + k] = t.c[i][0].x;
        if (b < x.rows && k + 1 < w.rows) out[b * w.rows + k + 1] = t.c[i][0].y;
    }
}

// One block per prompt: logits from the n_split partial slots, then the head (targets NULL:
// prediction only).
__global__ void __launch_bounds__(kLossThreads) head_loss_kernel(
    const float* __restrict__ zpart, int n_split, const float* __restrict__ bias,
    const float* __restrict__ centers, int K, const float* __restrict__ targets, int B, float lambda3,
    float* __restrict__ dz, float2* __restrict__ part, float* __restrict__ pred,
    float* __restrict__ probs) {
    __shared__ float z_s[kMaxK];
    chain_launches();
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // four threads a bin add a quarter of the slots each (eight loads in flight), then two
    // exchanges; the same order whatever the launch
    for (int i0 = 0; i0 < 4 * K; i0 += kLossThreads) {
        const int i = i0 + threadIdx.x, k = i >> 2;
        float acc = 0.f;
        if (k < K) {
            const float* p = zpart + (int64_t)b * K + k;
            const int64_t slot = (int64_t)B * K;
            for (int s0 = i & 3; s0 < n_split; s0 += 32) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = s0 + 4 * j < n_split ? __ldcg(p + (s0 + 4 * j) * slot) : 0.f;
                acc += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
            }
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (k < K && (i & 3) == 0) z_s[k] = acc + (bias ? bias[k] : 0.f);
    }
    __syncthreads();
    if (warp != 0) return;
    // softmax over the K bins, the expectation of Eq. 3-2, and the nearest bin of y_b.
    // y_hat is formed relative to the centre of the largest logit r: y_hat = c_r + dy with
    // dy = sum_k p_hat_k (c_k - c_r), so that c_k - y_hat = (c_k - c_r) - dy does not
    // cancel when p_hat is concentrated on r.
    float m = -INFINITY;
    int r = 0;
    for (int k = lane; k < K; k += 32)
        if (z_s[k] > m) { m = z_s[k]; r = k; }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {  // (max, first index)
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const int orr = __shfl_xor_sync(0xffffffffu, r, off);
        if (om > m || (om == m && orr < r)) { m = om; r = orr; }
    }
    const float cr = centers[r];
    float Z = 0.f, dy = 0.f;
    for (int k = lane; k < K; k += 32) {
        const float e = __expf(z_s[k] - m);
        Z += e;
        dy = fmaf(e, centers[k] - cr, dy);
    }
    Z = warp_sum(Z);
    dy = warp_sum(dy) / Z;
    const float yh = cr + dy;
    if (pred && lane == 0) pred[b] = yh;
    if (probs)
        for (int k = lane; k < K; k += 32) probs[(int64_t)b * K + k] = __expf(z_s[k] - m) / Z;
    if (!targets) return;  // prediction only
    const float y = targets[b];
    float best_d = INFINITY;
    int best_k = 0;
    for (int k = lane; k < K; k += 32) {
        const float d = fabsf(y - centers[k]);
        if (d < best_d) { best_d = d; best_k = k; }  // lowest k of this lane on a tie
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {  // (distance, index): the lowest index wins ties
        const float od = __shfl_xor_sync(0xffffffffu, best_d, off);
        const int ok = __shfl_xor_sync(0xffffffffu, best_k, off);
        if (od < best_d || (od == best_d && ok < best_k)) { best_d = od; best_k = ok; }
    }
    const int i = best_k;
    float norm = 0.f;
    for (int k = lane; k < K; k += 32) norm += __expf(-fabsf((float)(k - i)));
    norm = warp_sum(norm);
    const float lnZ = __logf(Z), err = yh - y, inv_b = 1.f / (float)B;
    float ce = 0.f;
    for (int k = lane; k < K; k += 32) {
        const float p = __expf(-fabsf((float)(k - i))) / norm;
        const float lp_hat = z_s[k] - m - lnZ;  // ln p_hat_k
        const float p_hat = __expf(lp_hat);
        ce -= p * lp_hat;
        dz[(int64_t)b * K + k] =
            (lambda3 * (p_hat - p) + (1.f - lambda3) * 2.f * err * p_hat * ((centers[k] - cr) - dy)) * inv_b;
    }
    ce = warp_sum(ce);
    if (lane == 0) part[b] = make_float2(ce, err * err);
}

// Gradients of the layer y = W x from dz = dL/dy: blocks [0, n_w) are tiles of
// dL/dW [K, D] (column-major over the D tiles; the first D tile also gives dL/dbias), blocks
// [n_w, n_w + n_x) tiles of dL/dx [B, D], and one last block the loss.  gate (or NULL):
// dL/dx counts only where gate > 0 (the ReLU's derivative of the layer below).
struct LayerGradArgs {
    GemmSide dz_k;      // rows = bins, k = prompts (side contiguous)
    GemmSide dz_b;      // rows = prompts, k = bins (k contiguous)
    GemmSide x_d, w_d;  // rows = D columns, k = prompts / bins (side contiguous)
    int B, K;
    int64_t D;
    int n_wk, n_w, n_x;
    float* grad_W;
    float* grad_bias;
    float* grad_x;
    const float* gate;
    const float2* part;
    float lambda3;
    float* loss;
};
using GradWTile = SgemmTile<2, 4, 32, false, false>;
using GradXTile = SgemmTile<2, 4, 32, true, false>;
__global__ void __launch_bounds__(256) layer_grad_kernel(const LayerGradArgs a) {
    constexpr int kFloats = GradWTile::kSmemFloats > GradXTile::kSmemFloats ? GradWTile::kSmemFloats
                                                                            : GradXTile::kSmemFloats;
    __shared__ __align__(16) float sm[kFloats];
    chain_launches();
    int blk = blockIdx.x;
    if (blk < a.n_w) {
        const int64_t k0 = (int64_t)(blk % a.n_wk) * GradWTile::BM, d0 = (int64_t)(blk / a.n_wk) * GradWTile::BN;
        GradWTile t;
        float db = 0.f;
        if (d0 == 0) t.template run<true>(sm, a.dz_k, k0, a.x_d, d0, 0, a.B, &db);
        else t.run(sm, a.dz_k, k0, a.x_d, d0, 0, a.B);
        if (a.grad_bias && d0 == 0 && threadIdx.x < GradWTile::BM && k0 + threadIdx.x < a.K)
            a.grad_bias[k0 + threadIdx.x] = db;
        if (!a.grad_W) return;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int64_t k = k0 + t.row(i), d = d0 + t.col(0);
            if (k >= a.K) continue;
            const float v[4] = {t.c[i][0].x, t.c[i][0].y, t.c[i][1].x, t.c[i][1].y};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (d + j < a.D) a.grad_W[k * a.D + d + j] = v[j];
        }
        return;
    }
    blk -= a.n_w;
    if (blk < a.n_x) {
        const int64_t n_bt = (a.B + GradXTile::BM - 1) / GradXTile::BM;
        const int64_t b0 = (blk % n_bt) * GradXTile::BM, d0 = (blk / n_bt) * GradXTile::BN;
        GradXTile t;
        t.run(sm, a.dz_b, b0, a.w_d, d0, 0, a.K);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int64_t b = b0 + t.row(i), d = d0 + t.col(0);
            if (b >= a.B) continue;
            const float v[4] = {t.c[i][0].x, t.c[i][0].y, t.c[i][1].x, t.c[i][1].y};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (d + j < a.D)
                    a.grad_x[b * a.D + d + j] = a.gate && !(a.gate[b * a.D + d + j] > 0.f) ? 0.f : v[j];
        }
        return;
    }
    // the loss: batch means of the CE and squared-error terms (256 strided sums, then a tree)
    float ce = 0.f, se = 0.f;
    for (int b = threadIdx.x; b < a.B; b += 256) {
        const float2 p = a.part[b];
        ce += p.x;
        se += p.y;
    }
    ce = warp_sum(ce);
    se = warp_sum(se);
    if ((threadIdx.x & 31) == 0) {
        sm[threadIdx.x >> 5] = ce;
        sm[8 + (threadIdx.x >> 5)] = se;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ce = se = 0.f;
        for (int w = 0; w < 8; ++w) {
            ce += sm[w];
            se += sm[8 + w];
        }
        a.loss[0] = (a.lambda3 * ce + (1.f - a.lambda3) * se) / (float)a.B;
    }
}

// out[m, n] = sum_k A(m, k) B(n, k) (+ bias[n], then max with 0, when kRelu): block (n tile of
// 64, m tile, rank of the cluster along k).  The ranks' tiles meet in shared memory, and each
// rank adds its share of the rows over all ranks in rank order.
template <int TM, int BK, bool kAlongB>
using WideTile = SgemmTile<TM, 4, BK, true, kAlongB>;

template <int TM, int BK, bool kAlongB, bool kRelu>
__global__ void __launch_bounds__(256, 2) wide_gemm_kernel(GemmSide A, GemmSide Bm, int64_t n_k,
                                                           const float* __restrict__ bias,
                                                           float* __restrict__ out) {
    using T = WideTile<TM, BK, kAlongB>;
    constexpr int SC = T::BN + 4;
    __shared__ __align__(16) float sm[T::kSmemFloats > T::BM * SC ? T::kSmemFloats : T::BM * SC];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)blockIdx.z, ranks = (int)gridDim.z;  // the cluster spans z
    const int64_t n0 = (int64_t)blockIdx.x * T::BN, m0 = (int64_t)blockIdx.y * T::BM;
    // the share's divisions before the wait for the launch before this one: 64 prompts, D and F 1024,
    // training step 48.2 us with them after it, 46.7
    const int64_t k0 = rank_begin(n_k, BK, rank, ranks), k1 = rank_begin(n_k, BK, rank + 1, ranks);
    chain_launches();
    T t;
    t.run(sm, A, m0, Bm, n0, k0, k1);
#pragma unroll
    for (int i = 0; i < TM; ++i)
        *reinterpret_cast<float4*>(sm + t.row(i) * SC + t.col(0)) =
            make_float4(t.c[i][0].x, t.c[i][0].y, t.c[i][1].x, t.c[i][1].y);
    cl.sync();
    const int rows = T::BM / ranks;
    for (int e = threadIdx.x; e < rows * T::BN; e += 256) {
        const int r = rank * rows + e / T::BN, x = e % T::BN;
        const int64_t m = m0 + r, n = n0 + x;
        if (m >= A.rows || n >= Bm.rows) continue;
        float v = 0.f;
        for (int j = 0; j < ranks; ++j) v += cl.map_shared_rank(sm, j)[r * SC + x];
        if (kRelu) {
            v += bias ? bias[n] : 0.f;
            v = v > 0.f ? v : 0.f;
        }
        out[m * Bm.rows + n] = v;
    }
    cl.sync();  // no CTA leaves while another reads its tile
}

// dL/dW1[f, x] = sum_b g[b, f] h[b, x] and dL/db1[f] = sum_b g[b, f] (by the first x tile).
// Either output may be NULL.
using OuterTile = SgemmTile<8, 4, 16, false, false>;
__global__ void __launch_bounds__(256, 2) outer_kernel(GemmSide g, GemmSide h, int64_t B, int vec,
                                                       float* __restrict__ gW, float* __restrict__ gb) {
    __shared__ __align__(16) float sm[OuterTile::kSmemFloats];
    chain_launches();
    const int64_t x0 = (int64_t)blockIdx.x * OuterTile::BN, f0 = (int64_t)blockIdx.y * OuterTile::BM;
    OuterTile t;
    if (x0 == 0 && gb) {
        float db = 0.f;
        t.template run<true>(sm, g, f0, h, x0, 0, B, &db);
        if (threadIdx.x < OuterTile::BM && f0 + threadIdx.x < g.rows) gb[f0 + threadIdx.x] = db;
    } else {
        t.run(sm, g, f0, h, x0, 0, B);
    }
    if (!gW) return;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t f = f0 + t.row(i), x = x0 + t.col(0);
        if (f >= g.rows) continue;
        float* o = gW + f * h.rows + x;
        const float4 v = make_float4(t.c[i][0].x, t.c[i][0].y, t.c[i][1].x, t.c[i][1].y);
        if (vec && x + 4 <= h.rows) {
            *reinterpret_cast<float4*>(o) = v;
        } else {
            if (x < h.rows) o[0] = v.x;
            if (x + 1 < h.rows) o[1] = v.y;
            if (x + 2 < h.rows) o[2] = v.z;
            if (x + 3 < h.rows) o[3] = v.w;
        }
    }
}

// u[b, f] = max(sum_x W1[f, x] h[b, x] + b1[f], 0) for a batch of at most NB prompts: one warp a
// hidden unit, lanes along D, then a fixed butterfly.  With so few prompts
// reading W1 is the bound, and a tile of wide_gemm_kernel has only a slice of it in flight (one
// prompt, 4096 x 1024: 31 us cold, which is 0.5 TB/s).  Prediction through the MLP, F 1024, with that
// kernel and with this one: 1 prompt, D 4096, 32 bins 35.7 and 18.5 us; 4 prompts, D 8192, 128 bins
// 65.8 and 35.0; 8 prompts, D 4096, 32 bins 37.0 and 24.7, with cold caches 39.9 and 37.9.  For 16
// prompts the tiles are as good, with cold caches better (35.8 against 39.9).
constexpr int kRowBatch = 8;
template <int NB>
__global__ void __launch_bounds__(128) hidden_rows_kernel(GemmSide h, GemmSide w, int64_t D,
                                                          const float* __restrict__ bias, float* __restrict__ u) {
    chain_launches();
    const int lane = threadIdx.x & 31;
    const int64_t f = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (f >= w.rows) return;
    float2 acc[NB][2];
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
    // a lane takes four of every 128 columns: neighbouring ones, in one load, where the rows allow it
    // (D then is a multiple of 4), else each 32 apart, so that a load covers 128 bytes of the row
    const auto add = [&](auto vec) {
        const auto four = [&](const float* row, int64_t x) {
            if constexpr (decltype(vec)::value) return *reinterpret_cast<const float4*>(row + x);
            return make_float4(row[x], x + 32 < D ? row[x + 32] : 0.f, x + 64 < D ? row[x + 64] : 0.f,
                               x + 96 < D ? row[x + 96] : 0.f);
        };
        for (int64_t x = decltype(vec)::value ? 4 * lane : lane; x < D; x += 128) {
            // every load of the pass first (prompts past the batch count as zero), then the FMAs
            const float4 wv = four(w.p + f * w.ld, x);
            float4 hv[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) hv[j] = j < h.rows ? four(h.p + j * h.ld, x) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                acc[j][0] = __ffma2_rn(make_float2(wv.x, wv.y), make_float2(hv[j].x, hv[j].y), acc[j][0]);
                acc[j][1] = __ffma2_rn(make_float2(wv.z, wv.w), make_float2(hv[j].z, hv[j].w), acc[j][1]);
            }
        }
    };
    if (h.vec && w.vec) add(std::true_type{});
    else add(std::false_type{});
    const float b = bias ? bias[f] : 0.f;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        const float v = warp_sum((acc[j][0].x + acc[j][0].y) + (acc[j][1].x + acc[j][1].y)) + b;
        if (lane == 0 && j < h.rows) u[j * w.rows + f] = v > 0.f ? v : 0.f;
    }
}

// A matrix with `rows` rows of `n` contiguous floats: as an operand whose side is the rows
// (k along a row) or whose side is the columns (k over the rows).
GemmSide side_rows(const float* p, int64_t rows, int64_t n) {
    return GemmSide{p, n, rows, n % 4 == 0 && aligned16(p) ? 1 : 0};
}
GemmSide side_cols(const float* p, int64_t n) { return side_rows(p, n, n); }

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), dim3 grid, int threads, cudaStream_t st, bool dependent, int cluster_z,
                   Args... args) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cfg.attrs = attr;
    if (dependent) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster_z > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = 1;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = (unsigned)cluster_z;
    }
    return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Splits of a layer's contraction in logit_part_kernel: enough blocks of 32 x 32 logits to
// occupy every SM twice, none shorter than one slice.
struct LogitSplit {
    int n, len;
};
LogitSplit logit_split(const estp_ctx* ctx, int B, int K, int64_t D) {
    const int64_t tiles = (int64_t)ceil_div(B, LogitTile::BM) * ceil_div(K, LogitTile::BN);
    int64_t n = 2 * ctx->num_sms / tiles;
    n = n < 1 ? 1 : n;
    const int64_t slices = (D + 63) / 64;
    if (n > slices) n = slices;
    const int64_t len = (slices + n - 1) / n * 64;
    return LogitSplit{ceil_div(D, len), (int)len};
}

// Logits of x [B, D] through W [K, D], then the head: dz and part (training) or pred / probs.
cudaError_t head_forward(estp_ctx* ctx, const float* x, int B, int64_t D, const float* W, const float* bias,
                         const float* centers, int K, const float* targets, float lambda3, LogitSplit sp,
                         float* zpart, float* dz, float2* part, float* pred, float* probs, bool dependent,
                         cudaStream_t st) {
    cudaError_t e = launch(logit_part_kernel,
                           dim3((unsigned)ceil_div(B, LogitTile::BM), (unsigned)ceil_div(K, LogitTile::BN), (unsigned)sp.n),
                           256, st, dependent, 1, side_rows(x, B, D), side_rows(W, K, D), D, sp.len, zpart);
    if (e != cudaSuccess) return e;
    return launch(head_loss_kernel, dim3((unsigned)B), kLossThreads, st, true, 1, (const float*)zpart, sp.n, bias, centers,
                  K, targets, B, lambda3, dz, part, pred, probs);
}

// Gradients of that layer (grad_x gated by `gate` when given) and the loss.
cudaError_t layer_grads(const float* x, int B, int64_t D, const float* W, int K, const float* dz,
                        const float2* part, float lambda3, float* loss, float* grad_W, float* grad_bias,
                        float* grad_x, const float* gate, cudaStream_t st) {
    LayerGradArgs a{};
    a.dz_k = side_cols(dz, K);
    a.dz_b = side_rows(dz, B, K);
    a.x_d = side_cols(x, D);
    a.w_d = side_cols(W, D);
    a.B = B; a.K = K; a.D = D;
    a.n_wk = ceil_div(K, GradWTile::BM);
    a.n_w = grad_W ? a.n_wk * ceil_div(D, GradWTile::BN) : grad_bias ? a.n_wk : 0;
    a.n_x = grad_x ? ceil_div(B, GradXTile::BM) * ceil_div(D, GradXTile::BN) : 0;
    a.grad_W = grad_W; a.grad_bias = grad_bias; a.grad_x = grad_x; a.gate = gate;
    a.part = part; a.lambda3 = lambda3; a.loss = loss;
    return launch(layer_grad_kernel, dim3((unsigned)(a.n_w + a.n_x + 1)), 256, st, true, 1, a);
}

// Rows of tiles of `side` rows that one launch covers: the y extent of a grid stops at 65535.
int64_t rows_a_launch(int side) { return (int64_t)65535 * side; }

// out [M, N] of wide_gemm_kernel.  The tile height follows M (a batch of prompts), so that a
// small batch does not multiply padding; the cluster's width: wide_ranks.
template <bool kAlongB, bool kRelu>
cudaError_t wide_gemm(estp_ctx* ctx, const GemmSide& A, const GemmSide& Bm, int64_t n_k, const float* bias,
                      float* out, bool dependent, cudaStream_t st) {
    const int64_t M = A.rows, N = Bm.rows;
    const int tm = M > 64 ? 8 : M > 32 ? 4 : M > 16 ? 2 : 1;
    const int S = wide_ranks((int64_t)ceil_div(N, 64) * ceil_div(M, 16 * tm), n_k, ctx->num_sms);
    cudaError_t e = cudaSuccess;
    for (int64_t m = 0; m < M && e == cudaSuccess; m += rows_a_launch(16 * tm)) {
        const int64_t rows = M - m < rows_a_launch(16 * tm) ? M - m : rows_a_launch(16 * tm);
        const GemmSide a{A.p + m * A.ld, A.ld, rows, A.vec};
        const dim3 grid((unsigned)ceil_div(N, 64), (unsigned)ceil_div(rows, 16 * tm), (unsigned)S);
        auto go = [&](auto kern) {
            return launch(kern, grid, 256, st, dependent || m > 0, S, a, Bm, n_k, bias, out + m * N);
        };
        e = tm == 8 ? go(wide_gemm_kernel<8, 16, kAlongB, kRelu>)
          : tm == 4 ? go(wide_gemm_kernel<4, 32, kAlongB, kRelu>)
          : tm == 2 ? go(wide_gemm_kernel<2, 32, kAlongB, kRelu>)
                    : go(wide_gemm_kernel<1, 64, kAlongB, kRelu>);
    }
    return e;
}

// The hidden layer u = max(W1 h + b1, 0), the first launch of its call.
cudaError_t hidden_layer(estp_ctx* ctx, const float* pooled, int B, int64_t D, const estp_mlp_head& head, float* u,
                         cudaStream_t st) {
    const GemmSide h = side_rows(pooled, B, D), w = side_rows(head.W1, head.F, D);
    if (B > kRowBatch) return wide_gemm<true, true>(ctx, h, w, D, head.b1, u, false, st);
    auto go = [&](auto kern) { return launch(kern, dim3((unsigned)ceil_div(head.F, 4)), 128, st, false, 1, h, w, D, head.b1, u); };
    return B > 4 ? go(hidden_rows_kernel<8>) : B > 2 ? go(hidden_rows_kernel<4>)
         : B > 1 ? go(hidden_rows_kernel<2>) : go(hidden_rows_kernel<1>);
}

}  // namespace

estp_status launch_head_loss(estp_ctx* ctx, const float* pooled, int B, int64_t D,
                             const estp_head& head, const float* targets, float lambda3,
                             float* loss, float* grad_W, float* grad_bias, float* grad_pooled,
                             cudaStream_t st) {
    const int K = head.K;
    const LogitSplit sp = logit_split(ctx, B, K, D);
    // workspace: dz [B, K] | part [B] | partial logits [splits, B, K]
    const size_t off_part = align_up(sizeof(float) * (size_t)B * K, 256);
    const size_t off_z = off_part + align_up(sizeof(float2) * (size_t)B, 256);
    estp_status s = ws_reserve(ctx, off_z + sizeof(float) * (size_t)sp.n * B * K);
    if (s != ESTP_OK) return s;
    char* ws = static_cast<char*>(ctx->ws);
    float* dz = reinterpret_cast<float*>(ws);
    float2* part = reinterpret_cast<float2*>(ws + off_part);
    cudaError_t e = head_forward(ctx, pooled, B, D, head.W, head.bias, head.centers, K, targets, lambda3, sp,
                                 reinterpret_cast<float*>(ws + off_z), dz, part, nullptr, nullptr, false, st);
    if (e != cudaSuccess) return cuda_fail(e, "head forward launch");
    e = layer_grads(pooled, B, D, head.W, K, dz, part, lambda3, loss, grad_W, grad_bias, grad_pooled, nullptr, st);
    if (e != cudaSuccess) return cuda_fail(e, "head gradient launch");
    e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "head loss launch");
}

estp_status launch_mlp_head_predict(estp_ctx* ctx, const float* pooled, int B, int64_t D,
                                    const estp_mlp_head& head, float* pred, float* probs,
                                    cudaStream_t st) {
    const int F = head.F, K = head.K;
    const LogitSplit sp = logit_split(ctx, B, K, F);
    // workspace: u [B, F] | partial logits
    const size_t off_z = align_up(sizeof(float) * (size_t)B * F, 256);
    estp_status s = ws_reserve(ctx, off_z + sizeof(float) * (size_t)sp.n * B * K);
    if (s != ESTP_OK) return s;
    char* ws = static_cast<char*>(ctx->ws);
    float* u = reinterpret_cast<float*>(ws);
    cudaError_t e = hidden_layer(ctx, pooled, B, D, head, u, st);
    if (e != cudaSuccess) return cuda_fail(e, "mlp hidden launch");
    e = head_forward(ctx, u, B, F, head.W2, head.b2, head.centers, K, nullptr, 0.f, sp,
                     reinterpret_cast<float*>(ws + off_z), nullptr, nullptr, pred, probs, true, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "mlp head launch");
}

estp_status launch_mlp_head_loss(estp_ctx* ctx, const float* pooled, int B, int64_t D,
                                 const estp_mlp_head& head, const float* targets, float lambda3,
                                 float* loss, const estp_mlp_grads& g, cudaStream_t st) {
    const int F = head.F, K = head.K;
    const LogitSplit sp = logit_split(ctx, B, K, F);
    // workspace: u [B, F] | g = dL/du where u > 0 [B, F] | dz [B, K] | part [B] | partial logits
    const size_t off_g = align_up(sizeof(float) * (size_t)B * F, 256);
    const size_t off_dz = 2 * off_g;
    const size_t off_part = off_dz + align_up(sizeof(float) * (size_t)B * K, 256);
    const size_t off_z = off_part + align_up(sizeof(float2) * (size_t)B, 256);
    estp_status s = ws_reserve(ctx, off_z + sizeof(float) * (size_t)sp.n * B * K);
    if (s != ESTP_OK) return s;
    char* ws = static_cast<char*>(ctx->ws);
    float* u = reinterpret_cast<float*>(ws);
    float* gu = reinterpret_cast<float*>(ws + off_g);
    float* dz = reinterpret_cast<float*>(ws + off_dz);
    float2* part = reinterpret_cast<float2*>(ws + off_part);
    const bool lower = g.W1 || g.b1 || g.pooled;  // gradients below the hidden layer
    cudaError_t e = hidden_layer(ctx, pooled, B, D, head, u, st);
    if (e != cudaSuccess) return cuda_fail(e, "mlp hidden launch");
    e = head_forward(ctx, u, B, F, head.W2, head.b2, head.centers, K, targets, lambda3, sp,
                     reinterpret_cast<float*>(ws + off_z), dz, part, nullptr, nullptr, true, st);
    if (e != cudaSuccess) return cuda_fail(e, "mlp head launch");
    // second layer: dL/dW2, dL/db2, dL/du through the ReLU, and the loss
    e = layer_grads(u, B, F, head.W2, K, dz, part, lambda3, loss, g.W2, g.b2, lower ? gu : nullptr, u, st);
    if (e != cudaSuccess) return cuda_fail(e, "mlp second-layer gradient launch");
    if (g.W1 || g.b1) {  // first layer: dL/dW1, dL/db1
        const GemmSide h = side_cols(pooled, D), gs = side_cols(gu, F);
        const int vec = h.vec && (!g.W1 || aligned16(g.W1)) ? 1 : 0;
        for (int64_t f = 0; f < F && e == cudaSuccess; f += rows_a_launch(OuterTile::BM)) {
            const int64_t rows = F - f < rows_a_launch(OuterTile::BM) ? F - f : rows_a_launch(OuterTile::BM);
            e = launch(outer_kernel, dim3((unsigned)(g.W1 ? ceil_div(D, OuterTile::BN) : 1), (unsigned)ceil_div(rows, OuterTile::BM)),
                       256, st, true, 1, GemmSide{gs.p + f, gs.ld, rows, gs.vec}, h, (int64_t)B, vec,
                       g.W1 ? g.W1 + f * D : nullptr, g.b1 ? g.b1 + f : nullptr);
        }
        if (e != cudaSuccess) return cuda_fail(e, "mlp first-layer gradient launch");
    }
    if (g.pooled) {  // dL/dpooled = W1^T g
        e = wide_gemm<false, false>(ctx, side_rows(gu, B, F), side_cols(head.W1, D), F, nullptr, g.pooled, true, st);
        if (e != cudaSuccess) return cuda_fail(e, "mlp input-gradient launch");
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? ESTP_OK : cuda_fail(e, "mlp head loss launch");
}

}  // namespace estp
