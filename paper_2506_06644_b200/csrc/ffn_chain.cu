// Spark FFN (Section 2.1, Eq. 2) for 5..16 tokens of a small model with bf16 weights, on the fifth-generation tensor cores: the
// products of ffn_tc.cu as four kernels, chained by programmatic launches (no block waits on another block):
//   prep    RMSNorm scale (optional), x -> two bf16 terms (x = hi + lo), sums cleared
//   scores  S = K1t . X[:, :r]^T, a block per tile of neurons (stream_gemm.cuh); per-token score sums for Eq. 11
//   act     T = K2t . X[:, r:]^T the same way, started while the scores are still being formed: only its epilogue waits for them;
//           theta per token (Eq. 10/11), U = [S > theta] . GELU(S - theta) . T as two bf16 terms, counts and index lists
//   out     Y^T += Vt^T . U, K = neurons split over blocks, fp32 reductions into y
// Where the weights are a few megabytes nothing but latencies is left, and a launch whose blocks are in place when the kernel ahead
// ends costs less than a grid-wide barrier.  d = 256, d_ff = 1024, 5 tokens: 14.4 us, the one kernel of ffn_tc.cu 16.3; 64 tokens 22.6
// and 20.5; d = 512, d_ff = 3000, 5 tokens: 14.4 and 16.4, 20 tokens 18.4 and 18.5; d = 2304, d_ff = 9216, 5 tokens: 28.7 and 26.8.
#include "ffn_params.h"
#include "kernels.h"
#include "stream_gemm.cuh"

using namespace spark;
using namespace spark::tc;

namespace {

constexpr int kTok = 16;              // token rows of the padded operands: one group of an epilogue
constexpr int kSumWays = 16;
constexpr int kMinRows = 32;          // neurons of a tile at least: every tile reads all of X

struct ChainParams {
    FfnParams f;
    double* sums;                 // [kSumWays][kTok][2]
    __nv_bfloat16* xs;            // [2 kTok][d]: hi rows, lo rows
    float* S;                     // [kTok][d_ff] scores, token-major
    __nv_bfloat16* us;            // [2 kTok][d_ff]
    StreamPlan sp;                // of the kernel's product
};
inline size_t sums_bytes() { return sizeof(double) * kSumWays * kTok * 2; }
inline size_t xs_bytes(int64_t d) { return round_up(static_cast<size_t>(2 * kTok) * d * 2, 1024); }
inline size_t s_bytes(int64_t d_ff) { return round_up(static_cast<size_t>(kTok) * d_ff * 4, 1024); }

// ---- prep: four blocks per token row, a quarter of the row each ----------------------------------------------
constexpr int kPrepSplit = 4;
__global__ void __launch_bounds__(256) ffn_chain_prep_kernel(const ChainParams p) {
    __shared__ float red[8];
    const int n = blockIdx.x / kPrepSplit, qr = blockIdx.x % kPrepSplit, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = p.f.d, q0 = qr * (d / 4) / kPrepSplit, q1 = (qr + 1) * (d / 4) / kPrepSplit;      // float4 of this quarter row
    dep_wait();
    dep_trigger();
    if (blockIdx.x == 0) {
        for (int i = tid; i < kSumWays * kTok * 2; i += 256) p.sums[i] = 0.0;
        if (p.f.count != nullptr && tid < p.f.B) p.f.count[tid] = 0;
    }
    const float4* xr = reinterpret_cast<const float4*>(p.f.x + static_cast<int64_t>(n) * d);
    float sc = 1.f;
    if (p.f.norm_w != nullptr) {   // every quarter sums the whole row
        float ss = 0.f;
        for (int i = tid; i < d / 4; i += 256) {
            const float4 v = xr[i];
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        ss = warp_sum(ss);
        if (lane == 0) red[warp] = ss;
        __syncthreads();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += red[w];
        sc = rsqrtf(tot / static_cast<float>(d) + p.f.eps);
    }
    uint2* hi = reinterpret_cast<uint2*>(p.xs + static_cast<int64_t>(n) * d);
    uint2* lo = reinterpret_cast<uint2*>(p.xs + static_cast<int64_t>(kTok + n) * d);       // rows of tokens that are not there may hold anything
    for (int i = q0 + tid; i < q1; i += 256) {
        float4 v = xr[i];
        if (p.f.norm_w != nullptr) {
            const float4 w = reinterpret_cast<const float4*>(p.f.norm_w)[i];
            v = make_float4(v.x * sc * w.x, v.y * sc * w.y, v.z * sc * w.z, v.w * sc * w.w);
        }
        uint2 h, l;
        split_pair(v.x, v.y, h.x, l.x);
        split_pair(v.z, v.w, h.y, l.y);
        hi[i] = h;
        lo[i] = l;
    }
}

// ---- scores ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kTcThreads, 1)
ffn_chain_scores_kernel(const ChainParams p, const __grid_constant__ CUtensorMap map_k1, const __grid_constant__ CUtensorMap map_x) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ StreamShared sh;
    __shared__ float win[4][32 * 17];                              // per epilogue warp: 32 neurons x 16 tokens
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, B = p.f.B;
    const int64_t dff = p.f.d_ff;
    stream_gemm<kStreamLate>(
        p.sp, sh, tc_raw, &map_k1, &map_x, p.f.hdr,
        [&] {   // y = y_init (or 0) while the weights stream: the output kernel adds into it
            const int total4 = B * (p.f.d / 4);
            const float4* yi = reinterpret_cast<const float4*>(p.f.y_init);
            float4* yo = reinterpret_cast<float4*>(p.f.y);
            if (p.f.y_init != p.f.y)
                for (int i = blockIdx.x * 128 + (tid - 64); i < total4; i += gridDim.x * 128) yo[i] = yi != nullptr ? yi[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        },
        [&](int tile, bool, int r, int, const float (&v)[16]) {
            const int row = tile * p.sp.rows + r;
            const bool mine = r < p.sp.rows && row < dff;
            float* w = win[warp - 2];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (i < B && mine) p.S[i * dff + row] = v[i];
                w[lane * 17 + i] = mine ? v[i] : 0.f;
            }
            __syncwarp();
            double s1 = 0.0, s2 = 0.0;                             // lane: token lane % 16, half of the neurons
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const double x = static_cast<double>(w[((lane >> 4) * 16 + i) * 17 + (lane & 15)]);
                s1 += x;
                s2 = fma(x, x, s2);
            }
            s1 += __shfl_xor_sync(kFull, s1, 16);
            s2 += __shfl_xor_sync(kFull, s2, 16);
            if ((lane & 15) < B) red_add_f64(p.sums + (((4 * tile + (warp & 3)) % kSumWays) * kTok + (lane & 15)) * 2 + (lane >> 4), lane < 16 ? s1 : s2);
            __syncwarp();
        });
}

// ---- act: T, theta, masks, U = [S > theta] . GELU(S - theta) . T in two bf16 terms ----------------------------
__global__ void __launch_bounds__(kTcThreads, 1)
ffn_chain_act_kernel(const ChainParams p, const __grid_constant__ CUtensorMap map_k2, const __grid_constant__ CUtensorMap map_x) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ StreamShared sh;
    __shared__ float theta_s[kTok];
    const int tid = threadIdx.x, lane = tid & 31, B = p.f.B;
    const int64_t dff = p.f.d_ff;
    stream_gemm<kStreamEarlyX>(
        p.sp, sh, tc_raw, &map_k2, &map_x, p.f.hdr,
        [&] {   // eight threads per token, two ways each
            const int n = (tid - 64) >> 3, part = tid & 7;
            double s1 = 0.0, s2 = 0.0;
            if (n < B) {
#pragma unroll
                for (int w = 0; w < kSumWays / 8; ++w) {
                    const double2 c = __ldcg(reinterpret_cast<const double2*>(p.sums + ((part * (kSumWays / 8) + w) * kTok + n) * 2));
                    s1 += c.x;
                    s2 += c.y;
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                s1 += __shfl_xor_sync(kFull, s1, o);
                s2 += __shfl_xor_sync(kFull, s2, o);
            }
            if (part == 0) {
                float th = INFINITY;                               // tokens that are not there
                if (n < B) {
                    th = -INFINITY;
                    if (!p.f.identity) {
                        const double mean = s1 * p.f.inv_n;
                        const float var = static_cast<float>((s2 - s1 * mean) * p.f.inv_nm1);
                        th = static_cast<float>(mean) + sqrtf(fmaxf(var, 0.f)) * static_cast<float>(p.f.z);
                    }
                    if (blockIdx.x == 0 && p.f.theta != nullptr) p.f.theta[n] = th;
                }
                theta_s[n] = th;
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");         // the four epilogue warps
        },
        [&](int tile, bool, int r, int, const float (&t)[16]) {
            const int row = tile * p.sp.rows + r;
            const bool mine = r < p.sp.rows && row < dff, odd = lane & 1;
            float u[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = i < B && mine ? __ldcg(p.S + i * dff + row) : 0.f;
            unsigned on = 0u;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float th = theta_s[i], a = p.f.identity ? u[i] : u[i] - th;
                const bool active = mine && u[i] > th;
                on |= active ? 1u << i : 0u;
                u[i] = active ? (p.f.erf_form ? gelu_erf(a) : gelu_logistic(a)) * t[i] : 0.f;
            }
            // even lanes store this pair of neurons for the even tokens, odd lanes for the odd ones
            __nv_bfloat16* uh = p.us + (odd ? 1 : 0) * dff + row - (odd ? 1 : 0);
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
                const float own = odd ? u[i + 1] : u[i], other = __shfl_xor_sync(kFull, odd ? u[i] : u[i + 1], 1);
                unsigned hi, lo;
                split_pair(odd ? other : own, odd ? own : other, hi, lo);
                if (mine && i + (odd ? 1 : 0) < B) {
                    *reinterpret_cast<unsigned*>(uh + i * dff) = hi;
                    *reinterpret_cast<unsigned*>(uh + (kTok + i) * dff) = lo;
                }
            }
            if (p.f.count != nullptr) {
                // a warp's share of a token's list is contiguous and ascending; warps take their places in the order in which they
                // get here.  Lane i asks for token i: one round trip for sixteen tokens
                unsigned b[16];
                int at = 0;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    b[i] = __ballot_sync(kFull, on >> i & 1u);
                    if (lane == i) at = __popc(b[i]);
                }
                if (at > 0) at = atomicAdd(&p.f.count[lane], at);
                if (p.f.idx != nullptr) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int first = __shfl_sync(kFull, at, i);
                        if (on >> i & 1u) p.f.idx[i * dff + first + __popc(b[i] & ((1u << lane) - 1u))] = row;
                    }
                }
            }
        });
}

// ---- out -----------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kTcThreads, 1)
ffn_chain_out_kernel(const ChainParams p, const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_u) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ StreamShared sh;
    stream_gemm<kStreamMN>(p.sp, sh, tc_raw, &map_v, &map_u, p.f.hdr, [] {}, [&](int tile, bool, int r, int n0, const float (&v)[16]) {
        const int64_t d = p.f.d, col = tile * kStreamRows + r;
        if (col >= d) return;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (n0 + i < p.f.B) atomicAdd(p.f.y + (n0 + i) * d + col, v[i]);
    });
}

}  // namespace

namespace spark {

size_t ffn_chain_workspace_bytes(int64_t d, int64_t d_ff) {
    return sums_bytes() + xs_bytes(d) + s_bytes(d_ff) + static_cast<size_t>(2 * kTok) * d_ff * 2;
}

// SPARK_ERR_WORKSPACE = shape or workspace not served by this path (the caller falls back).  The shape has passed ffn_tc_launch()'s checks.
int ffn_chain_launch(spark_ctx* ctx, FfnParams& f, cudaStream_t stream) {
    const int d = f.d, r = f.r, d_ff = f.d_ff, B = f.B, sms = ctx->num_sms;
    if (B > kTok || ctx->scratch_bytes < kAttnCellBytes + ffn_chain_workspace_bytes(d, d_ff)) return SPARK_ERR_WORKSPACE;
    ChainParams p;
    p.f = f;
    char* w = ctx->scratch + kAttnCellBytes;                       // behind the attention's persistent cells
    p.sums = reinterpret_cast<double*>(w);
    p.xs = reinterpret_cast<__nv_bfloat16*>(w + sums_bytes());
    p.S = reinterpret_cast<float*>(w + sums_bytes() + xs_bytes(d));
    p.us = reinterpret_cast<__nv_bfloat16*>(w + sums_bytes() + xs_bytes(d) + s_bytes(d_ff));
    int rows = ((d_ff + sms - 1) / sms + 7) & ~7;                  // a tile per SM
    if (rows < kMinRows) rows = kMinRows;
    if (rows > kStreamRows) rows = kStreamRows;
    const int tiles = (d_ff + rows - 1) / rows;

    CUtensorMap m_k1, m_k2, m_x1, m_x2, m_v, m_u;
    if (!make_map(&m_k1, f.K1t, d_ff, r, r, rows, true) || !make_map(&m_k2, f.K2t, d_ff, d - r, d - r, rows, true) ||
        !make_map(&m_x1, p.xs, 2 * kTok, r, d, 2 * kTok, false) || !make_map(&m_x2, p.xs + r, 2 * kTok, d - r, d, 2 * kTok, false) ||
        !make_map(&m_v, f.Vt, d_ff, d, d, kChunk, true) || !make_map(&m_u, p.us, 2 * kTok, d_ff, d_ff, 2 * kTok, false))
        return SPARK_ERR_WORKSPACE;
    auto chunks = [](int k) { return (k + kChunk - 1) / kChunk; };
    constexpr int kSmem = 72 * 1024;                               // blocks of three kernels that follow one another side by side on an SM
    auto launch = [&](const void* kern, const CUtensorMap* mw, const CUtensorMap* mx) -> int {
        void* args[] = {&p, const_cast<CUtensorMap*>(mw), const_cast<CUtensorMap*>(mx)};
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess ||
            launch_kernel(ctx, kern, static_cast<unsigned>(p.sp.grid), kTcThreads, stream_smem(p.sp), stream, false, args, true) != cudaSuccess)
            return SPARK_ERR_CUDA;
        return SPARK_OK;
    };
    if (!stream_plan(p.sp, sms, tiles, chunks(r), B, kSmem, true, rows)) return SPARK_ERR_WORKSPACE;
    {
        void* args[] = {&p};
        if (launch_kernel(ctx, reinterpret_cast<const void*>(ffn_chain_prep_kernel), static_cast<unsigned>(B * kPrepSplit), 256, 0, stream, false, args) != cudaSuccess) return SPARK_ERR_CUDA;
    }
    if (const int rc = launch(reinterpret_cast<const void*>(ffn_chain_scores_kernel), &m_k1, &m_x1); rc != SPARK_OK) return rc;
    if (!stream_plan(p.sp, sms, tiles, chunks(d - r), B, kSmem, true, rows)) return SPARK_ERR_CUDA;
    if (const int rc = launch(reinterpret_cast<const void*>(ffn_chain_act_kernel), &m_k2, &m_x2); rc != SPARK_OK) return rc;
    if (!stream_plan(p.sp, sms, (d + kStreamRows - 1) / kStreamRows, chunks(d_ff), B, kSmem)) return SPARK_ERR_CUDA;
    return launch(reinterpret_cast<const void*>(ffn_chain_out_kernel), &m_v, &m_u);
}

}  // namespace spark
