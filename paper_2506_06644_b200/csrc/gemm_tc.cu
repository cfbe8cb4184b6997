// Dense projection for 2..64 tokens with bf16 weights on the fifth-generation tensor cores:
// y[b][:] = Wt . f(x[b][:]) (+ y_add[b][:]), f = optional division per group, optional RMSNorm -- the
// decoder layer's QKV and output projections for a batch or a chunk of a prompt, the LM head of a batch.  Two kernels:
//   prep   f(x) -> two bf16 terms (x = hi + lo, 16 significant bits) in the workspace, three (all 24 bits) for up to four tokens;
//          the addend (or 0) into those output tiles that two or more blocks of the GEMM share; the caller's clear-region side job
//   gemm   the weight-streaming GEMM of stream_gemm.cuh, any number of output rows and any n_in (multiple of 8; TMA fills what
//          lies outside with zeros); a tile that one block holds whole is stored, a shared one reduced into y
// Row counts that are no multiple of 128 used to take the mma.sync kernels: 105401 x 2048, 64 tokens, 375 -> 81 us; 5 tokens
// 76 -> 70.  The 256000 x 2304 head went from whole tiles per block and a wave of blocks per 148 of them to a persistent
// sequence: 64 tokens 256 -> 201 us, 8 tokens 201 -> 181.  Two to four tokens were bound by the plain ALUs: 256000 x 2304, 2 tokens,
// 261 -> 177 us; 16000 x 2304 26.3 -> 18.2; 4096 x 2304 12.4 -> 9.7; 1000 x 1000 6.2 both.
#include "kernels.h"
#include "stream_gemm.cuh"

using namespace spark;
using namespace spark::tc;

namespace {

constexpr int kGemmMaxTok = 64;
constexpr int kGemmPrepSplit = 4;

struct GemmParams {
    const float* x;
    const float* norm_w;
    float eps;
    int B, n_in, n_out;
    const float* y_add;
    float* y;
    const float* x_div;
    int x_div_group;
    uint4* zero_ptr;
    int zero_n16;
    __nv_bfloat16* xs;       // [xrows][n_in]
    StreamPlan sp;
    WsHeader* hdr;
};

// Four blocks per (padded) token row, a quarter of the row each.
template <bool FEW>
__global__ void __launch_bounds__(256) gemm_tc_prep_kernel(const GemmParams p) {
    __shared__ float red[8];
    const int n = blockIdx.x / kGemmPrepSplit, qr = blockIdx.x % kGemmPrepSplit, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_in = p.n_in, w4 = n_in / 4;
    const int q0 = static_cast<int>(static_cast<int64_t>(qr) * w4 / kGemmPrepSplit), q1 = static_cast<int>(static_cast<int64_t>(qr + 1) * w4 / kGemmPrepSplit);
    dep_wait();
    dep_trigger();
    for (int i = blockIdx.x * 256 + tid; i < p.zero_n16; i += gridDim.x * 256) p.zero_ptr[i] = make_uint4(0u, 0u, 0u, 0u);
    if (p.y_add != p.y) {            // shared tiles start from the addend (or 0); when they alias y already holds it
        if (p.sp.split > 1) {        // every tile is shared
            const int64_t total = static_cast<int64_t>(p.B) * p.n_out, t0 = static_cast<int64_t>(blockIdx.x) * 256 + tid, step = static_cast<int64_t>(gridDim.x) * 256;
            if ((p.n_out & 3) == 0 && ((reinterpret_cast<uintptr_t>(p.y) | reinterpret_cast<uintptr_t>(p.y_add)) & 15u) == 0) {
                const float4* ya = reinterpret_cast<const float4*>(p.y_add);
                for (int64_t i = t0; i < total / 4; i += step) reinterpret_cast<float4*>(p.y)[i] = ya != nullptr ? ya[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                for (int64_t i = t0; i < total; i += step) p.y[i] = p.y_add != nullptr ? p.y_add[i] : 0.f;
            }
        } else if (p.sp.split == 0 && p.sp.per == 0) {
            for (int g = 1 + blockIdx.x; g < p.sp.grid; g += gridDim.x) {
                const StreamPart part = stream_part(p.sp, g), ahead = stream_part(p.sp, g - 1);
                if (part.c == 0 || (ahead.tile == part.tile && ahead.c > 0)) continue;      // between two tiles, or not the tile's first cut
                const int row = part.tile * kStreamRows + (tid & 127);
                if (row < p.n_out)
                    for (int b = tid >> 7; b < p.B; b += 2) {
                        const int64_t at = static_cast<int64_t>(b) * p.n_out + row;
                        p.y[at] = p.y_add != nullptr ? p.y_add[at] : 0.f;
                    }
            }
        }
    }
    if (n >= p.B) return;            // rows of padding tokens may hold anything: their columns of the product are not looked at
    const float4* xr = reinterpret_cast<const float4*>(p.x + static_cast<int64_t>(n) * n_in);
    auto divided = [&](int c4) -> float4 {
        float4 v = xr[c4];
        if (p.x_div != nullptr) {
            const float dv = p.x_div[static_cast<int64_t>(n) * (n_in / p.x_div_group) + (c4 * 4) / p.x_div_group];
            const float inv = dv > 0.f ? 1.f / dv : 0.f;
            v = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
        }
        return v;
    };
    float sc = 1.f;
    if (p.norm_w != nullptr) {       // every quarter sums the whole (divided) row
        float ss = 0.f;
        for (int i = tid; i < w4; i += 256) {
            const float4 v = divided(i);
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        ss = warp_sum(ss);
        if (lane == 0) red[warp] = ss;
        __syncthreads();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += red[w];
        sc = rsqrtf(tot / static_cast<float>(n_in) + p.eps);
    }
    for (int i = q0 + tid; i < q1; i += 256) {
        float4 v = divided(i);
        if (p.norm_w != nullptr) {
            const float4 w = reinterpret_cast<const float4*>(p.norm_w)[i];
            v = make_float4(v.x * sc * w.x, v.y * sc * w.y, v.z * sc * w.z, v.w * sc * w.w);
        }
        uint2 h, m, l;
        uint2* row = reinterpret_cast<uint2*>(p.xs + static_cast<int64_t>(n) * n_in) + i;
        const int64_t term = static_cast<int64_t>(p.sp.ntok) * (n_in / 4);
        if (FEW) {
            split_pair3(v.x, v.y, h.x, m.x, l.x);
            split_pair3(v.z, v.w, h.y, m.y, l.y);
            row[2 * term] = l;
        } else {
            split_pair(v.x, v.y, h.x, m.x);
            split_pair(v.z, v.w, h.y, m.y);
        }
        row[0] = h;
        row[term] = m;
    }
}

template <bool FEW>
__global__ void __launch_bounds__(kTcThreads, 1)
gemm_tc_kernel(const GemmParams p, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ StreamShared sh;
    stream_gemm<FEW ? kStreamFew : 0>(p.sp, sh, tc_raw, &map_w, &map_x, p.hdr, [] {}, [&](int tile, bool whole, int r, int n0, const float (&v)[16]) {
        const int row = tile * kStreamRows + r;
        if (row >= p.n_out) return;
        const int64_t at = static_cast<int64_t>(n0) * p.n_out + row;
#pragma unroll
        for (int i = 0; i < (FEW ? 4 : 16); ++i)
            if (n0 + i < p.B) {
                float* y = p.y + at + static_cast<int64_t>(i) * p.n_out;
                if (!whole) atomicAdd(y, v[i]);
                else *y = p.y_add != nullptr ? v[i] + p.y_add[at + static_cast<int64_t>(i) * p.n_out] : v[i];
            }
    });
}

}  // namespace

namespace spark {

// SPARK_ERR_WORKSPACE = shape or workspace not served by this path (the caller falls back).
int gemm_tc_launch(spark_ctx* ctx, const GemvArgs& a, cudaStream_t stream) {
    if (a.wdtype != SPARK_BF16 || a.B < 2 || a.B > kGemmMaxTok || (a.n_in & 7) != 0 || a.n_in < kChunk) return SPARK_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(a.Wt) & 15u) != 0) return SPARK_ERR_WORKSPACE;
    GemmParams p;
    const bool few = a.B <= 4;
    const int64_t call = (a.n_in + kChunk - 1) / kChunk, tiles = (a.n_out + kStreamRows - 1) / kStreamRows;
    if (tiles * call >= (1LL << 30)) return SPARK_ERR_WORKSPACE;
    const size_t limit = static_cast<size_t>(ctx->max_smem_optin) - sizeof(StreamShared) - 64;
    if (!stream_plan(p.sp, ctx->num_sms, static_cast<int>(tiles), static_cast<int>(call), static_cast<int>(a.B), limit, false, kStreamRows, few)) return SPARK_ERR_WORKSPACE;
    // the split input sits behind the attention's cells, where the FFN chunk path keeps its own (neither outlives its call)
    const size_t xb = static_cast<size_t>(p.sp.xrows) * a.n_in * 2;
    if (ctx->scratch == nullptr || ctx->scratch_bytes < kAttnCellBytes + xb) return SPARK_ERR_WORKSPACE;

    p.x = a.x; p.norm_w = a.norm_w; p.eps = a.rms_eps;
    p.B = static_cast<int>(a.B); p.n_in = static_cast<int>(a.n_in); p.n_out = static_cast<int>(a.n_out);
    p.y_add = a.y_add; p.y = a.y;
    p.x_div = a.x_div; p.x_div_group = static_cast<int>(a.x_div ? a.x_div_group : 1);
    p.zero_ptr = static_cast<uint4*>(a.zero_ptr); p.zero_n16 = static_cast<int>(a.zero_bytes / 16);
    p.xs = reinterpret_cast<__nv_bfloat16*>(ctx->scratch + kAttnCellBytes);
    p.hdr = ctx->hdr;

    CUtensorMap m_w, m_x;
    if (!make_map(&m_w, a.Wt, a.n_out, a.n_in, a.n_in, kStreamRows, true) ||
        !make_map(&m_x, p.xs, p.sp.xrows, a.n_in, a.n_in, p.sp.xrows, false))
        return SPARK_ERR_WORKSPACE;
    const void* kern = few ? reinterpret_cast<const void*>(gemm_tc_kernel<true>) : reinterpret_cast<const void*>(gemm_tc_kernel<false>);
    const void* prep = few ? reinterpret_cast<const void*>(gemm_tc_prep_kernel<true>) : reinterpret_cast<const void*>(gemm_tc_prep_kernel<false>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(limit)) != cudaSuccess) return SPARK_ERR_CUDA;
    {
        void* args[] = {&p};
        if (launch_kernel(ctx, prep, static_cast<unsigned>((few ? 16 : p.sp.ntok) * kGemmPrepSplit), 256, 0, stream, false, args) != cudaSuccess)
            return SPARK_ERR_CUDA;
    }
    {
        void* args[] = {&p, &m_w, &m_x};
        if (launch_kernel(ctx, kern, static_cast<unsigned>(p.sp.grid), kTcThreads, stream_smem(p.sp), stream, false, args, true) != cudaSuccess)
            return SPARK_ERR_CUDA;
    }
    return SPARK_OK;
}

}  // namespace spark
