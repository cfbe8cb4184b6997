// A span of a prompt: hundreds of consecutive tokens of one sequence through a decoder layer at once (spark_prefill).
//
// A prompt in calls of 64 tokens reads every weight once per 64 tokens and pays thirteen launches of 5 to 15 us for each layer
// and chunk; what a token then sees does not depend on the chunking, so the prefill entry points take as many tokens together
// as the workspace holds (up to 1024).  The products are then bound by the tensor cores: D[rows][tokens] = W . X^T with 128 rows
// x 128 tokens per tile, X as two bf16 terms (hi | lo: one MMA of N = 256 serves both), persistent blocks over the tiles, token
// tiles fastest so that a weight tile comes from HBM once.  Every product of more than 2304 columns is cut into segments that
// alternate between two tensor-memory accumulators; the epilogue warps add the segments in fp32, which keeps the accumulator's
// truncation at 144 steps and hides the epilogue of a tile under the next one.  Kernels per layer and span:
//   prep (norm1) -> QKV -> rope (queries into operand form, cache append, quantiles) -> attention (two kernels, span_attn.cu)
//   -> prep (softmax division) -> Wo + h -> prep (norm2) -> K1 scores -> theta -> K2, whose epilogue forms
//   u = [s > theta] GELU(s - theta) t in two bf16 terms -> V + h2
// 4000 tokens through eight layers of the 2B shape: 45.9 ms in 64-token calls, 9.5 ms this way.
#include <cmath>

#include "ffn_params.h"
#include "kernels.h"
#include "stream_gemm.cuh"

using namespace spark;
using namespace spark::tc;

namespace {

constexpr int kSpanMax = 1024;        // tokens
constexpr int kSpanTile = 128;        // tokens per tile; spans are padded to a multiple of it
constexpr int kSpanStages = 4;
constexpr int kSpanStageBytes = kStreamTileBytes + 2 * kSpanTile * kChunk * 2;
constexpr int kSpanSeg = 36;          // K chunks per segment at most
constexpr uint32_t kSpanCols = 512;   // two accumulators of 128 rows x (hi | lo) tokens
constexpr int kSpanThreads = 64 + 8 * 32;      // warp 0: TMA, warp 1: MMA + tensor memory, warps 2..9: epilogue

struct SpanGemm {
    int rows, T, call;
    int tiles_t, tiles;      // token tiles; all work items: tiles, or pieces of tiles
    int split;               // pieces of a tile's K range, added into y with reductions (1: none)
    int nseg;                // segments of an item
    int lo_row;              // rows of X's second term start here
    const float* add;        // nullable [T][rows]
    float* y;                // [T][rows]
    // U form: y is not written
    const float* S;          // [T][rows]
    const float* theta;      // [T]
    int identity, erf_form;
    __nv_bfloat16* u;        // [2 * Tp][rows]: hi rows, lo rows
    WsHeader* hdr;
};

struct SpanShared {
    unsigned long long full[kSpanStages], empty[kSpanStages];
    unsigned long long acc_full[2], acc_empty[2];
    uint32_t tmem;
    int abort_flag;
};

// MN: the matrix is stored [K][rows] (V); U: the epilogue forms the activations.
template <bool MN, bool U>
__global__ void __launch_bounds__(kSpanThreads, 1)
span_gemm_kernel(const SpanGemm p, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ SpanShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 64) {
        tma_prefetch_desc(&map_w);
        tma_prefetch_desc(&map_x);
    }
    if (tid == 0) {
        for (int s = 0; s < kSpanStages; ++s) {
            mbar_init(smem_addr(&sh.full[s]), 1u);
            mbar_init(smem_addr(&sh.empty[s]), 1u);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_addr(&sh.acc_full[b]), 1u);
            mbar_init(smem_addr(&sh.acc_empty[b]), 8u);
        }
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_addr(&sh.tmem), kSpanCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t base = (smem_addr(tc_raw) + 1023u) & ~1023u;
    const uint32_t tmem = sh.tmem;
    volatile int* abort_flag = &sh.abort_flag;
    struct Item {
        int m, tt, c0, c1;       // row tile, token tile, K chunks
    };
    auto item = [&](int i) -> Item {
        const int tile = i / p.split, k = i - tile * p.split, m = tile / p.tiles_t;
        return Item{m, tile - m * p.tiles_t, k * p.call / p.split, (k + 1) * p.call / p.split};
    };
    dep_trigger();           // the kernel behind does not touch what it shares with this one before its wait

    if (warp == 0) {
        if (lane == 0) {
            int it = 0, s = 0;
            uint32_t parity = 1u;
            auto load_w = [&](int st, int m, int c) {
                const uint32_t bar = smem_addr(&sh.full[st]), dst = base + st * kSpanStageBytes;
                mbar_expect_tx(bar, kSpanStageBytes);
                if (MN) {
                    tma_load_2d(dst, &map_w, bar, m * 128, c * kChunk);
                    tma_load_2d(dst + kChunk * 128, &map_w, bar, m * 128 + 64, c * kChunk);
                } else {
                    tma_load_2d(dst, &map_w, bar, c * kChunk, m * 128);
                }
            };
            auto load_x = [&](int st, int t, int c) {
                const uint32_t bar = smem_addr(&sh.full[st]), dst = base + st * kSpanStageBytes + kStreamTileBytes;
                tma_load_2d(dst, &map_x, bar, c * kChunk, t * kSpanTile);
                tma_load_2d(dst + kSpanTile * 128, &map_x, bar, c * kChunk, p.lo_row + t * kSpanTile);
            };
            // the first stages of weights do not depend on the kernel ahead
            int pre = 0;
            const Item first = item(blockIdx.x);
            if (static_cast<int>(blockIdx.x) < p.tiles)
                for (; pre < min(first.c1 - first.c0, kSpanStages); ++pre) load_w(pre, first.m, first.c0 + pre);
            dep_wait();
            for (int i = 0; i < pre; ++i) load_x(i, first.tt, first.c0 + i);
            bool ok = true;
            for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x) {
                const Item w = item(tile);
                for (int c = w.c0; c < w.c1; ++c, ++it) {
                    if (it >= pre) {
                        if (it >= kSpanStages && !mbar_wait(smem_addr(&sh.empty[s]), parity, abort_flag)) { ok = false; break; }
                        load_w(s, w.m, c);
                        load_x(s, w.tt, c);
                    }
                    if (++s == kSpanStages) { s = 0; parity ^= 1u; }
                }
            }
            if (*abort_flag != 0) {          // the copies in flight land (bounded) before the block goes
                for (int i = max(0, it - kSpanStages); i < it; ++i) {
                    const long long c0 = clock64();
                    while (!mbar_try(smem_addr(&sh.full[i % kSpanStages]), static_cast<uint32_t>(i / kSpanStages) & 1u))
                        if (clock64() - c0 > kTcSpinLimit) break;
                }
            }
        }
    } else if (warp == 1) {
        const uint32_t elected = elect_lane(), idesc = instr_desc(128, 2 * kSpanTile, MN);
        int s = 0, seg = 0;
        uint32_t parity = 0u;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x) {
            const Item w = item(tile);
            for (int g = 0; g < p.nseg && ok; ++g, ++seg) {
                const int c0 = w.c0 + g * (w.c1 - w.c0) / p.nseg, c1 = w.c0 + (g + 1) * (w.c1 - w.c0) / p.nseg, b = seg & 1;
                if (seg >= 2) ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_empty[b]), ((seg >> 1) & 1) ^ 1, abort_flag));
                const uint32_t acc = tmem + static_cast<uint32_t>(b) * 256u;
                tc_fence_after();
                for (int c = c0; c < c1 && ok; ++c) {
                    ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), parity, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a0 = base + s * kSpanStageBytes;
                    const uint64_t ad = MN ? smem_desc(a0, kChunk * 128, 1024u) : smem_desc(a0, 0u, 1024u);
                    const uint64_t xd = smem_desc(a0 + kStreamTileBytes, 0u, 1024u);
#pragma unroll
                    for (int j = 0; j < kChunk / 16; ++j)      // descriptors count in 16-byte units
                        umma_bf16_elected(acc, ad + j * (MN ? 128 : 2), xd + 2 * j, idesc, (c > c0 || j > 0) ? 1u : 0u, elected);
                    umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                    if (++s == kSpanStages) { s = 0; parity ^= 1u; }
                }
                if (ok) umma_commit_elected(smem_addr(&sh.acc_full[b]), elected);
            }
        }
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2;
        dep_wait();
        int seg = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x) {
            const Item w = item(tile);
            const int row = w.m * 128 + q * 32 + lane, t0 = w.tt * kSpanTile + half * 64;
            const int64_t at = static_cast<int64_t>(t0) * p.rows + row;
            if constexpr (U) {
                // one segment; sixteen tokens at a time: scores in (one group ahead), activation, two bf16 terms out
                float next[16];
                auto request = [&](int j) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        next[i] = row < p.rows && t0 + 16 * j + i < p.T ? __ldcg(p.S + at + static_cast<int64_t>(16 * j + i) * p.rows) : -INFINITY;
                };
                request(0);
                const int b = seg & 1;
                ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_full[b]), (seg >> 1) & 1, abort_flag));
                if (!ok) break;
                ++seg;
                tc_fence_after();
                const uint32_t taddr = tmem + static_cast<uint32_t>(b * 256 + half * 64) + (static_cast<uint32_t>(q * 32) << 16);
                const bool odd = lane & 1;
                // even lanes store this pair of rows for the even tokens, odd lanes for the odd ones
                __nv_bfloat16* uh = p.u + at + (odd ? static_cast<int64_t>(p.rows) - 1 : 0);
                const int64_t lo = static_cast<int64_t>(p.lo_row) * p.rows;
#pragma unroll 1
                for (int j = 0; j < 4; ++j) {
                    float sv[16], v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) sv[i] = next[i];
                    if (j < 3) request(j + 1);
                    tmem_ld16_sum(taddr + 16 * j, taddr + kSpanTile + 16 * j, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float th = __ldg(p.theta + min(t0 + 16 * j + i, p.T - 1));
                        const float a = p.identity ? sv[i] : sv[i] - th;
                        v[i] = sv[i] > th ? (p.erf_form ? gelu_erf(a) : gelu_logistic(a)) * v[i] : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float mine = odd ? v[i + 1] : v[i], other = __shfl_xor_sync(kFull, odd ? v[i] : v[i + 1], 1);
                        unsigned hi, l;
                        split_pair(odd ? other : mine, odd ? mine : other, hi, l);
                        if (row < p.rows && t0 + 16 * j + i + (odd ? 1 : 0) < p.T) {
                            __nv_bfloat16* dst = uh + static_cast<int64_t>(16 * j + i) * p.rows;
                            *reinterpret_cast<unsigned*>(dst) = hi;
                            *reinterpret_cast<unsigned*>(dst + lo) = l;
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.acc_empty[b])) : "memory");
            } else {
                float acc[64];
                for (int g = 0; g < p.nseg; ++g, ++seg) {
                    const int b = seg & 1;
                    ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_full[b]), (seg >> 1) & 1, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t taddr = tmem + static_cast<uint32_t>(b * 256 + half * 64) + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float v[16];
                        tmem_ld16_sum(taddr + 16 * j, taddr + kSpanTile + 16 * j, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[16 * j + i] = g == 0 ? v[i] : acc[16 * j + i] + v[i];
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.acc_empty[b])) : "memory");
                }
                if (!ok) break;
                if (row >= p.rows) continue;
                if (p.split > 1) {           // y holds the addend already
#pragma unroll
                    for (int i = 0; i < 64; ++i)
                        if (t0 + i < p.T) atomicAdd(p.y + at + static_cast<int64_t>(i) * p.rows, acc[i]);
                    continue;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float av[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        av[i] = p.add != nullptr && t0 + 16 * j + i < p.T ? __ldcg(p.add + at + static_cast<int64_t>(16 * j + i) * p.rows) : 0.f;
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (t0 + 16 * j + i < p.T) p.y[at + static_cast<int64_t>(16 * j + i) * p.rows] = acc[16 * j + i] + av[i];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, kSpanCols);
    }
    if (tid == 0 && sh.abort_flag != 0) atomicCAS(&p.hdr->status, SPARK_OK, SPARK_ERR_TIMEOUT);
}

// ---- prep: one block per token: optional division per head, optional RMSNorm, two bf16 terms -------------------------------
struct SpanPrep {
    const float* x;          // [T][n]
    const float* norm_w;     // nullable
    float eps;
    const float* div;        // nullable [T][n / group]
    int n, group, lo_row;
    __nv_bfloat16* xs;       // [2 * Tp][n]
    float* copy;             // nullable: x goes here as well (what a product in pieces adds into)
};
__global__ void __launch_bounds__(256) span_prep_kernel(const SpanPrep p) {
    __shared__ float red[8];
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n4 = p.n / 4;
    dep_wait();
    dep_trigger();
    const float4* xr = reinterpret_cast<const float4*>(p.x + static_cast<int64_t>(t) * p.n);
    auto load = [&](int i) -> float4 {
        float4 v = xr[i];
        if (p.div != nullptr) {
            const float d = p.div[static_cast<int64_t>(t) * (p.n / p.group) + 4 * i / p.group], inv = d > 0.f ? 1.f / d : 0.f;
            v = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
        }
        return v;
    };
    constexpr int kKeep = 4;             // rows of up to 4096 values stay in registers between the two passes
    float4 keep[kKeep];
#pragma unroll
    for (int u = 0; u < kKeep; ++u) keep[u] = tid + 256 * u < n4 ? load(tid + 256 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.copy != nullptr) {
        float4* dst = reinterpret_cast<float4*>(p.copy + static_cast<int64_t>(t) * p.n);
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
            if (tid + 256 * u < n4) dst[tid + 256 * u] = keep[u];
        for (int i = tid + 256 * kKeep; i < n4; i += 256) dst[i] = xr[i];
    }
    float sc = 1.f;
    if (p.norm_w != nullptr) {
        float ss = 0.f;
#pragma unroll
        for (int u = 0; u < kKeep; ++u) ss += keep[u].x * keep[u].x + keep[u].y * keep[u].y + keep[u].z * keep[u].z + keep[u].w * keep[u].w;
        for (int i = tid + 256 * kKeep; i < n4; i += 256) {
            const float4 v = load(i);
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        ss = warp_sum(ss);
        if (lane == 0) red[warp] = ss;
        __syncthreads();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += red[w];
        sc = rsqrtf(tot / static_cast<float>(p.n) + p.eps);
    }
    uint2* hi = reinterpret_cast<uint2*>(p.xs + static_cast<int64_t>(t) * p.n);
    uint2* lo = reinterpret_cast<uint2*>(p.xs + static_cast<int64_t>(p.lo_row + t) * p.n);
    auto store = [&](int i, float4 v) {
        if (p.norm_w != nullptr) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(p.norm_w) + i);
            v = make_float4(v.x * sc * w.x, v.y * sc * w.y, v.z * sc * w.z, v.w * sc * w.w);
        }
        uint2 h, l;
        split_pair(v.x, v.y, h.x, l.x);
        split_pair(v.z, v.w, h.y, l.y);
        hi[i] = h;
        lo[i] = l;
    };
#pragma unroll
    for (int u = 0; u < kKeep; ++u)
        if (tid + 256 * u < n4) store(tid + 256 * u, keep[u]);
    for (int i = tid + 256 * kKeep; i < n4; i += 256) store(i, load(i));
}

// ---- theta: one block per token (Eq. 11 over the token's scores) -------------------------------------------------------------
struct SpanTheta {
    const float* S;          // [T][n]
    int n, identity;
    double z, inv_n, inv_nm1;
    float* theta;
};
__global__ void __launch_bounds__(256) span_theta_kernel(const SpanTheta p) {
    __shared__ double red[8][2];
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    dep_wait();
    dep_trigger();
    double s1 = 0.0, s2 = 0.0;
    if (!p.identity) {
        const float4* sr = reinterpret_cast<const float4*>(p.S + static_cast<int64_t>(t) * p.n);      // n is a multiple of 8
        for (int i0 = tid; i0 < p.n / 4; i0 += 256 * 4) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i0 + 256 * u < p.n / 4 ? __ldcg(sr + i0 + 256 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double a = v[u].x, b = v[u].y, c = v[u].z, d = v[u].w;
                s1 += (a + b) + (c + d);
                s2 += fma(a, a, b * b) + fma(c, c, d * d);
            }
        }
        s1 = warp_sum_f64(s1);
        s2 = warp_sum_f64(s2);
        if (lane == 0) {
            red[warp][0] = s1;
            red[warp][1] = s2;
        }
    }
    __syncthreads();
    if (tid == 0) {
        float th = -INFINITY;
        if (!p.identity) {
            s1 = s2 = 0.0;
            for (int w = 0; w < 8; ++w) {
                s1 += red[w][0];
                s2 += red[w][1];
            }
            const double mean = s1 * p.inv_n;
            const float var = static_cast<float>((s2 - s1 * mean) * p.inv_nm1);
            th = static_cast<float>(mean) + sqrtf(fmaxf(var, 0.f)) * static_cast<float>(p.z);
        }
        p.theta[t] = th;
    }
}

// ---- rope: one block per token: rotary encoding per half, queries into the attention's operand form, cache append ----------
struct SpanRope {
    const float* qkv;        // [T][(n_q + 2 n_kv) hd]
    __nv_bfloat16* k1c;
    __nv_bfloat16* k2c;
    __nv_bfloat16* vc;
    int n_q, n_kv, gq, hd, r, tps, colcap, start, window, k_attn;
    int64_t cap;
    float q_scale;
    double* zt;
    double* sums;            // cleared for the attention, like smax, o and lsum
    unsigned* smax;
    float* o;                // [T][n_q][hd]
    float* lsum;             // [T][n_q]
    __nv_bfloat16* qhi;
    __nv_bfloat16* qlo;
    __nv_bfloat16* q2hi;
    __nv_bfloat16* q2lo;
    double inv_freq[2][64];
};
__global__ void __launch_bounds__(256) span_rope_kernel(const __grid_constant__ SpanRope p) {
    // two groups of 128 threads take every other head
    const int t = blockIdx.x, pr = threadIdx.x & 127, grp = threadIdx.x >> 7, pos = p.start + t, hr = p.r / 2;
    const int sub = t / p.tps, col0 = (t - sub * p.tps) * p.gq;
    dep_wait();
    dep_trigger();
    for (int i = threadIdx.x; i < p.n_q * p.hd / 4; i += 256) reinterpret_cast<float4*>(p.o + static_cast<int64_t>(t) * p.n_q * p.hd)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int h = threadIdx.x; h < p.n_q; h += 256) {
        const int64_t vcol = static_cast<int64_t>(sub * p.n_kv + h / p.gq) * p.colcap + col0 + h % p.gq;
        p.sums[2 * vcol] = p.sums[2 * vcol + 1] = 0.0;
        p.smax[vcol] = 0u;
        p.lsum[static_cast<int64_t>(t) * p.n_q + h] = 0.f;
    }
    if (threadIdx.x == 255) {         // the threshold quantile over the rows the token sees
        const int n = pos + 1, L = (p.window > 0 && p.window < n) ? p.window : n;
        p.zt[t] = p.k_attn >= L ? 0.0 : -normcdfinv(static_cast<double>(p.k_attn) / static_cast<double>(L));
    }
    if (pr >= p.hd / 2) return;
    // pairs (i, i + m/2) inside each part of m dims: the first r/2 threads have part [0, r), the others [r, hd)
    const bool second = pr >= hr;
    const int m = second ? p.hd - p.r : p.r, pi = second ? pr - hr : pr, ia = (second ? p.r : 0) + pi, ib = ia + m / 2;
    // angle = pos * base^(-2i/m): the product and its reduction to one turn in fp64 (positions reach tens of thousands of
    // radians), sine and cosine of the reduced angle in fp32; once per token, for all heads
    const double turns = static_cast<double>(pos) * p.inv_freq[second ? 1 : 0][pi] * 0.15915494309189533577;
    float sn, cs;
    sincosf(static_cast<float>((turns - floor(turns)) * 6.28318530717958647692), &sn, &cs);
    const float* row = p.qkv + static_cast<int64_t>(t) * (p.n_q + 2 * p.n_kv) * p.hd;
    __nv_bfloat16* oh = second ? p.q2hi : p.qhi;
    __nv_bfloat16* ol = second ? p.q2lo : p.qlo;
    // four heads at a time, their loads in flight together
    for (int h0 = grp; h0 < p.n_q; h0 += 8) {
        float a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int h = min(h0 + 2 * u, p.n_q - 1);
            a[u] = __ldg(row + h * p.hd + ia);
            b[u] = __ldg(row + h * p.hd + ib);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int h = h0 + 2 * u, g = h / p.gq;
            if (h >= p.n_q) break;
            const float ra = (a[u] * cs - b[u] * sn) * p.q_scale, rb = (a[u] * sn + b[u] * cs) * p.q_scale;
            const int64_t at = (static_cast<int64_t>(sub * p.n_kv + g) * p.colcap + col0 + h - g * p.gq) * m + pi;
            const __nv_bfloat16 ha = __float2bfloat16_rn(ra), hb = __float2bfloat16_rn(rb);
            oh[at] = ha;
            oh[at + m / 2] = hb;
            ol[at] = __float2bfloat16_rn(ra - __bfloat162float(ha));
            ol[at + m / 2] = __float2bfloat16_rn(rb - __bfloat162float(hb));
        }
    }
    __nv_bfloat16* kc = second ? p.k2c : p.k1c;
    for (int g0 = grp; g0 < p.n_kv; g0 += 8) {
        float a[4], b[4];
        float2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int g = min(g0 + 2 * u, p.n_kv - 1);
            a[u] = __ldg(row + (p.n_q + g) * p.hd + ia);
            b[u] = __ldg(row + (p.n_q + g) * p.hd + ib);
            v[u] = __ldg(reinterpret_cast<const float2*>(row + (p.n_q + p.n_kv + g) * p.hd + 2 * pr));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int g = g0 + 2 * u;
            if (g >= p.n_kv) break;
            __nv_bfloat16* dst = kc + (g * p.cap + pos) * m + pi;
            dst[0] = __float2bfloat16_rn(a[u] * cs - b[u] * sn);
            dst[m / 2] = __float2bfloat16_rn(a[u] * sn + b[u] * cs);
            *reinterpret_cast<__nv_bfloat162*>(p.vc + (g * p.cap + pos) * p.hd + 2 * pr) = __floats2bfloat162_rn(v[u].x, v[u].y);
        }
    }
}

// ---- host ---------------------------------------------------------------------------------------------------------------------
// The span's part of the workspace, behind the attention's cells.  The attention's arrays and the FFN's share their place.
struct SpanLayout {
    int64_t Tp;
    size_t xs, qkv, ao, lsum, h2, theta, shared, S, u, bytes;
};
SpanLayout span_layout(int64_t T, int64_t d, int64_t d_ff, int64_t n_q, int64_t n_kv, int64_t hd) {
    SpanLayout l;
    l.Tp = (T + kSpanTile - 1) / kSpanTile * kSpanTile;
    const size_t Tp = static_cast<size_t>(l.Tp), nqo = static_cast<size_t>(n_q * hd), nqkv = static_cast<size_t>((n_q + 2 * n_kv) * hd);
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t here = at;
        at += round_up(bytes, 1024);
        return here;
    };
    l.xs = take(2 * Tp * (static_cast<size_t>(d) > nqo ? static_cast<size_t>(d) : nqo) * 2);
    l.qkv = take(Tp * nqkv * 4);
    l.ao = take(Tp * nqo * 4);
    l.lsum = take(Tp * static_cast<size_t>(n_q) * 4);
    l.h2 = take(Tp * static_cast<size_t>(d) * 4);
    l.theta = take(Tp * 4);
    l.shared = at;
    const size_t attn = attn_span_bytes(l.Tp, n_q, n_kv, hd);
    l.S = take(Tp * static_cast<size_t>(d_ff) * 4);
    l.u = take(2 * Tp * static_cast<size_t>(d_ff) * 2);
    l.bytes = at > l.shared + attn ? at : l.shared + attn;
    return l;
}

// Pieces of the K range of a product that is added into an addend: while the tiles are fewer than the SMs (a short span's output
// projection and V product: 18 row tiles at the 2B shape; 130 tokens, V 75 -> 20 us, the call 0.65 -> 0.48 ms), not below eight K chunks a piece.
int span_split(const spark_ctx* ctx, int64_t rows, int64_t T, int64_t K) {
    const int64_t tiles = (rows + 127) / 128 * ((T + kSpanTile - 1) / kSpanTile), call = (K + kChunk - 1) / kChunk;
    int64_t s = ctx->num_sms / tiles;
    if (s > call / 8) s = call / 8;
    return s < 1 ? 1 : static_cast<int>(s);
}

// X operand and weights of one product.
template <bool MN, bool U>
int span_gemm(spark_ctx* ctx, SpanGemm p, const void* W, int64_t K, const __nv_bfloat16* X, int64_t ldx, int64_t Tp, cudaStream_t stream) {
    p.call = static_cast<int>((K + kChunk - 1) / kChunk);
    p.tiles_t = static_cast<int>((p.T + kSpanTile - 1) / kSpanTile);
    if (p.split < 1) p.split = 1;
    p.nseg = U ? 1 : ((p.call + p.split - 1) / p.split + kSpanSeg - 1) / kSpanSeg;
    p.tiles = (p.rows + 127) / 128 * p.tiles_t * p.split;
    p.lo_row = static_cast<int>(Tp);
    p.hdr = ctx->hdr;
    CUtensorMap m_w, m_x;
    if (!(MN ? make_map(&m_w, W, K, p.rows, p.rows, kChunk, true) : make_map(&m_w, W, p.rows, K, K, 128, true)) ||
        !make_map(&m_x, X, 2 * Tp, K, ldx, kSpanTile, false))
        return SPARK_ERR_WORKSPACE;
    const size_t smem = static_cast<size_t>(kSpanStages) * kSpanStageBytes + 1024;
    const void* kern = reinterpret_cast<const void*>(span_gemm_kernel<MN, U>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) return SPARK_ERR_CUDA;
    void* args[] = {&p, &m_w, &m_x};
    const int grid = p.tiles < ctx->num_sms ? p.tiles : ctx->num_sms;
    return launch_kernel(ctx, kern, static_cast<unsigned>(grid), kSpanThreads, smem, stream, false, args, true) == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace

namespace spark {

size_t span_workspace_bytes(int64_t max_dff, int64_t n_q, int64_t hd, int64_t max_d) {
    if (max_dff < 8 || max_d < 16) return 0;
    return kAttnCellBytes + span_layout(kSpanMax, max_d, max_dff, n_q, n_q, hd).bytes;
}

int64_t span_tokens(const spark_ctx* ctx, const spark_layer_weights* w, const spark_layer_cfg* cfg, const spark_kv_cache* cache, int64_t n_layers,
                    const float* h, int64_t n_tokens) {
    if (n_tokens <= 64 || ctx->chunk_dense == 0 || ctx->scratch == nullptr || (reinterpret_cast<uintptr_t>(h) & 15u) != 0) return 0;
    int64_t T = n_tokens < kSpanMax ? n_tokens : kSpanMax;
    for (int64_t l = 0; l < n_layers; ++l) {
        const spark_layer_cfg& c = cfg[l];
        if ((c.flags & ~(SPARK_GELU_ERF | SPARK_SHARED_CACHE)) != 0) return 0;
        if (c.n_q < 1 || c.n_kv < 1 || c.n_q % c.n_kv != 0 || c.hd < 16 || c.hd > 256 || c.r_attn < 8 || c.r_attn > 128 || c.hd - c.r_attn < 8 || c.hd - c.r_attn > 128 ||
            (c.r_attn & 7) != 0 || ((c.hd - c.r_attn) & 7) != 0 || c.k_attn < 1 || c.window < 0)
            return 0;
        const int64_t gq = c.n_q / c.n_kv;
        if (gq != 1 && gq != 2 && gq != 4 && gq != 8) return 0;
        if ((c.n_kv & (c.n_kv - 1)) != 0 || c.n_kv * c.cap >= (1LL << 31) || c.n_q > 1024) return 0;
        if (c.d < 16 || (c.d & 7) != 0 || c.d > (1 << 20) || c.r_ff < 8 || c.r_ff >= c.d || (c.r_ff & 7) != 0 || c.d_ff < 8 || (c.d_ff & 7) != 0 || c.d_ff > (1 << 24) || c.k_ff < 1)
            return 0;
        const void* need[] = {w[l].norm1, w[l].norm2, w[l].Wqkv, w[l].Wo, w[l].K1t, w[l].K2t, w[l].Vt, cache[l].k1c, cache[l].k2c, cache[l].vc};
        for (const void* ptr : need)
            if (ptr == nullptr || (reinterpret_cast<uintptr_t>(ptr) & 15u) != 0) return 0;
        while (T > 64 && kAttnCellBytes + span_layout(T, c.d, c.d_ff, c.n_q, c.n_kv, c.hd).bytes > ctx->scratch_bytes)
            T = (T - 1) / kSpanTile * kSpanTile;
    }
    if (T <= 64) return 0;
    const int64_t spans = (n_tokens + T - 1) / T, even = (n_tokens + spans - 1) / spans;
    const int64_t padded = (even + kSpanTile - 1) / kSpanTile * kSpanTile;
    return padded < T ? padded : T;
}

int span_layer_launch(spark_ctx* ctx, const spark_layer_weights* w, const spark_layer_cfg* cfg, const spark_kv_cache* cache, float* h, int64_t T,
                      int64_t start, cudaStream_t stream) {
    const int64_t d = cfg->d, d_ff = cfg->d_ff, n_q = cfg->n_q, n_kv = cfg->n_kv, hd = cfg->hd, nqo = n_q * hd, nqkv = (n_q + 2 * n_kv) * hd;
    const SpanLayout l = span_layout(T, d, d_ff, n_q, n_kv, hd);
    char* base = ctx->scratch + kAttnCellBytes;
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(base + l.xs);
    float* qkv = reinterpret_cast<float*>(base + l.qkv);
    float* ao = reinterpret_cast<float*>(base + l.ao);
    float* lsum = reinterpret_cast<float*>(base + l.lsum);
    float* h2 = reinterpret_cast<float*>(base + l.h2);
    float* theta = reinterpret_cast<float*>(base + l.theta);
    float* S = reinterpret_cast<float*>(base + l.S);
    __nv_bfloat16* u = reinterpret_cast<__nv_bfloat16*>(base + l.u);

    const int split_o = span_split(ctx, d, T, nqo), split_v = span_split(ctx, d, T, d_ff);
    auto prep = [&](const float* x, const float* norm_w, const float* div, int64_t n, int64_t group, float* copy) -> int {
        SpanPrep p{x, norm_w, cfg->rms_eps, div, static_cast<int>(n), static_cast<int>(group), static_cast<int>(l.Tp), xs, copy};
        void* args[] = {&p};
        return launch_kernel(ctx, reinterpret_cast<const void*>(span_prep_kernel), static_cast<unsigned>(T), 256, 0, stream, false, args, true) == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
    };
    SpanGemm g = {};
    g.T = static_cast<int>(T);
    auto product = [&](int64_t rows, const void* W, int64_t K, const float* add, float* y) -> int {
        g.rows = static_cast<int>(rows); g.add = add; g.y = y;
        return span_gemm<false, false>(ctx, g, W, K, xs, K, l.Tp, stream);
    };
    int rc = prep(h, w->norm1, nullptr, d, 1, split_o > 1 ? h2 : nullptr);
    if (rc == SPARK_OK) rc = product(nqkv, w->Wqkv, d, nullptr, qkv);
    if (rc != SPARK_OK) return rc;

    AttnSpan a;
    a.k1c = cache->k1c; a.k2c = cache->k2c; a.vc = cache->vc;
    a.T = T; a.n_q = n_q; a.n_kv = n_kv; a.hd = hd; a.r = cfg->r_attn; a.cap = cfg->cap; a.start = start;
    a.window = cfg->window; a.k_attn = cfg->k_attn;
    a.o = ao; a.lsum = lsum;
    if (!attn_span_layout(a, base + l.shared)) return SPARK_ERR_UNSUPPORTED;
    {
        SpanRope p;
        p.qkv = qkv;
        p.k1c = static_cast<__nv_bfloat16*>(cache->k1c); p.k2c = static_cast<__nv_bfloat16*>(cache->k2c); p.vc = static_cast<__nv_bfloat16*>(cache->vc);
        p.n_q = static_cast<int>(n_q); p.n_kv = static_cast<int>(n_kv); p.gq = static_cast<int>(n_q / n_kv); p.hd = static_cast<int>(hd); p.r = static_cast<int>(cfg->r_attn);
        p.tps = a.tps; p.colcap = a.colcap; p.start = static_cast<int>(start);
        p.window = static_cast<int>(cfg->window > 0x7fffffff ? 0x7fffffff : cfg->window);
        p.k_attn = static_cast<int>(cfg->k_attn > 0x7fffffff ? 0x7fffffff : cfg->k_attn);
        p.cap = cfg->cap;
        p.q_scale = 1.0f / std::sqrt(static_cast<float>(hd));
        p.zt = a.zt; p.sums = a.sums; p.smax = a.smax; p.o = ao; p.lsum = lsum; p.qhi = a.qhi; p.qlo = a.qlo; p.q2hi = a.q2hi; p.q2lo = a.q2lo;
        for (int part = 0; part < 2; ++part) {
            const int64_t m = part == 0 ? cfg->r_attn : hd - cfg->r_attn;
            for (int64_t i = 0; i < m / 2; ++i)
                p.inv_freq[part][i] = std::pow(static_cast<double>(cfg->rope_base), -2.0 * static_cast<double>(i) / static_cast<double>(m));
        }
        void* args[] = {&p};
        if (launch_kernel(ctx, reinterpret_cast<const void*>(span_rope_kernel), static_cast<unsigned>(T), 256, 0, stream, false, args, true) != cudaSuccess) return SPARK_ERR_CUDA;
    }
    rc = attn_span_launch(ctx, a, stream);
    if (rc == SPARK_OK) rc = prep(ao, nullptr, lsum, nqo, hd, nullptr);
    g.split = split_o;
    if (rc == SPARK_OK) rc = product(d, w->Wo, nqo, h, h2);
    g.split = 1;
    if (rc == SPARK_OK) rc = prep(h2, w->norm2, nullptr, d, 1, split_v > 1 ? h : nullptr);
    if (rc != SPARK_OK) return rc;

    g.rows = static_cast<int>(d_ff); g.add = nullptr; g.y = S;
    rc = span_gemm<false, false>(ctx, g, w->K1t, cfg->r_ff, xs, d, l.Tp, stream);
    if (rc != SPARK_OK) return rc;
    const int identity = cfg->k_ff >= d_ff ? 1 : 0;
    {
        SpanTheta p;
        p.S = S; p.n = static_cast<int>(d_ff); p.identity = identity;
        p.z = identity ? 0.0 : spark_normal_upper_quantile(static_cast<double>(cfg->k_ff) / static_cast<double>(d_ff));
        p.inv_n = 1.0 / static_cast<double>(d_ff);
        p.inv_nm1 = 1.0 / static_cast<double>(d_ff - 1);
        p.theta = theta;
        void* args[] = {&p};
        if (launch_kernel(ctx, reinterpret_cast<const void*>(span_theta_kernel), static_cast<unsigned>(T), 256, 0, stream, false, args, true) != cudaSuccess) return SPARK_ERR_CUDA;
    }
    g.S = S; g.theta = theta; g.identity = identity; g.erf_form = (cfg->flags & SPARK_GELU_ERF) ? 1 : 0; g.u = u;
    rc = span_gemm<false, true>(ctx, g, w->K2t, d - cfg->r_ff, xs + cfg->r_ff, d, l.Tp, stream);
    if (rc != SPARK_OK) return rc;
    g.rows = static_cast<int>(d); g.add = h2; g.y = h; g.split = split_v;
    return span_gemm<true, false>(ctx, g, w->Vt, d_ff, u, d_ff, l.Tp, stream);
}

}  // namespace spark
