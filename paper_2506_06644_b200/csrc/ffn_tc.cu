// Spark FFN (Section 2.1, Eq. 2) for a chunk of 5..64 tokens with bf16 weights, on the fifth-generation
// tensor cores.  With this many tokens the union of the tokens' active sets (Appendix B) covers most
// neurons, every weight row is read anyway, and the three products are real GEMMs with the tokens as
// the N dimension.  One kernel, one block per SM; its blocks meet at three grid-wide barriers:
//   x     RMSNorm scale (optional), x -> two bf16 terms (x = hi + lo), a part of a token's row per block          | barrier
//   S     scores K1t . X[:, :r]^T of the block's neurons, per-token score sums for Eq. 11                         | barrier
//   T, U  products K2t . X[:, r:]^T (they run while the sums travel), theta per token (Eq. 10/11),
//         U = [S > theta] . GELU(S - theta) . T as two bf16 terms                                                  | barrier
//   Y     Y^T += Vt^T . U: M = 128 model columns (Vt enters MN-major, as it is stored), N = tokens,
//         K = neurons split over blocks, fp32 reductions into y
// The fp32 activations enter every product as an error-compensated two-term bf16 split: the scores decide index sets, so a bare
// bf16 rounding (2^-9) is not enough, and the two terms carry 16 mantissa bits.  Both terms are one operand tile of N = 2 x tokens.
// What bounds it is the weight stream.  One warp requests the weights of all three products through one ring of stages, so the
// stream runs on under the barriers, and the first weights of the output product past the ring are asked into L2 while the block waits
// for U.  Scores and products stay in tensor memory.
#include "ffn_params.h"
#include "kernels.h"
#include "stream_gemm.cuh"

using namespace spark;
using namespace spark::tc;

namespace {

constexpr int kTok = 64;              // token rows of the padded operands
constexpr int kFfnThreads = 320;      // warp 0: TMA, warp 1: MMA + tensor memory, warps 2..9: everything else
constexpr int kEpi = 256;
constexpr int kMaxStages = 10;
constexpr int kMaxTiles = 2;          // tiles of neurons per block: 2 x 2 accumulators of 128 columns fill tensor memory
constexpr int kMinRows = 32;          // neurons of a tile at least: every tile reads all of X
constexpr int kAhead = 4;             // chunks of the output product's weights asked into L2 while the block waits for U

// ---- layout of the chunk path's part of the workspace ----------------------------------------------
struct TcRegion {
    __nv_bfloat16* xs;            // [2 ntok][d]: hi rows, lo rows
    __nv_bfloat16* us;            // [2 ntok][d_ff]
};
inline size_t tc_region_bytes(int64_t d, int64_t d_ff) {
    return round_up(static_cast<size_t>(2 * kTok) * d * 2, 1024) + round_up(static_cast<size_t>(2 * kTok) * d_ff * 2, 1024);
}
inline TcRegion tc_region(char* base, int64_t d) {
    return TcRegion{reinterpret_cast<__nv_bfloat16*>(base), reinterpret_cast<__nv_bfloat16*>(base + round_up(static_cast<size_t>(2 * kTok) * d * 2, 1024))};
}

struct TcParams {
    FfnParams f;
    TcRegion g;
    int ntok;            // B rounded up to a multiple of 16: half of the MMAs' N
    int rows, tiles;     // neurons per tile, tiles (block b takes tiles b and b + blocks)
    int parts;           // blocks per token row in the conversion of x
    int ksplit, otiles;  // output: blocks per tile of 128 model columns, tiles
    int stages, stage_bytes;
    uint32_t tmem_cols;
};

struct FfnShared {
    unsigned long long full[kMaxStages], empty[kMaxStages];
    unsigned long long acc_s[kMaxTiles], acc_t[kMaxTiles], acc_o;     // accumulators final
    unsigned long long x_ready, u_ready;                              // the grid's X, U may be loaded
    uint32_t tmem;
    int abort_flag;
    float red[8];
    float theta[kTok];
    double sums[4][2][kTok];                                          // per quarter of a tile and token: score sum, sum of squares
    float win[8][32 * 17];                                            // per warp: 32 neurons x 16 tokens
};

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// Data that other blocks wrote with ordinary stores, behind an acquire, before this thread's TMA loads read it.
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(map), "r"(x), "r"(y) : "memory");
}
// Issued by one elected lane of a warp that walks its loop as a whole.
__device__ __forceinline__ void mbar_expect_tx_elected(uint32_t bar, uint32_t bytes, uint32_t elected) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar), "r"(bytes), "r"(elected) : "memory");
}
__device__ __forceinline__ void tma_load_2d_elected(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, uint32_t elected) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
                 " @q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n}"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(elected) : "memory");
}

// Grid-wide barrier: arrival counters that only grow (the fused layer kernel counts on with the same ones).  One warp arrives and polls.
__device__ __forceinline__ void grid_arrive(WsHeader* hdr) { red_release_add_u32(&hdr->l1_ways[blockIdx.x % kCellWays].count, 1u); }
__device__ __forceinline__ bool grid_wait(WsHeader* hdr, unsigned gen, volatile int* abort_flag) {
    const int lane = threadIdx.x & 31;
    const unsigned target = gen * gridDim.x;
    const long long t0 = clock64(), limit = spin_limit(hdr);
    for (;;) {
        unsigned v = lane < kCellWays ? ld_acquire_u32(&hdr->l1_ways[lane].count) : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (static_cast<int>(v - target) >= 0) return true;
        if (__any_sync(kFull, *abort_flag != 0 || clock64() - t0 > limit)) {
            if (lane == 0) *abort_flag = 1;
            return false;
        }
    }
}

__global__ void __launch_bounds__(kFfnThreads, 1)
ffn_tc_kernel(const TcParams p, const __grid_constant__ CUtensorMap map_k1, const __grid_constant__ CUtensorMap map_x1,
              const __grid_constant__ CUtensorMap map_k2, const __grid_constant__ CUtensorMap map_x2, const __grid_constant__ CUtensorMap map_v,
              const __grid_constant__ CUtensorMap map_u) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ FfnShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x, B = p.f.B, d = p.f.d, stages = p.stages;
    const int64_t dff = p.f.d_ff;
    const int c1n = (p.f.r + kChunk - 1) / kChunk, c2n = (d - p.f.r + kChunk - 1) / kChunk;
    const int nt = cta < p.tiles ? (p.tiles - 1 - cta) / gridDim.x + 1 : 0;          // the block's tiles of neurons
    const int otile = cta / p.ksplit, piece = cta - otile * p.ksplit, cvn = (p.f.d_ff + kChunk - 1) / kChunk;
    const bool outs = otile < p.otiles;
    const int cv0 = outs ? static_cast<int>(static_cast<int64_t>(piece) * cvn / p.ksplit) : 0, cv1 = outs ? static_cast<int>(static_cast<int64_t>(piece + 1) * cvn / p.ksplit) : 0;
    const int n1 = nt * c1n, n12 = n1 + nt * c2n;                 // chunks of the scores, and of the products behind them
    if (tid < 32) {
        if (tid < stages) {
            mbar_init(smem_addr(&sh.full[tid]), 1u);
            mbar_init(smem_addr(&sh.empty[tid]), 1u);
        } else if (tid < stages + kMaxTiles) {
            mbar_init(smem_addr(&sh.acc_s[tid - stages]), 1u);
            mbar_init(smem_addr(&sh.acc_t[tid - stages]), 1u);
        } else if (tid == stages + kMaxTiles) {
            mbar_init(smem_addr(&sh.acc_o), 1u);
            mbar_init(smem_addr(&sh.x_ready), 1u);
            mbar_init(smem_addr(&sh.u_ready), 1u);
            sh.abort_flag = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        proxy_fence();
    } else if (tid >= 64 && tid < 70) {
        const CUtensorMap* maps[6] = {&map_k1, &map_x1, &map_k2, &map_x2, &map_v, &map_u};
#pragma unroll
        for (int i = 0; i < 6; ++i)
            if (tid == 64 + i) tma_prefetch_desc(maps[i]);
    }
    if (warp == 1) tmem_alloc(smem_addr(&sh.tmem), p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t base = (smem_addr(tc_raw) + 1023u) & ~1023u;
    const uint32_t tmem = sh.tmem;
    volatile int* abort_flag = &sh.abort_flag;

    if (warp == 0) {
        // The whole warp walks the loops, one elected lane issues, and nothing divides: with `i % stages` and the maps chosen per
        // chunk inside `if (lane == 0)` a chunk took 0.45 us whatever its size, and this warp bounded the kernel.
        const uint32_t elected = elect_lane();
        const uint32_t xbytes = static_cast<uint32_t>(2 * p.ntok) * (kChunk * 2), wbytes = static_cast<uint32_t>(p.rows) * (kChunk * 2), sb = static_cast<uint32_t>(p.stage_bytes);
        const uint32_t full0 = smem_addr(&sh.full[0]), empty0 = smem_addr(&sh.empty[0]);
        int s = 0, issued = 0;                        // next stage; chunks whose weights have been requested
        uint32_t parity = 1u;                         // of the next wait for an empty stage: the first round finds them empty
        bool ok = true;
        auto wait_empty = [&]() { return ok = ok && __all_sync(kFull, mbar_wait(empty0 + 8 * s, parity, abort_flag)); };
        auto advance = [&]() {
            ++issued;
            if (++s == stages) { s = 0; parity ^= 1u; }
        };
        const int pre = min(n1, stages), row0 = cta * p.rows, row_step = gridDim.x * p.rows;
        int c = 0, row = row0;
        auto step = [&](int cn) {
            if (++c == cn) { c = 0; row += row_step; }
        };
        // scores: the weights of the first stages, X behind the barrier, then both
        for (int i = 0; i < pre; ++i, step(c1n), advance()) {
            mbar_expect_tx_elected(full0 + 8 * s, wbytes + xbytes, elected);
            tma_load_2d_elected(base + s * sb, &map_k1, full0 + 8 * s, c * kChunk, row, elected);
        }
        if (nt > 0) {
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.x_ready), 0u, abort_flag));
            proxy_fence();
            for (int i = 0, cx = 0; i < pre && ok; ++i) {
                tma_load_2d_elected(base + i * sb + kStreamTileBytes, &map_x1, full0 + 8 * i, cx * kChunk, 0, elected);
                if (++cx == c1n) cx = 0;
            }
        }
        for (int i = pre; i < n1 && wait_empty(); ++i, step(c1n), advance()) {
            mbar_expect_tx_elected(full0 + 8 * s, wbytes + xbytes, elected);
            tma_load_2d_elected(base + s * sb, &map_k1, full0 + 8 * s, c * kChunk, row, elected);
            tma_load_2d_elected(base + s * sb + kStreamTileBytes, &map_x1, full0 + 8 * s, c * kChunk, 0, elected);
        }
        c = 0;
        row = row0;
        for (int i = n1; i < n12 && wait_empty(); ++i, step(c2n), advance()) {
            mbar_expect_tx_elected(full0 + 8 * s, wbytes + xbytes, elected);
            tma_load_2d_elected(base + s * sb, &map_k2, full0 + 8 * s, c * kChunk, row, elected);
            tma_load_2d_elected(base + s * sb + kStreamTileBytes, &map_x2, full0 + 8 * s, c * kChunk, 0, elected);
        }
        // output: weights into every stage that comes free and the next ones into L2, U behind the barrier, then both
        if (outs) {
            const int col = otile * kStreamRows, ahead = min(cv1 - cv0, stages), s0 = s;
            auto load_v = [&](int cv) {
                mbar_expect_tx_elected(full0 + 8 * s, kStreamTileBytes + xbytes, elected);
                tma_load_2d_elected(base + s * sb, &map_v, full0 + 8 * s, col, cv * kChunk, elected);
                tma_load_2d_elected(base + s * sb + kChunk * 128, &map_v, full0 + 8 * s, col + 64, cv * kChunk, elected);
            };
            for (int i = 0; i < ahead && wait_empty(); ++i, advance()) load_v(cv0 + i);
            if (lane == 0)
                for (int cv = cv0 + ahead; cv < min(cv1, cv0 + ahead + kAhead); ++cv) {
                    tma_prefetch_2d(&map_v, col, cv * kChunk);
                    tma_prefetch_2d(&map_v, col + 64, cv * kChunk);
                }
            __syncwarp();
            ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.u_ready), 0u, abort_flag));
            proxy_fence();
            for (int i = 0, si = s0; i < ahead && ok; ++i) {
                tma_load_2d_elected(base + si * sb + kStreamTileBytes, &map_u, full0 + 8 * si, (cv0 + i) * kChunk, 0, elected);
                if (++si == stages) si = 0;
            }
            for (int cv = cv0 + ahead; cv < cv1 && wait_empty(); ++cv, advance()) {
                load_v(cv);
                tma_load_2d_elected(base + s * sb + kStreamTileBytes, &map_u, full0 + 8 * s, cv * kChunk, 0, elected);
            }
        }
        if (*abort_flag != 0 && lane == 0) {      // the copies in flight get a bounded time to land before the block goes
            for (int i = max(0, issued - stages); i < issued; ++i) {
                const long long t0 = clock64();
                while (!mbar_try(smem_addr(&sh.full[i % stages]), static_cast<uint32_t>(i / stages) & 1u))
                    if (clock64() - t0 > kTcSpinLimit / 64) break;
            }
        }
    } else if (warp == 1) {
        const uint32_t elected = elect_lane();
        int s = 0;
        uint32_t parity = 0u;
        bool ok = true;
        auto product = [&](int len, uint32_t acc, bool mn, unsigned long long* done) {
            const uint32_t idesc = instr_desc(128, 2 * p.ntok, mn), lbo = mn ? kChunk * 128u : 0u;
            const uint64_t step = mn ? 128 : 2;          // 16 K elements on, in 16-byte units: sixteen rows of 128 bytes, or 32 bytes of a row
            uint32_t more = 0u;
            for (int i = 0; i < len && ok; ++i, more = 1u) {
                ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), parity, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = base + s * p.stage_bytes;
                // a tile of fewer than 128 neurons: the rows behind are what the stage held before, and their results are not looked at
                const uint64_t ad = smem_desc(a0, lbo, 1024u), xd = smem_desc(a0 + kStreamTileBytes, 0u, 1024u);
#pragma unroll
                for (int j = 0; j < kChunk / 16; ++j) umma_bf16_elected(acc, ad + step * j, xd + 2 * j, idesc, j == 0 ? more : 1u, elected);
                umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                if (++s == stages) { s = 0; parity ^= 1u; }
            }
            if (ok) umma_commit_elected(smem_addr(done), elected);
        };
        for (int t = 0; t < nt; ++t) product(c1n, tmem + static_cast<uint32_t>(4 * t * p.ntok), false, &sh.acc_s[t]);
        for (int t = 0; t < nt; ++t) product(c2n, tmem + static_cast<uint32_t>((4 * t + 2) * p.ntok), false, &sh.acc_t[t]);
        if (outs) product(cv1 - cv0, tmem, true, &sh.acc_o);        // over the scores: U is complete, so they have been read
    } else {
        const int et = tid - 64, ew = warp - 2, q = warp & 3, half = ew >> 2;      // tensor-memory lanes 32 q ..; the warp's groups of 16 tokens
        const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
        WsHeader* hdr = p.f.hdr;
        dep_wait();
        dep_trigger();
        const unsigned epoch = ld_acquire_u32(&hdr->epoch), gen = ld_acquire_u32(&hdr->l1_gen);
        // ---- x in two terms; y = y_init (or 0), count = 0, the cells of the launch after next ----
        for (int i = cta; i < B * p.parts; i += gridDim.x) {
            const int t = i / p.parts, part = i - t * p.parts, d4 = d >> 2;
            const float4* xr = reinterpret_cast<const float4*>(p.f.x + static_cast<int64_t>(t) * d);
            float sc = 1.f;
            if (p.f.norm_w != nullptr) {        // every part sums the whole row (9 KB out of L2)
                float ss = 0.f;
                for (int j = et; j < d4; j += kEpi) {
                    const float4 v = xr[j];
                    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
                }
                ss = warp_sum(ss);
                if (lane == 0) sh.red[ew] = ss;
                epi_sync();
                float tot = 0.f;
#pragma unroll
                for (int w = 0; w < 8; ++w) tot += sh.red[w];
                sc = rsqrtf(tot / static_cast<float>(d) + p.f.eps);
                epi_sync();
            }
            uint2* hi = reinterpret_cast<uint2*>(p.g.xs + static_cast<int64_t>(t) * d);
            uint2* lo = reinterpret_cast<uint2*>(p.g.xs + static_cast<int64_t>(p.ntok + t) * d);
            for (int j = part * d4 / p.parts + et; j < (part + 1) * d4 / p.parts; j += kEpi) {
                float4 v = xr[j];
                if (p.f.norm_w != nullptr) {
                    const float4 w = reinterpret_cast<const float4*>(p.f.norm_w)[j];
                    v = make_float4(v.x * sc * w.x, v.y * sc * w.y, v.z * sc * w.z, v.w * sc * w.w);
                }
                uint2 h, l;
                split_pair(v.x, v.y, h.x, l.x);
                split_pair(v.z, v.w, h.y, l.y);
                hi[j] = h;
                lo[j] = l;
            }
        }
        if (cta == 0 && p.f.count != nullptr && et < B) p.f.count[et] = 0;
        epi_sync();
        if (ew == 0) {
            if (lane == 0) grid_arrive(hdr);
            __syncwarp();
            grid_wait(hdr, gen + 1u, abort_flag);
            if (lane == 0) mbar_arrive(smem_addr(&sh.x_ready));
        } else {
            SumCell* next = &hdr->ffn_cells[(epoch + 2u) & 3u][0][0][0];       // last used two launches ago
            const int i0 = cta * (kEpi - 32) + et - 32, step = gridDim.x * (kEpi - 32);
            for (int i = i0; i < kTok * kCellWays; i += step) { next[i].s1 = 0.0; next[i].s2 = 0.0; next[i].count = 0u; }
            if (p.f.y_init != p.f.y) {
                const int total4 = B * (d >> 2);
                const float4* yi = reinterpret_cast<const float4*>(p.f.y_init);
                float4* yo = reinterpret_cast<float4*>(p.f.y);
                for (int i = i0; i < total4; i += step) yo[i] = yi != nullptr ? yi[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        // ---- score sums ----
        SumCell* cells = &hdr->ffn_cells[epoch & 3u][0][0][0];                 // [token][way]
        bool ok = true;
        for (int t = 0; t < nt && ok; ++t) {
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_s[t]), 0u, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const int r = q * 32 + lane;
            const bool mine = r < p.rows && (cta + t * static_cast<int>(gridDim.x)) * p.rows + r < dff;
            float* w = sh.win[ew];
            for (int n0 = 16 * half; n0 < p.ntok && q * 32 < p.rows; n0 += 32) {
                float v[16];
                const uint32_t at = tmem + lanes + static_cast<uint32_t>(4 * t * p.ntok + n0);
                tmem_ld16_sum(at, at + p.ntok, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) w[lane * 17 + i] = mine ? v[i] : 0.f;
                __syncwarp();
                double s1 = 0.0, s2 = 0.0;                // lane: token lane % 16, half of the neurons
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const double x = static_cast<double>(w[((lane >> 4) * 16 + i) * 17 + (lane & 15)]);
                    s1 += x;
                    s2 = fma(x, x, s2);
                }
                s1 += __shfl_xor_sync(kFull, s1, 16);
                s2 += __shfl_xor_sync(kFull, s2, 16);
                double* out = &sh.sums[q][lane >> 4][n0 + (lane & 15)];
                *out = (t > 0 ? *out : 0.0) + (lane < 16 ? s1 : s2);
                __syncwarp();
            }
        }
        epi_sync();
        if (nt > 0 && ok) {
            const int b = et & 63, which = et >> 6;       // the quarters of the tile together: one addition per block, token and sum
            if (which < 2 && b < B) {
                double v = sh.sums[0][which][b];
                for (int w = 1; w < (p.rows + 31) / 32; ++w) v += sh.sums[w][which][b];
                SumCell* c = cells + b * kCellWays + (cta & (kCellWays - 1));
                red_add_f64(which == 0 ? &c->s1 : &c->s2, v);
            }
        }
        epi_sync();
        if (ew == 0) {
            if (lane == 0) grid_arrive(hdr);
            __syncwarp();
            grid_wait(hdr, gen + 2u, abort_flag);
        }
        epi_sync();
        // ---- theta: four threads per token, four ways each ----
        {
            const int b = et >> 2;
            double s1 = 0.0, s2 = 0.0;
            if (b < B) {
#pragma unroll
                for (int w = 0; w < kCellWays / 4; ++w) {
                    const double2 c = __ldcg(reinterpret_cast<const double2*>(cells + b * kCellWays + (et & 3) * (kCellWays / 4) + w));
                    s1 += c.x;
                    s2 += c.y;
                }
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                s1 += __shfl_xor_sync(kFull, s1, o);
                s2 += __shfl_xor_sync(kFull, s2, o);
            }
            if ((et & 3) == 0) {
                float th = INFINITY;                       // tokens that are not there
                if (b < B) {
                    th = -INFINITY;
                    if (!p.f.identity) {
                        const double mean = s1 * p.f.inv_n;
                        const float var = static_cast<float>((s2 - s1 * mean) * p.f.inv_nm1);
                        th = static_cast<float>(mean) + sqrtf(fmaxf(var, 0.f)) * static_cast<float>(p.f.z);
                    }
                    if (cta == 0 && p.f.theta != nullptr) p.f.theta[b] = th;
                }
                sh.theta[b] = th;
            }
        }
        epi_sync();
        // ---- U ----
        unsigned act[kMaxTiles] = {0u, 0u};               // tokens for which this lane's neuron is active: 16 bits per group of tokens
#pragma unroll
        for (int t = 0; t < kMaxTiles; ++t) {
            if (t >= nt || !ok) break;
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_t[t]), 0u, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const int r = q * 32 + lane, row = (cta + t * static_cast<int>(gridDim.x)) * p.rows + r;
            const bool mine = r < p.rows && row < dff, odd = lane & 1;
            for (int n0 = 16 * half, g = 0; n0 < p.ntok && q * 32 < p.rows; n0 += 32, ++g) {
                const uint32_t at = tmem + lanes + static_cast<uint32_t>(4 * t * p.ntok + n0);
                float u[16], v[16];
                tmem_ld16_sum(at, at + p.ntok, u);
                tmem_ld16_sum(at + 2 * p.ntok, at + 3 * p.ntok, v);
                unsigned on = 0u;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float th = sh.theta[n0 + i];
                    const bool active = mine && u[i] > th;
                    const float a = p.f.identity ? u[i] : u[i] - th;
                    on |= active ? 1u << i : 0u;
                    u[i] = active ? (p.f.erf_form ? gelu_erf(a) : gelu_logistic(a)) * v[i] : 0.f;
                }
                act[t] |= on << (16 * g);
                // even lanes store this pair of neurons for the even tokens, odd lanes for the odd ones
                __nv_bfloat16* uh = p.g.us + (n0 + (odd ? 1 : 0)) * dff + row - (odd ? 1 : 0);
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    const float own = odd ? u[i + 1] : u[i], other = __shfl_xor_sync(kFull, odd ? u[i] : u[i + 1], 1);
                    unsigned hi, lo;
                    split_pair(odd ? other : own, odd ? own : other, hi, lo);
                    if (mine && n0 + i + (odd ? 1 : 0) < B) {
                        *reinterpret_cast<unsigned*>(uh + i * dff) = hi;
                        *reinterpret_cast<unsigned*>(uh + (p.ntok + i) * dff) = lo;
                    }
                }
            }
        }
        tc_fence_before();
        epi_sync();
        if (ew == 0) {
            if (lane == 0) grid_arrive(hdr);
            __syncwarp();
            grid_wait(hdr, gen + 3u, abort_flag);
            if (lane == 0) {
                mbar_arrive(smem_addr(&sh.u_ready));
                if (cta == 0) {                            // every block has read both by now
                    hdr->epoch = epoch + 1u;
                    hdr->l1_gen = gen + 3u;
                }
            }
            __syncwarp();
        }
        // ---- counts and index lists, under the output product ----
        if (p.f.count != nullptr && ok) {
            // a warp's share of a token's list is contiguous and ascending; warps take their places in the order in which they
            // get here.  Lane i asks for token n0 + i: one round trip for sixteen tokens
#pragma unroll
            for (int t = 0; t < kMaxTiles; ++t) {
                if (t >= nt) break;
                const int row = (cta + t * static_cast<int>(gridDim.x)) * p.rows + q * 32 + lane;
                for (int n0 = 16 * half, g = 0; n0 < p.ntok && q * 32 < p.rows; n0 += 32, ++g) {
                    const unsigned on = act[t] >> (16 * g) & 0xffffu;
                    int at = 0;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const unsigned b = __ballot_sync(kFull, on >> i & 1u);
                        if (lane == i) at = __popc(b);
                    }
                    if (at > 0) at = atomicAdd(&p.f.count[n0 + lane], at);
                    if (p.f.idx != nullptr) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const unsigned b = __ballot_sync(kFull, on >> i & 1u);
                            const int first = __shfl_sync(kFull, at, i);
                            if (on >> i & 1u) p.f.idx[(n0 + i) * dff + first + __popc(b & ((1u << lane) - 1u))] = row;
                        }
                    }
                }
            }
        }
        // ---- Y ----
        if (outs && __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_o), 0u, abort_flag))) {
            tc_fence_after();
            const int64_t col = otile * kStreamRows + q * 32 + lane;
            for (int n0 = 16 * half; n0 < p.ntok; n0 += 32) {
                float v[16];
                tmem_ld16_sum(tmem + lanes + n0, tmem + lanes + p.ntok + n0, v);
                if (col < d) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (n0 + i < B) atomicAdd(p.f.y + static_cast<int64_t>(n0 + i) * d + col, v[i]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, p.tmem_cols);
    }
    if (tid == 0 && sh.abort_flag != 0) atomicCAS(&p.f.hdr->status, SPARK_OK, SPARK_ERR_TIMEOUT);
}

}  // namespace

namespace spark {

size_t ffn_tc_workspace_bytes(int64_t d, int64_t d_ff) {
    const size_t one = tc_region_bytes(d, d_ff), chain = ffn_chain_workspace_bytes(d, d_ff);
    return one > chain ? one : chain;
}

// SPARK_ERR_WORKSPACE = shape or workspace not served by this path (the caller falls back).
int ffn_tc_launch(spark_ctx* ctx, FfnParams& f, cudaStream_t stream) {
    const int d = f.d, r = f.r, d_ff = f.d_ff, B = f.B, sms = ctx->num_sms;
    // operand rows start on 16-byte boundaries; widths that are no multiple of a box arrive padded with zeros
    if (B < 1 || B > kTok || (d & 7) != 0 || (r & 7) != 0 || (d_ff & 7) != 0 || r < kChunk || d - r < kChunk || d_ff < kChunk || f.K1s != nullptr) return SPARK_ERR_WORKSPACE;
    if (ctx->scratch == nullptr || ctx->scratch_bytes < kAttnCellBytes + tc_region_bytes(d, d_ff)) return SPARK_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(f.K1t) | reinterpret_cast<uintptr_t>(f.K2t) | reinterpret_cast<uintptr_t>(f.Vt)) & 15u) return SPARK_ERR_WORKSPACE;

    // Up to 16 MB of weights (2.5 us of the stream) and 16 tokens as a chain of kernels: a barrier costs more than a chained launch, a
    // launch stops the stream.  Measured at 1 MB, 6 MB: 16.3, 16.4 us here and 14.4, 14.4 there; at 67 MB, 6 tokens: 26.1 and 26.6.
    if (B <= 16 && static_cast<int64_t>(d) * d_ff * 4 <= (16 << 20)) {
        const int rc = ffn_chain_launch(ctx, f, stream);
        if (rc != SPARK_ERR_WORKSPACE) return rc;
    }
    TcParams p;
    p.f = f;
    p.g = tc_region(ctx->scratch + kAttnCellBytes, d);             // behind the attention's persistent cells
    p.ntok = (B + 15) & ~15;
    // as many neurons per tile as give every block the same number of tiles: 9B, 14336 neurons: 138 tiles of 104 instead of 112 of 128
    const int per = ((d_ff + kStreamRows - 1) / kStreamRows + sms - 1) / sms;
    p.otiles = (d + kStreamRows - 1) / kStreamRows;
    if (per > kMaxTiles || p.otiles > sms) return SPARK_ERR_WORKSPACE;
    p.rows = ((d_ff + per * sms - 1) / (per * sms) + 7) & ~7;
    if (p.rows < kMinRows) p.rows = kMinRows;
    p.tiles = (d_ff + p.rows - 1) / p.rows;
    const int cvn = (d_ff + kChunk - 1) / kChunk;
    p.ksplit = sms / p.otiles < cvn ? sms / p.otiles : cvn;
    p.parts = sms / B > 1 ? sms / B : 1;
    p.stage_bytes = kStreamTileBytes + 2 * p.ntok * kChunk * 2;
    const int limit = ctx->max_smem_optin - static_cast<int>(sizeof(FfnShared)) - 256, fit = (limit - 1024) / p.stage_bytes;
    if (fit < 2) return SPARK_ERR_WORKSPACE;
    const int most = per * ((r + kChunk - 1) / kChunk + (d - r + kChunk - 1) / kChunk) + (cvn + p.ksplit - 1) / p.ksplit;      // chunks of a block
    p.stages = fit < kMaxStages ? fit : kMaxStages;
    if (p.stages > most) p.stages = most;              // small shapes: room for the blocks of the kernel ahead
    p.tmem_cols = 32;
    while (p.tmem_cols < static_cast<uint32_t>(4 * per * p.ntok)) p.tmem_cols *= 2;

    CUtensorMap m_k1, m_k2, m_x1, m_x2, m_v, m_u;
    if (!make_map(&m_k1, f.K1t, d_ff, r, r, p.rows, true) || !make_map(&m_k2, f.K2t, d_ff, d - r, d - r, p.rows, true) ||
        !make_map(&m_x1, p.g.xs, 2 * p.ntok, r, d, 2 * p.ntok, false) || !make_map(&m_x2, p.g.xs + r, 2 * p.ntok, d - r, d, 2 * p.ntok, false) ||
        !make_map(&m_v, f.Vt, d_ff, d, d, kChunk, true) || !make_map(&m_u, p.g.us, 2 * p.ntok, d_ff, d_ff, 2 * p.ntok, false))
        return SPARK_ERR_WORKSPACE;
    // Blocks that hold tensor memory while they wait for other blocks: no more of their kind may share an SM than there are columns
    // for, so each takes at least the shared memory that keeps the next one out.
    const size_t want = static_cast<size_t>(p.stages) * p.stage_bytes + 1024, least = (static_cast<size_t>(ctx->max_smem_optin) + 1024) / (512 / p.tmem_cols + 1);
    const void* kern = reinterpret_cast<const void*>(ffn_tc_kernel);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess) return SPARK_ERR_CUDA;
    void* args[] = {&p, &m_k1, &m_x1, &m_k2, &m_x2, &m_v, &m_u};
    return launch_kernel(ctx, kern, static_cast<unsigned>(sms), kFfnThreads, want > least ? want : least, stream, true, args) == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
