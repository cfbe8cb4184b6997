// Spark attention (Section 2.2, Eq. 7) for a span of a prompt: T consecutive tokens of one sequence over one cache, token t seeing
// rows [lo_t, n_t), n_t = start + t + 1.  The queries of a KV head are taken 128 (token, head) columns at a time -- a "virtual
// head": tps = 128 / heads-per-KV-head tokens, columns ordered token-major -- and are the M dimension of every product, so that
// a thread owns one column: the sums over the cached rows, the threshold, the weights' sum are scalars in its registers.  With
// the selection of Eq. 7 as a mask on dense weights every row is read once per virtual head.  Two kernels:
//   sums   S1 = Q1 . k1c^T, 128 rows per tile; per column the sum, the sum of squares (around the tile's first row, in fp64 above)
//          and the maximum of the scores the token may see.  The scores themselves are not kept:
//   main   per tile of 64 rows S1 again and S2 = Q2 . k2c^T, weights w = [s1 > theta] exp(s1 - max) softplus(s2) as two bf16
//          terms, written over the scores in tensor memory, O += W . V with W as the tensor-memory operand; the sum of
//          exp(s1 - max) over the survivors normalises (left to the caller).
// The queries enter as two bf16 terms like everywhere else.  The (virtual head, row tile) pairs form one sequence cut into equal
// parts, one per SM: a block walks one to three pieces; their results are added into o and lsum.
// What bounds it: main's tensor work per 128 columns x 128 rows (S1 and S2 with K = 2 x 128, O with two terms: 4096 cycles);
// sixteen warps form the weights of two tiles in turn meanwhile (eight warps with 64 rows each, everything unrolled: 4.3 us per
// tile, issue slots 29 % busy).
#include "kernels.h"
#include "stream_gemm.cuh"

using namespace spark;
using namespace spark::tc;

namespace {

constexpr int kVCols = 128;           // columns of a virtual head
constexpr int kVSubMax = 128;         // sub-chunks (groups of tps tokens) of a span
constexpr int kVThreads = 64 + 8 * 32;      // warp 0: TMA, warp 1: MMA + tensor memory, warps 2..9: columns
constexpr int kQBox = kVCols * 128;   // 64 K elements of 128 operand rows
constexpr int kSumSlots = 4;
constexpr int kSumRows = 128;
constexpr int kMainSlots = 3;
constexpr int kMainRows = 64;
constexpr int kMainBox = kMainRows * 128;
constexpr int kMainSlotBytes = 4 * kMainBox;
constexpr int kMainWarps = 16;        // main: four warps per lane quadrant -- two tiles in work, two halves of their rows
constexpr int kMainThreads = 64 + 32 * kMainWarps;

struct VParams {
    int T, n_q, n_kv, gq, hd, r, tps, nsub, start, window, k_attn;
    int nk1, nk2, nvb;                // 64-element boxes of a query's two parts and of a value row
    const double* zt;
    double* sums;                     // [columns][2]
    unsigned* smax;                   // [columns] ordered
    float* o;
    float* lsum;
    WsHeader* hdr;
    int tiles[kVSubMax + 1];          // row tiles of all virtual heads of the sub-chunks before this one
    int first[kVSubMax];              // first row tile of a sub-chunk
};

struct Piece {                        // consecutive row tiles of one virtual head
    int sub, g, tile0, n;
};
__device__ __forceinline__ Piece piece_at(const VParams& p, int tile, int end, int sub) {
    while (tile >= p.tiles[sub + 1]) ++sub;
    const int per = (p.tiles[sub + 1] - p.tiles[sub]) / p.n_kv, i = tile - p.tiles[sub], g = i / per;
    return Piece{sub, g, p.first[sub] + i - g * per, min(end - tile, per - (i - g * per))};
}
struct Column {                       // what a thread knows of its column
    int t, h, lo, n;
    bool valid;
};
__device__ __forceinline__ Column column_of(const VParams& p, const Piece& pc, int col) {
    Column c;
    c.t = pc.sub * p.tps + col / p.gq;
    c.h = pc.g * p.gq + col % p.gq;
    c.valid = c.t < p.T;
    c.n = p.start + c.t + 1;
    c.lo = (p.window > 0 && p.window < c.n) ? c.n - p.window : 0;
    return c;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
// D[tmem] (+)= A[tmem] . B[smem]
__device__ __forceinline__ void umma_ts_elected(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const unsigned (&v)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
                   "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// The block's range of the sequence.
__device__ __forceinline__ void my_range(const VParams& p, int& t0, int& t1) {
    const int total = p.tiles[p.nsub], part = total / gridDim.x, rem = total - part * gridDim.x, b = blockIdx.x;
    t0 = b * part + min(b, rem);
    t1 = t0 + part + (b < rem ? 1 : 0);
}

// ---- sums ---------------------------------------------------------------------------------------------------------------------
struct SumShared {
    unsigned long long full[kSumSlots], empty[kSumSlots], acc_full[2], acc_empty[2], q_full, q_empty;
    uint32_t tmem;
    int abort_flag;
};

__global__ void __launch_bounds__(kVThreads, 1)
span_attn_sums_kernel(const __grid_constant__ VParams p, const __grid_constant__ CUtensorMap map_k1, const __grid_constant__ CUtensorMap map_qhi,
                      const __grid_constant__ CUtensorMap map_qlo) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ SumShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 64)
        for (const CUtensorMap* m : {&map_k1, &map_qhi, &map_qlo}) tma_prefetch_desc(m);
    if (tid == 0) {
        for (int s = 0; s < kSumSlots; ++s) {
            mbar_init(smem_addr(&sh.full[s]), 1u);
            mbar_init(smem_addr(&sh.empty[s]), 1u);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_addr(&sh.acc_full[b]), 1u);
            mbar_init(smem_addr(&sh.acc_empty[b]), 8u);
        }
        mbar_init(smem_addr(&sh.q_full), 1u);
        mbar_init(smem_addr(&sh.q_empty), 1u);
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_addr(&sh.tmem), 256u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t qbase = (smem_addr(tc_raw) + 1023u) & ~1023u, ring = qbase + 4 * kQBox;
    const uint32_t tmem = sh.tmem;
    volatile int* abort_flag = &sh.abort_flag;
    int t0, t1;
    my_range(p, t0, t1);
    dep_wait();                  // everything read here comes from the kernels ahead
    dep_trigger();

    if (warp == 0) {
        if (lane == 0) {
            int it = 0, pieces = 0, sub = 0;
            bool ok = true;
            for (int tile = t0; tile < t1 && ok;) {
                const Piece pc = piece_at(p, tile, t1, sub);
                sub = pc.sub;
                const int vrow = (sub * p.n_kv + pc.g) * kVCols;
                if (pieces > 0 && !mbar_wait(smem_addr(&sh.q_empty), static_cast<uint32_t>(pieces - 1) & 1u, abort_flag)) break;
                const uint32_t qbar = smem_addr(&sh.q_full);
                mbar_expect_tx(qbar, static_cast<uint32_t>(2 * p.nk1) * kQBox);
                for (int kc = 0; kc < p.nk1; ++kc) {
                    tma_load_2d(qbase + kc * kQBox, &map_qhi, qbar, kc * kChunk, vrow);
                    tma_load_2d(qbase + (p.nk1 + kc) * kQBox, &map_qlo, qbar, kc * kChunk, vrow);
                }
                for (int i = 0; i < pc.n; ++i, ++it) {
                    const int s = it % kSumSlots;
                    if (it >= kSumSlots && !mbar_wait(smem_addr(&sh.empty[s]), ((it / kSumSlots) & 1) ^ 1, abort_flag)) { ok = false; break; }
                    const uint32_t bar = smem_addr(&sh.full[s]);
                    mbar_expect_tx(bar, static_cast<uint32_t>(p.nk1) * kQBox);
                    for (int kc = 0; kc < p.nk1; ++kc) tma_load_3d(ring + (2 * s + kc) * kQBox, &map_k1, bar, kc * kChunk, (pc.tile0 + i) * kSumRows, pc.g);
                }
                tile += pc.n;
                ++pieces;
            }
            if (*abort_flag != 0) {          // the copies in flight land (bounded) before the block goes
                const long long c0 = clock64();
                while (!mbar_try(smem_addr(&sh.q_full), static_cast<uint32_t>(pieces - 1) & 1u) && clock64() - c0 < kTcSpinLimit) {}
                for (int i = max(0, it - kSumSlots); i < it; ++i)
                    while (!mbar_try(smem_addr(&sh.full[i % kSumSlots]), (i / kSumSlots) & 1) && clock64() - c0 < kTcSpinLimit) {}
            }
        }
    } else if (warp == 1) {
        const uint32_t elected = elect_lane(), idesc = instr_desc(128, kSumRows, false);
        int it = 0, pieces = 0, sub = 0;
        bool ok = true;
        for (int tile = t0; tile < t1 && ok;) {
            const Piece pc = piece_at(p, tile, t1, sub);
            sub = pc.sub;
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.q_full), static_cast<uint32_t>(pieces) & 1u, abort_flag));
            for (int i = 0; i < pc.n && ok; ++i, ++it) {
                const int s = it % kSumSlots, b = it & 1;
                if (it >= 2) ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_empty[b]), ((it >> 1) & 1) ^ 1, abort_flag));
                ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), (it / kSumSlots) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after();
                uint32_t more = 0u;
                for (int t = 0; t < 2; ++t)
                    for (int kc = 0; kc < p.nk1; ++kc) {
                        const uint64_t qd = smem_desc(qbase + (t * p.nk1 + kc) * kQBox, 0u, 1024u), kd = smem_desc(ring + (2 * s + kc) * kQBox, 0u, 1024u);
#pragma unroll
                        for (int j = 0; j < kChunk / 16; ++j, more = 1u) umma_bf16_elected(tmem + b * kSumRows, qd + 2 * j, kd + 2 * j, idesc, more, elected);
                    }
                umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                umma_commit_elected(smem_addr(&sh.acc_full[b]), elected);
            }
            if (ok) umma_commit_elected(smem_addr(&sh.q_empty), elected);
            tile += pc.n;
            ++pieces;
        }
    } else {
        // two warps per tensor-memory lane quadrant: lane = column, each with half of the tile's rows
        const int q = warp & 3, half = (warp - 2) >> 2, col = q * 32 + lane;
        int it = 0, sub = 0;
        bool ok = true;
        for (int tile = t0; tile < t1 && ok;) {
            const Piece pc = piece_at(p, tile, t1, sub);
            sub = pc.sub;
            const Column c = column_of(p, pc, col);
            double s1 = 0.0, s2 = 0.0;
            float mx = -INFINITY;
            for (int i = 0; i < pc.n; ++i, ++it) {
                const int b = it & 1, row0 = (pc.tile0 + i) * kSumRows + half * 64;
                ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_full[b]), (it >> 1) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after();
                float v[64];
                const uint32_t taddr = tmem + b * kSumRows + half * 64 + (static_cast<uint32_t>(q * 32) << 16);
                tmem_ld32(taddr, *reinterpret_cast<float(*)[32]>(v));
                tmem_ld32(taddr + 32, *reinterpret_cast<float(*)[32]>(v + 32));
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&sh.acc_empty[b]));
                // sums around one of the tile's own values (keeps the fp32 partial sums accurate when |mean| >> std)
                float f1 = 0.f, f2 = 0.f, ref;
                int cnt = 64;
                if (__all_sync(kFull, row0 >= c.lo && row0 + 64 <= c.n)) {
                    ref = v[0];
#pragma unroll
                    for (int k = 0; k < 64; ++k) {
                        const float d = v[k] - ref;
                        f1 += d;
                        f2 = fmaf(d, d, f2);
                        mx = fmaxf(mx, v[k]);
                    }
                } else {
                    const int a = max(c.lo - row0, 0), e = min(c.n - row0, 64);      // the rows [a, e) of the tile
                    cnt = max(e - a, 0);
                    ref = a <= 0 ? v[0] : (e >= 64 ? v[63] : 0.f);
#pragma unroll
                    for (int k = 0; k < 64; ++k) {
                        const bool in = k >= a && k < e;
                        const float d = in ? v[k] - ref : 0.f;
                        f1 += d;
                        f2 = fmaf(d, d, f2);
                        mx = fmaxf(mx, in ? v[k] : -INFINITY);
                    }
                    if (cnt == 0) ref = 0.f;
                }
                const double rd = ref, nd = cnt;
                s1 += static_cast<double>(f1) + nd * rd;
                s2 += static_cast<double>(f2) + rd * (2.0 * f1 + nd * rd);
            }
            if (ok && c.valid) {
                const int64_t vcol = static_cast<int64_t>(sub * p.n_kv + pc.g) * kVCols + col;
                red_add_f64(p.sums + 2 * vcol, s1);
                red_add_f64(p.sums + 2 * vcol + 1, s2);
                atomicMax(p.smax + vcol, f32_to_ordered(mx));
            }
            tile += pc.n;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, 256u);
    }
    if (tid == 0 && sh.abort_flag != 0) atomicCAS(&p.hdr->status, SPARK_OK, SPARK_ERR_TIMEOUT);
}

// ---- main ---------------------------------------------------------------------------------------------------------------------
struct MainShared {
    unsigned long long full[kMainSlots], empty[kMainSlots], s_full[2], p_full[2], pv_done[2], q_full, q_empty, o_full;
    uint32_t tmem;
    int abort_flag;
};
// Sixteen scores and sixteen gate products of this thread's column, one wait.
__device__ __forceinline__ void tmem_ld16_pair(uint32_t ta, uint32_t tb, float (&a)[16], float (&b)[16]) {
    unsigned r[16], s[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(s[0]), "=r"(s[1]),
                   "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7]), "=r"(s[8]), "=r"(s[9]), "=r"(s[10]),
                   "=r"(s[11]), "=r"(s[12]), "=r"(s[13]), "=r"(s[14]), "=r"(s[15])
                 : "r"(ta), "r"(tb) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        a[i] = __uint_as_float(r[i]);
        b[i] = __uint_as_float(s[i]);
    }
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__global__ void __launch_bounds__(kMainThreads, 1)
span_attn_main_kernel(const __grid_constant__ VParams p, const __grid_constant__ CUtensorMap map_k1, const __grid_constant__ CUtensorMap map_k2,
                      const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_qhi, const __grid_constant__ CUtensorMap map_qlo,
                      const __grid_constant__ CUtensorMap map_q2hi, const __grid_constant__ CUtensorMap map_q2lo) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ MainShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 64)
        for (const CUtensorMap* m : {&map_k1, &map_k2, &map_v, &map_qhi, &map_qlo, &map_q2hi, &map_q2lo}) tma_prefetch_desc(m);
    if (tid == 0) {
        for (int s = 0; s < kMainSlots; ++s) {
            mbar_init(smem_addr(&sh.full[s]), 1u);
            mbar_init(smem_addr(&sh.empty[s]), 1u);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_addr(&sh.s_full[b]), 1u);
            mbar_init(smem_addr(&sh.p_full[b]), 8u);
            mbar_init(smem_addr(&sh.pv_done[b]), 1u);
        }
        mbar_init(smem_addr(&sh.q_full), 1u);
        mbar_init(smem_addr(&sh.q_empty), kMainWarps);
        mbar_init(smem_addr(&sh.o_full), 1u);
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_addr(&sh.tmem), 512u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // shared memory: Q1 hi, Q1 lo, Q2 hi, Q2 lo (at most two boxes each), then the ring
    const uint32_t qbase = (smem_addr(tc_raw) + 1023u) & ~1023u, ring = qbase + 8 * kQBox;
    unsigned char* qgen = tc_raw + (qbase - smem_addr(tc_raw));
    const uint32_t tmem = sh.tmem;               // O: columns 0..255; buffer b: scores 256 + 128 b, gate products 64 behind them
    volatile int* abort_flag = &sh.abort_flag;
    int t0, t1;
    my_range(p, t0, t1);
    dep_wait();
    dep_trigger();

    // ring items of a piece of n tiles: K(0), then per tile K(i + 1) if there is one, V(i)
    if (warp == 0) {
        if (lane == 0) {
            int it = 0, pieces = 0, sub = 0;
            bool ok = true;
            for (int tile = t0; tile < t1 && ok;) {
                const Piece pc = piece_at(p, tile, t1, sub);
                sub = pc.sub;
                const int vrow = (sub * p.n_kv + pc.g) * kVCols;
                auto slot = [&]() -> bool { return it < kMainSlots || mbar_wait(smem_addr(&sh.empty[it % kMainSlots]), ((it / kMainSlots) & 1) ^ 1, abort_flag); };
                auto load_k = [&](int i) {
                    if (!(ok = ok && slot())) return;
                    const uint32_t bar = smem_addr(&sh.full[it % kMainSlots]), dst = ring + (it % kMainSlots) * kMainSlotBytes;
                    mbar_expect_tx(bar, static_cast<uint32_t>(p.nk1 + p.nk2) * kMainBox);
                    for (int kc = 0; kc < p.nk1; ++kc) tma_load_3d(dst + kc * kMainBox, &map_k1, bar, kc * kChunk, (pc.tile0 + i) * kMainRows, pc.g);
                    for (int kc = 0; kc < p.nk2; ++kc) tma_load_3d(dst + (2 + kc) * kMainBox, &map_k2, bar, kc * kChunk, (pc.tile0 + i) * kMainRows, pc.g);
                    ++it;
                };
                auto load_v = [&](int i) {
                    if (!(ok = ok && slot())) return;
                    const uint32_t bar = smem_addr(&sh.full[it % kMainSlots]), dst = ring + (it % kMainSlots) * kMainSlotBytes;
                    mbar_expect_tx(bar, static_cast<uint32_t>(p.nvb) * kMainBox);
                    for (int vb = 0; vb < p.nvb; ++vb) tma_load_3d(dst + vb * kMainBox, &map_v, bar, vb * 64, (pc.tile0 + i) * kMainRows, pc.g);
                    ++it;
                };
                if (pieces > 0 && !mbar_wait(smem_addr(&sh.q_empty), static_cast<uint32_t>(pieces - 1) & 1u, abort_flag)) break;
                const uint32_t qbar = smem_addr(&sh.q_full);
                mbar_expect_tx(qbar, static_cast<uint32_t>(2 * (p.nk1 + p.nk2)) * kQBox);
                for (int kc = 0; kc < p.nk1; ++kc) {
                    tma_load_2d(qbase + kc * kQBox, &map_qhi, qbar, kc * kChunk, vrow);
                    tma_load_2d(qbase + (2 + kc) * kQBox, &map_qlo, qbar, kc * kChunk, vrow);
                }
                for (int kc = 0; kc < p.nk2; ++kc) {
                    tma_load_2d(qbase + (4 + kc) * kQBox, &map_q2hi, qbar, kc * kChunk, vrow);
                    tma_load_2d(qbase + (6 + kc) * kQBox, &map_q2lo, qbar, kc * kChunk, vrow);
                }
                load_k(0);
                for (int i = 0; i < pc.n && ok; ++i) {
                    if (i + 1 < pc.n) load_k(i + 1);
                    load_v(i);
                }
                tile += pc.n;
                ++pieces;
            }
            if (*abort_flag != 0) {
                const long long c0 = clock64();
                while (!mbar_try(smem_addr(&sh.q_full), static_cast<uint32_t>(pieces - 1) & 1u) && clock64() - c0 < kTcSpinLimit) {}
                for (int i = max(0, it - kMainSlots); i < it; ++i)
                    while (!mbar_try(smem_addr(&sh.full[i % kMainSlots]), (i / kMainSlots) & 1) && clock64() - c0 < kTcSpinLimit) {}
            }
        }
    } else if (warp == 1) {
        const uint32_t elected = elect_lane(), idesc_s = instr_desc(128, kMainRows, false);
        const uint32_t idesc_o = instr_desc(128, p.nvb * 64, false) | (1u << 16);      // B (the value rows) MN-major
        int it = 0, cnt = 0, pieces = 0, sub = 0;
        bool ok = true;
        for (int tile = t0; tile < t1 && ok;) {
            const Piece pc = piece_at(p, tile, t1, sub);
            sub = pc.sub;
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.q_full), static_cast<uint32_t>(pieces) & 1u, abort_flag));
            auto scores = [&](int gi) {          // S1 and S2 of tile number gi into buffer gi & 1
                const int b = gi & 1, s = it % kMainSlots;
                if (gi >= 2) ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.pv_done[b]), ((gi >> 1) & 1) ^ 1, abort_flag));
                ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), (it / kMainSlots) & 1, abort_flag));
                if (!ok) return;
                tc_fence_after();
                const uint32_t k0 = ring + s * kMainSlotBytes, acc = tmem + 256u + 128u * b;
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const int nk = w == 0 ? p.nk1 : p.nk2;
                    uint32_t more = 0u;
                    for (int t = 0; t < 2; ++t)
                        for (int kc = 0; kc < nk; ++kc) {
                            const uint64_t qd = smem_desc(qbase + (4 * w + 2 * t + kc) * kQBox, 0u, 1024u), kd = smem_desc(k0 + (2 * w + kc) * kMainBox, 0u, 1024u);
#pragma unroll
                            for (int j = 0; j < kChunk / 16; ++j, more = 1u) umma_bf16_elected(acc + 64u * w, qd + 2 * j, kd + 2 * j, idesc_s, more, elected);
                        }
                }
                umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                umma_commit_elected(smem_addr(&sh.s_full[b]), elected);
                ++it;
            };
            if (ok) scores(cnt);
            for (int i = 0; i < pc.n && ok; ++i) {
                const int gi = cnt + i, b = gi & 1;
                if (i + 1 < pc.n) scores(gi + 1);
                const int s = it % kMainSlots;
                ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.p_full[b]), (gi >> 1) & 1, abort_flag));
                ok = ok && __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), (it / kMainSlots) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const uint64_t vd = smem_desc(ring + s * kMainSlotBytes, kMainBox, 1024u);
                const uint32_t w0 = tmem + 256u + 128u * b;
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int j = 0; j < kMainRows / 16; ++j)      // sixteen rows: eight tensor-memory columns of weights, two 8-row groups of V
                        umma_ts_elected(tmem, w0 + 16u * j + 8u * t, vd + 128 * j, idesc_o, (i == 0 && t == 0 && j == 0) ? 0u : 1u, elected);
                umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                umma_commit_elected(smem_addr(&sh.pv_done[b]), elected);
                ++it;
            }
            if (ok) umma_commit_elected(smem_addr(&sh.o_full), elected);
            cnt += pc.n;
            tile += pc.n;
            ++pieces;
        }
    } else {
        // lane = column; warps 0..7 and 8..15 take alternate tiles, the two warps of a quadrant 32 rows each.  The weights of sixteen
        // rows go where their scores were: hi terms in the first eight columns, lo terms in the other eight.
        const int q = warp & 3, wi = warp - 2, wg = wi >> 3, half = (wi >> 2) & 1, col = q * 32 + lane;
        const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
        constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
        int cnt = 0, pieces = 0, sub = 0;
        bool ok = true;
        for (int tile = t0; tile < t1 && ok;) {
            const Piece pc = piece_at(p, tile, t1, sub);
            sub = pc.sub;
            const Column c = column_of(p, pc, col);
            float th = INFINITY, mx2 = 0.f, z = 0.f;      // threshold, maximum in units of log 2, sum of the softmax terms
            if (c.valid) {
                const int64_t vcol = static_cast<int64_t>(sub * p.n_kv + pc.g) * kVCols + col;
                const int L = c.n - c.lo;
                mx2 = ordered_to_f32(__ldcg(p.smax + vcol)) * kLog2e;
                th = -INFINITY;
                if (p.k_attn < L) {
                    const double s1 = __ldcg(p.sums + 2 * vcol), s2 = __ldcg(p.sums + 2 * vcol + 1), mean = s1 / L, var = (s2 - s1 * mean) / (L - 1);
                    th = static_cast<float>(mean + sqrt(var > 0.0 ? var : 0.0) * p.zt[c.t]);
                }
            }
            for (int i = 0; i < pc.n; ++i) {
                const int gi = cnt + i, b = gi & 1;
                if (b != wg) continue;
                ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.s_full[b]), (gi >> 1) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const int row0 = (pc.tile0 + i) * kMainRows + 32 * half;
                const bool inner = __all_sync(kFull, row0 >= c.lo && row0 + 32 <= c.n);      // no range test per element
#pragma unroll 1
                for (int hf = 0; hf < 2; ++hf) {
                    const uint32_t sc = tmem + 256u + 128u * b + 32u * half + 16u * hf + lanes;
                    float s1[16], s2[16];
                    tmem_ld16_pair(sc, sc + 64, s1, s2);
                    if (!inner) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const int row = row0 + 16 * hf + k;
                            s1[k] = row >= c.lo && row < c.n ? s1[k] : -INFINITY;
                        }
                    }
                    unsigned w[16];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        float v[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float a = s1[2 * k + e], g = s2[2 * k + e];
                            // softplus(g) = max(g, 0) + log(1 + x), x = exp(-|g|): the hardware logarithm of 1 + x loses x below 1e-4
                            const float x = ex2(-fabsf(g) * kLog2e);
                            const float l1p = x < 1e-4f ? fmaf(-0.5f * x, x, x) : lg2(1.f + x) * kLn2;
                            const float ex = a > th ? ex2(fmaf(a, kLog2e, -mx2)) : 0.f;
                            z += ex;
                            v[e] = ex * (fmaxf(g, 0.f) + l1p);
                        }
                        split_pair(v[0], v[1], w[k], w[8 + k]);
                    }
                    tmem_st16(sc, w);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&sh.p_full[b]));
            }
            if (!ok) break;
            // the piece's sums: through shared memory (the queries have been consumed), so that a warp adds runs of 128 bytes
            ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.o_full), static_cast<uint32_t>(pieces) & 1u, abort_flag));
            if (!ok) break;
            tc_fence_after();
            constexpr int kPitch = 36;
            float* stage = reinterpret_cast<float*>(qgen) + wi * (32 * 64);      // 8 KB per warp: 32 columns x 32 values at a time
            const unsigned long long orow = static_cast<unsigned long long>(c.valid ? reinterpret_cast<uintptr_t>(p.o + (static_cast<int64_t>(c.t) * p.n_q + c.h) * p.hd) : 0);
            for (int u = 0; u < 2; ++u) {                  // the quadrant's four warps take 64 value columns each
                const int c0 = 64 * (wi >> 2) + 32 * u;
                if (c0 >= p.hd) break;
                float v[32];
                tmem_ld32(tmem + c0 + lanes, v);
#pragma unroll
                for (int k = 0; k < 8; ++k) *reinterpret_cast<float4*>(stage + lane * kPitch + 4 * k) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                __syncwarp();
                for (int k = 0; k < 8; ++k) {              // four columns at a time, eight lanes each
                    const int cl = 4 * k + (lane >> 3), x = 4 * (lane & 7);
                    const unsigned long long row = __shfl_sync(kFull, orow, cl);
                    const float4 a = *reinterpret_cast<const float4*>(stage + cl * kPitch + x);
                    if (row != 0ull && c0 + x < p.hd) red_add_v4(reinterpret_cast<float*>(row) + c0 + x, a.x, a.y, a.z, a.w);
                }
                __syncwarp();
            }
            if (c.valid) atomicAdd(p.lsum + static_cast<int64_t>(c.t) * p.n_q + c.h, z);
            tc_fence_before();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the next piece's queries land where the staging was
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&sh.q_empty));
            cnt += pc.n;
            tile += pc.n;
            ++pieces;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, 512u);
    }
    if (tid == 0 && sh.abort_flag != 0) atomicCAS(&p.hdr->status, SPARK_OK, SPARK_ERR_TIMEOUT);
}

// [heads][rows][cols] bf16 with `cap` rows from head to head: what lies behind row `rows` reads as zeros (rows nobody has written
// yet may hold anything, and 0 x NaN would poison a sum).
bool make_map_rows(CUtensorMap* map, const void* ptr, int64_t heads, int64_t rows, int64_t cols, int64_t cap, int box_rows) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (enc == nullptr) return false;
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(heads)};
    const cuuint64_t strides[2] = {static_cast<cuuint64_t>(cols) * 2, static_cast<cuuint64_t>(cap) * static_cast<cuuint64_t>(cols) * 2};
    const cuuint32_t box[3] = {static_cast<cuuint32_t>(kChunk), static_cast<cuuint32_t>(box_rows), 1u};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The sequence of row tiles: sub-chunk after sub-chunk, KV head after KV head.
void fill_tiles(VParams& p, int rows_per_tile) {
    p.tiles[0] = 0;
    for (int sub = 0; sub < p.nsub; ++sub) {
        const int first_tok = p.start + sub * p.tps, end = p.start + ((sub + 1) * p.tps < p.T ? (sub + 1) * p.tps : p.T);
        const int lo = (p.window > 0 && p.window < first_tok + 1) ? first_tok + 1 - p.window : 0;
        p.first[sub] = lo / rows_per_tile;
        p.tiles[sub + 1] = p.tiles[sub] + p.n_kv * ((end + rows_per_tile - 1) / rows_per_tile - lo / rows_per_tile);
    }
}

}  // namespace

namespace spark {

int64_t attn_span_columns(int64_t T, int64_t n_q, int64_t n_kv) {
    const int64_t tps = kVCols / (n_q / n_kv);
    return (T + tps - 1) / tps * n_kv * kVCols;
}

size_t attn_span_bytes(int64_t T, int64_t n_q, int64_t n_kv, int64_t hd) {
    const size_t cols = static_cast<size_t>(attn_span_columns(T, n_q, n_kv));
    return round_up(static_cast<size_t>(T) * sizeof(double), 1024) + round_up(cols * 16, 1024) + round_up(cols * 4, 1024) +
           4 * 1024 + 2 * cols * static_cast<size_t>(hd) * 2;
}

bool attn_span_layout(AttnSpan& a, char* w) {
    const int64_t d2 = a.hd - a.r;
    a.tps = static_cast<int>(kVCols / (a.n_q / a.n_kv));
    a.nsub = static_cast<int>((a.T + a.tps - 1) / a.tps);
    a.colcap = kVCols;
    const size_t cols = static_cast<size_t>(attn_span_columns(a.T, a.n_q, a.n_kv));
    a.zt = reinterpret_cast<double*>(w); w += round_up(static_cast<size_t>(a.T) * sizeof(double), 1024);
    a.sums = reinterpret_cast<double*>(w); w += round_up(cols * 16, 1024);
    a.smax = reinterpret_cast<unsigned*>(w); w += round_up(cols * 4, 1024);
    a.qhi = reinterpret_cast<__nv_bfloat16*>(w); w += round_up(cols * a.r * 2, 1024);
    a.qlo = reinterpret_cast<__nv_bfloat16*>(w); w += round_up(cols * a.r * 2, 1024);
    a.q2hi = reinterpret_cast<__nv_bfloat16*>(w); w += round_up(cols * d2 * 2, 1024);
    a.q2lo = reinterpret_cast<__nv_bfloat16*>(w);
    return a.nsub <= kVSubMax;
}

int attn_span_launch(spark_ctx* ctx, const AttnSpan& a, cudaStream_t stream) {
    const int64_t d2 = a.hd - a.r, rows = a.start + a.T, vrows = static_cast<int64_t>(a.nsub) * a.n_kv * kVCols;
    const size_t smem_sums = 4 * static_cast<size_t>(kQBox) + kSumSlots * 2 * static_cast<size_t>(kQBox) + 1024;
    const size_t smem_main = 8 * static_cast<size_t>(kQBox) + kMainSlots * static_cast<size_t>(kMainSlotBytes) + 1024;
    VParams p;
    p.T = static_cast<int>(a.T); p.n_q = static_cast<int>(a.n_q); p.n_kv = static_cast<int>(a.n_kv); p.gq = static_cast<int>(a.n_q / a.n_kv);
    p.hd = static_cast<int>(a.hd); p.r = static_cast<int>(a.r); p.tps = a.tps; p.nsub = a.nsub; p.start = static_cast<int>(a.start);
    p.window = static_cast<int>(a.window > 0x7fffffff ? 0x7fffffff : a.window);
    p.k_attn = static_cast<int>(a.k_attn > 0x7fffffff ? 0x7fffffff : a.k_attn);
    p.nk1 = static_cast<int>((a.r + kChunk - 1) / kChunk); p.nk2 = static_cast<int>((d2 + kChunk - 1) / kChunk); p.nvb = static_cast<int>((a.hd + 63) / 64);
    p.zt = a.zt; p.sums = a.sums; p.smax = a.smax; p.o = a.o; p.lsum = a.lsum;
    p.hdr = ctx->hdr;
    CUtensorMap m_k1a, m_k1, m_k2, m_v, m_qhi, m_qlo, m_q2hi, m_q2lo;
    if (!make_map_rows(&m_k1a, a.k1c, a.n_kv, rows, a.r, a.cap, kSumRows) || !make_map_rows(&m_k1, a.k1c, a.n_kv, rows, a.r, a.cap, kMainRows) ||
        !make_map_rows(&m_k2, a.k2c, a.n_kv, rows, d2, a.cap, kMainRows) || !make_map_rows(&m_v, a.vc, a.n_kv, rows, a.hd, a.cap, kMainRows) ||
        !make_map(&m_qhi, a.qhi, vrows, a.r, a.r, kVCols, false) || !make_map(&m_qlo, a.qlo, vrows, a.r, a.r, kVCols, false) ||
        !make_map(&m_q2hi, a.q2hi, vrows, d2, d2, kVCols, false) || !make_map(&m_q2lo, a.q2lo, vrows, d2, d2, kVCols, false))
        return SPARK_ERR_WORKSPACE;
    if (cudaFuncSetAttribute(span_attn_sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_sums)) != cudaSuccess ||
        cudaFuncSetAttribute(span_attn_main_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_main)) != cudaSuccess)
        return SPARK_ERR_CUDA;
    auto grid = [&]() { return static_cast<unsigned>(p.tiles[p.nsub] < ctx->num_sms ? p.tiles[p.nsub] : ctx->num_sms); };
    fill_tiles(p, kSumRows);
    {
        void* args[] = {&p, &m_k1a, &m_qhi, &m_qlo};
        if (launch_kernel(ctx, reinterpret_cast<const void*>(span_attn_sums_kernel), grid(), kVThreads, smem_sums, stream, false, args, true) != cudaSuccess) return SPARK_ERR_CUDA;
    }
    fill_tiles(p, kMainRows);
    void* args[] = {&p, &m_k1, &m_k2, &m_v, &m_qhi, &m_qlo, &m_q2hi, &m_q2lo};
    return launch_kernel(ctx, reinterpret_cast<const void*>(span_attn_main_kernel), grid(), kMainThreads, smem_main, stream, false, args, true) == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
