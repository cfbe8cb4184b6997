// The weight-streaming GEMM of the token-chunk kernels (tcgen05): D[rows][tokens] = A[rows][K] . X[tokens][K]^T for up to
// 64 tokens, A a bf16 weight matrix that is read once, X the fp32 activations as two bf16 terms (hi rows, then lo rows).
//
// What bounds it is the weight stream, so the split of the work is by bytes: the (tile, K chunk) pairs of all tiles form one
// sequence, tile after tile, and every block takes a contiguous part of it, whatever the number of tiles.  A tile that falls to
// several blocks is completed by the caller's epilogue (reductions into an initialised output).  Per block: warp 0 moves
// 64-element K chunks of A (128 rows) and X (both terms in one box) with TMA through a ring of stages, warp 1 issues the MMAs and
// four epilogue warps drain one of two accumulator sets while the next segment runs.  Both terms are one operand tile of
// N = 2 x tokens, so the weight tile is read from shared memory once.  The weights do not depend on the kernel ahead: their first
// stages are requested before griddepcontrol.wait.  Bounded waits as in tc_common.cuh.
// Measured, 64 tokens, 256000 x 2304: 201 us = 5.9 TB/s (0.90 of the measured copy rate); 17 tokens 182 us (0.99).
#pragma once

#include "tc_common.cuh"

namespace spark {
namespace tc {

constexpr int kStreamMaxStages = 8;
constexpr int kStreamRows = 128;
constexpr int kStreamTileBytes = kStreamRows * kChunk * 2;

struct StreamShared {
    unsigned long long full[kStreamMaxStages], empty[kStreamMaxStages];
    unsigned long long acc_full[2], acc_empty[2];
    uint32_t tmem;
    int abort_flag;
};

struct StreamPlan {
    int total;               // K chunks of all tiles
    int grid, per;           // blocks; chunks a block takes (0: equal parts of the sequence or of each tile)
    int part, rem;           // an equal part is `part` chunks, one more for the first `rem` of them (of the sequence, or of a tile)
    int split;               // every tile is cut into this many pieces (0: no such regular cut)
    uint32_t inv_split;      // 65536 / split + 1: block / split for fewer than 65536 / split blocks
    int call;                // K chunks of a tile
    int rows;                // rows of a tile: 128, or a smaller multiple of 8 (the MMAs' other rows read whatever lies behind and are dropped)
    int ntok;                // token t's term i is row i * ntok + t of X: two terms, ntok a multiple of 16; kStreamFew: three terms, ntok = 4
    int xrows;               // rows of X: the MMAs' N
    int stages;
    int stage_bytes;
    uint32_t tmem_cols;
};

// A block's part of the sequence: its first tile, the K chunk it starts at and the number of chunks.  No division where every
// block has one piece of a tile: this sits in front of the first load.
struct StreamPart {
    int tile, c, n;
};
__host__ __device__ inline StreamPart stream_part(const StreamPlan& sp, int block) {
    if (sp.split > 0) {
        const int tile = static_cast<int>(static_cast<uint32_t>(block) * sp.inv_split >> 16), i = block - tile * sp.split;
        return StreamPart{tile, i * sp.part + (i < sp.rem ? i : sp.rem), sp.part + (i < sp.rem ? 1 : 0)};
    }
    const int p0 = sp.per > 0 ? block * sp.per : block * sp.part + (block < sp.rem ? block : sp.rem), tile = p0 / sp.call;
    const int left = sp.total - p0, n = sp.per > 0 ? (left < sp.per ? left : sp.per) : sp.part + (block < sp.rem ? 1 : 0);
    return StreamPart{tile, p0 - tile * sp.call, n};
}

// Alignment of the first tile, and room behind the last one for an operand of 128 rows that starts in it.
inline size_t stream_slack(const StreamPlan& sp) { return 1024 + static_cast<size_t>(sp.stage_bytes < kStreamTileBytes ? kStreamTileBytes - sp.stage_bytes : 0); }

// Host: fills in the plan for at most `smem_limit` bytes of dynamic shared memory.  whole: a block takes one whole tile, however many
// there are (the caller needs whole products).  False: does not fit.
inline bool stream_plan(StreamPlan& sp, int sms, int tiles, int call, int tokens, size_t smem_limit, bool whole = false, int rows = kStreamRows, bool few = false) {
    sp.call = call;
    sp.total = tiles * call;
    sp.rows = rows;
    sp.per = sp.split = 0;
    // A piece of a tile costs its block an epilogue (1.5 to 4 us with the reductions of 16 to 64 tokens), so blocks get one piece
    // of one tile, or whole tiles, where that leaves 0.6 / 0.9 of the SMs busy: fewer SMs still draw what HBM gives (4096 x 2304,
    // 64 tokens: 128 blocks of one piece 9.7 us, 148 equal parts of two pieces each 15.4 us).  Otherwise equal parts.
    const int ks = sms / tiles < call ? sms / tiles : call, m = (tiles + sms - 1) / sms;
    if (whole) {
        sp.per = call;
        sp.grid = tiles;
    } else if (ks >= 1 && (tiles * ks * 10 >= sms * 6 || ks == call)) {
        sp.split = ks;
        sp.grid = tiles * ks;
    } else if (tiles > sms && m <= 4 && (tiles + m - 1) / m * 10 >= sms * 9) {
        sp.per = m * call;
        sp.grid = (tiles + m - 1) / m;
    } else {
        sp.grid = sp.total < sms ? sp.total : sms;
    }
    const int of = sp.split > 0 ? call : sp.total, by = sp.split > 0 ? sp.split : sp.grid;
    sp.part = of / by;
    sp.rem = of % by;
    sp.inv_split = sp.split > 0 ? 65536u / static_cast<uint32_t>(sp.split) + 1u : 0u;
    sp.ntok = few ? 4 : (tokens + 15) & ~15;
    sp.xrows = few ? 16 : 2 * sp.ntok;
    sp.stage_bytes = (rows + sp.xrows) * kChunk * 2;
    const int fit = static_cast<int>((smem_limit - stream_slack(sp)) / sp.stage_bytes);
    // more than eight stages (128 KB of weights in flight per SM, three times what the latency of HBM needs) only delays the
    // small loads of the kernel ahead that queue behind them
    sp.stages = fit < kStreamMaxStages ? fit : kStreamMaxStages;
    // no more than a block has chunks, and a second accumulator only for a second piece: blocks of small products fit on an SM beside
    // those of the kernel ahead and set up under its tail
    const int most = sp.per > 0 ? sp.per : sp.part + (sp.rem > 0 ? 1 : 0);
    if (sp.stages > most) sp.stages = most > 2 ? most : 2;
    uint32_t cols = 32;
    while (cols < static_cast<uint32_t>((sp.split > 0 || sp.per == call ? 1 : 2) * sp.xrows)) cols *= 2;
    sp.tmem_cols = cols;
    return sp.stages >= 2 && cols <= 512 && tiles > 0 && call > 0;
}
inline size_t stream_smem(const StreamPlan& sp) { return static_cast<size_t>(sp.stages) * sp.stage_bytes + stream_slack(sp); }

// Variants of stream_gemm():
//   kStreamEarlyX   X is complete when the kernel starts: its producer is two places ahead in the stream and the kernel ahead is
//                   kStreamLate.  The products run before griddepcontrol.wait; only the epilogue needs the kernel ahead.
//   kStreamLate     the kernel behind may start once this one has seen the end of the kernel ahead (implied by kStreamEarlyX);
//                   otherwise at once: it only requests its weights before it waits for this kernel
//   kStreamMN       A is stored [K][rows] (two boxes of 64 rows per K chunk)
//   kStreamFew      up to four tokens in three bf16 terms each (x = hi + mid + lo, all 24 bits of an fp32 value): 12 of 16 rows of X
constexpr int kStreamEarlyX = 1, kStreamLate = 2, kStreamMN = 4, kStreamFew = 8;

// One block's work.  before() runs in the four epilogue warps once the kernel ahead is complete.  epi(tile, whole, row, n0, v):
// sixteen tokens' values of one row of a tile (a whole warp calls it; rows from sp.rows on are to be dropped); `whole`: the block
// holds all of the tile's K range.
template <int V, class Before, class Epi>
__device__ __forceinline__ void stream_gemm(const StreamPlan& sp, StreamShared& sh, unsigned char* raw, const CUtensorMap* map_w,
                                            const CUtensorMap* map_x, WsHeader* hdr, Before before, Epi epi) {
    constexpr bool kEarlyX = (V & kStreamEarlyX) != 0, kLate = (V & (kStreamEarlyX | kStreamLate)) != 0, kMN = (V & kStreamMN) != 0, kFew = (V & kStreamFew) != 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const StreamPart part = stream_part(sp, blockIdx.x);
    const int n = part.n;
    const uint32_t wbytes = static_cast<uint32_t>(sp.rows) * (kChunk * 2), stage_bytes = static_cast<uint32_t>(sp.stage_bytes);
    const int stages = sp.stages;
    if (tid == 64) {         // descriptors first: a miss behind the dependency wait costs 0.3 us
        tma_prefetch_desc(map_w);
        tma_prefetch_desc(map_x);
    }
    if (tid < 32) {
        if (tid < stages) {
            mbar_init(smem_addr(&sh.full[tid]), 1u);
            mbar_init(smem_addr(&sh.empty[tid]), 1u);
        } else if (tid < stages + 2) {
            const int b = tid - stages;
            mbar_init(smem_addr(&sh.acc_full[b]), 1u);
            mbar_init(smem_addr(&sh.acc_empty[b]), 4u);
        }
        if (tid == 0) sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_addr(&sh.tmem), sp.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t base = (smem_addr(raw) + 1023u) & ~1023u;
    const uint32_t tmem = sh.tmem;
    volatile int* abort_flag = &sh.abort_flag;
    if (!kLate) dep_trigger();
    auto load_w = [&](uint32_t dst, uint32_t bar, int c, int tile) {
        if (kMN) {
            tma_load_2d(dst, map_w, bar, tile * kStreamRows, c * kChunk);
            tma_load_2d(dst + kChunk * 128, map_w, bar, tile * kStreamRows + 64, c * kChunk);
        } else {
            tma_load_2d(dst, map_w, bar, c * kChunk, tile * sp.rows);
        }
    };

    if (warp == 0) {
        if (lane == 0) {
            int tile = part.tile, c = part.c, cx = c;
            const int pre = min(n, stages);
            for (int i = 0; i < pre; ++i) {
                const uint32_t bar = smem_addr(&sh.full[i]);
                mbar_expect_tx(bar, stage_bytes);
                load_w(base + i * stage_bytes, bar, c, tile);
                if (++c == sp.call) { c = 0; ++tile; }
            }
            if (!kEarlyX) dep_wait();
            for (int i = 0; i < pre; ++i) {
                tma_load_2d(base + i * stage_bytes + wbytes, map_x, smem_addr(&sh.full[i]), cx * kChunk, 0);
                if (++cx == sp.call) cx = 0;
            }
            int s = 0, issued = pre;
            uint32_t parity = 0u;
            for (int i = pre; i < n; ++i) {
                if (!mbar_wait(smem_addr(&sh.empty[s]), parity, abort_flag)) break;
                const uint32_t bar = smem_addr(&sh.full[s]), dst = base + s * stage_bytes;
                mbar_expect_tx(bar, stage_bytes);
                load_w(dst, bar, c, tile);
                tma_load_2d(dst + wbytes, map_x, bar, c * kChunk, 0);
                if (++c == sp.call) { c = 0; ++tile; }
                if (++s == stages) { s = 0; parity ^= 1u; }
                issued = i + 1;
            }
            if (*abort_flag != 0) {      // the copies in flight land (bounded) before the block goes
                for (int i = max(0, issued - stages); i < issued; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try(smem_addr(&sh.full[i % stages]), static_cast<uint32_t>(i / stages) & 1u))
                        if (clock64() - t0 > kTcSpinLimit) break;
                }
            }
        }
    } else if (warp == 1) {
        // the whole warp walks the loop; one elected lane issues
        const uint32_t elected = elect_lane(), idesc = instr_desc(128, sp.xrows, kMN);
        int s = 0, seg = 0;
        uint32_t parity = 0u;
        bool ok = true;
        for (int done = 0, len = min(n, sp.call - part.c); done < n && ok; done += len, len = min(n - done, sp.call)) {
            const int b = seg & 1;
            if (seg >= 2) ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.acc_empty[b]), ((seg >> 1) & 1) ^ 1, abort_flag));
            const uint32_t acc = tmem + static_cast<uint32_t>(b * sp.xrows);
            tc_fence_after();
            uint32_t more = 0u;
            for (int i = 0; i < len; ++i, more = 1u) {
                ok = __all_sync(kFull, mbar_wait(smem_addr(&sh.full[s]), parity, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = base + s * stage_bytes;
                // 16 K elements further: 32 bytes in a row of K, or sixteen rows of 128 bytes
                const uint64_t ad = smem_desc(a0, kMN ? kChunk * 128u : 0u, 1024u), xd = smem_desc(a0 + wbytes, 0u, 1024u);
#pragma unroll
                for (int j = 0; j < kChunk / 16; ++j)      // descriptors count in 16-byte units
                    umma_bf16_elected(acc, ad + (kMN ? 128 : 2) * j, xd + 2 * j, idesc, j == 0 ? more : 1u, elected);
                umma_commit_elected(smem_addr(&sh.empty[s]), elected);
                if (++s == stages) { s = 0; parity ^= 1u; }
            }
            if (ok) umma_commit_elected(smem_addr(&sh.acc_full[b]), elected);
            ++seg;
        }
    } else {
        const int q = warp & 3;                                    // tensor-memory lanes 32 q .. 32 q + 31
        dep_wait();
        if (kLate) dep_trigger();
        before();
        int seg = 0, tile = part.tile;
        for (int done = 0, len = min(n, sp.call - part.c); done < n; done += len, len = min(n - done, sp.call), ++tile) {
            const int b = seg & 1;
            if (!__all_sync(kFull, mbar_wait(smem_addr(&sh.acc_full[b]), (seg >> 1) & 1, abort_flag))) break;      // warp-uniform: tcgen05.ld is warp-wide
            tc_fence_after();
            const uint32_t taddr = tmem + static_cast<uint32_t>(b * sp.xrows) + (static_cast<uint32_t>(q * 32) << 16);
            for (int n0 = 0; n0 < sp.ntok && q * 32 < sp.rows; n0 += 16) {
                float v[16];
                if (kFew) {
                    tmem_ld16(taddr, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = i < 4 ? v[i] + (v[i + 4] + v[i + 8]) : 0.f;
                } else {
                    tmem_ld16_sum(taddr + n0, taddr + sp.ntok + n0, v);
                }
                epi(tile, len == sp.call, q * 32 + lane, n0, v);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.acc_empty[b])) : "memory");
            ++seg;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, sp.tmem_cols);
    }
    if (tid == 0 && sh.abort_flag != 0) atomicCAS(&hdr->status, SPARK_OK, SPARK_ERR_TIMEOUT);
}

// The two bf16 terms of an fp32 value pair: x = hi + lo, 16 significant bits.
__device__ __forceinline__ void split_pair(float a, float b, unsigned& hi, unsigned& lo) {
    hi = pack2_bf16(a, b);
    lo = pack2_bf16(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xffff0000u));
}

// The three bf16 terms of an fp32 value pair: x = hi + mid + lo.
__device__ __forceinline__ void split_pair3(float a, float b, unsigned& hi, unsigned& mid, unsigned& lo) {
    hi = pack2_bf16(a, b);
    const float ra = a - __uint_as_float(hi << 16), rb = b - __uint_as_float(hi & 0xffff0000u);
    mid = pack2_bf16(ra, rb);
    lo = pack2_bf16(ra - __uint_as_float(mid << 16), rb - __uint_as_float(mid & 0xffff0000u));
}

}  // namespace tc
}  // namespace spark
