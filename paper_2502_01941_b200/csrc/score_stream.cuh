// Window attention scoring for units of more than 128 window rows (two 128-row blocks of Q), the
// kernel the prefill path runs first on them: the TMA producer, MMA issuers, work items and
// per-(piece, window row) outputs (m, z) of score_tc.cuh, the fixed reference exponent, the repair at the
// end and the two-pipe exponentials of score_fast.cuh, and an epilogue that never
// waits for tensor memory.
//
// Eight epilogue warps, one per (row block, tensor-memory lane quarter); a thread is one whole
// window row, so a piece's z (and the item's reference m) is written by one thread with no exchange.  The accumulator
// columns of the next 32-column chunk -- of the next tile too, once its barrier is seen complete
// -- are requested into a second set of registers before the arithmetic of the current chunk
// starts, so the load's latency runs beside the exponentials.  Where a piece ends inside a chunk
// the chunk's exponentials are split between the two pieces by multiplying with 0/1 masks read
// from a shared-memory table (one packed multiply-add per column pair and piece), which costs
// half the instructions of a predicated addition per column.
//
// What bounds this kernel on a B200 held at a 1 kW power cap is energy per tile, not a pipe: its
// epilogue takes the same cycles per tile with or without the MMAs running beside it, but the GPU
// settles near 1.5 GHz with them and at its full 1.96 GHz without.  The polynomial costs 5.5 issue
// slots per logit against 2 for the special-function path, so a larger share on the FMA pipe
// (PE of every 16 column pairs) saves cycles and spends energy.  Measured with 3 against 5 of 16: at the cap (4 x 32
// layers of 32K) 3,980 against 3,999 us a call, below it (one to four layers of 16K, 4 to 32 layers of 4K to 8K) 0 to 2 %
// faster, with 16-token units alone 1 % slower.
#pragma once
#include "score_fast.cuh"

namespace shotkv {

template <int D>
struct ScoreStreamCfg {
    static constexpr int kSub = D / 64;
    static constexpr int kSubBytes = 128 * 128;
    static constexpr int kQBytes = 2 * kSub * kSubBytes;
    static constexpr int kStageBytes = kSub * kSubBytes;
    static constexpr int kStages = D == 128 ? 4 : 6;
    static constexpr int kBarBytes = 1024;
    static constexpr int kCombBytes = tc::kSplitMaskBytes;     // split masks: [columns of the piece that ends][column pair] float4
    static constexpr int kSmemBytes = kQBytes + kStages * kStageBytes + kBarBytes + kCombBytes + 1024;
    static constexpr int kEpiWarps = 8;
    static constexpr int kThreads = 128 + kEpiWarps * 32;      // producer, two MMA issuers, one idle warp; epilogue
};


// SHORT: for units of few tokens, whose piece ends are most of the epilogue's control.  A piece's sum is then not looked at
// for itself: out of range, or not a number, it makes the sum of the item's pieces so, none of which is negative, and
// that is looked at once an item.  A test and two stores at every piece end cost 4 x 32 layers of 32K in 16-token chunks
// 7,667 us a call against 7,112, in sentences of 10 to 40 6,222 against 6,055; with shots of 200 to 480 tokens the
// compiler's schedule of the loop without them is the slower one (3,967 against 4,013).
template <int D, int PE, bool SHORT>
__global__ void __launch_bounds__(ScoreStreamCfg<D>::kThreads, 1)
    score_stream_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const int q_box_rows,
                        const int k_box_rows, const __grid_constant__ ScoreTcParams p, const __grid_constant__ ShotTable tab) {
    using Cfg = ScoreStreamCfg<D>;
    constexpr int TN = tc::kTileKeys, MB = 2;
    extern __shared__ unsigned char smem_raw[];
    grid_release();
    tc::prefetch_maps(&tmQ, &tmK);
    tc::Pipe<Cfg> pp;
    tc::pipe_setup(pp, smem_raw, 4, 0, 2);
    float4* mtab = reinterpret_cast<float4*>(tc::pipe_scratch(pp, smem_raw));   // split masks
    tc::build_split_masks(mtab);
    __syncthreads();
    grid_wait();
    tc::stamp(p.clk, 0);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int item_begin, item_end;
    tc::item_range(p, item_begin, item_end);

    if (warp == 0) {
        if (lane == 0) tc::producer_role<D, MB, false, false>(pp, &tmQ, &tmK, q_box_rows, k_box_rows, p, item_begin, item_end);
    } else if (warp == 1 || warp == 2) {
        if (lane == 0) tc::mma_role<D, MB, false, 2>(pp, p, item_begin, item_end, warp - 1);
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ epilogue
        // a warp may touch the 32 tensor-memory lanes given by its index modulo 4
        const int blk = (warp - 4) >> 2, quad = warp & 3;  // 128-row block of Q, lane quarter
        const int row = blk * 128 + quad * 32 + lane;
        const bool live = row < p.R;                       // padding rows: their Q was never loaded
        const int plim = live ? p.N - p.W + (row % p.W) : p.N - 1;
        const float scale = p.scale_log2;
        const int units_per_prompt = p.L * p.Hkv;
        const uint32_t tlane = pp.tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(blk * TN);
        int tiles_before = 0;                              // tiles of earlier items (fixes the accumulator buffer of every tile)
        uint32_t tfphase = 0;                              // bit a: the phase of buffer a's barrier
        bool ok = true;
        uint32_t ra[32], rb[32];                           // even and odd chunks of a tile
        for (int it = item_begin; it < item_end && ok; ++it) {
            const int u = it / p.nchunk, j = it - u * p.nchunk;
            const int lo = j * p.chunk_keys, hi = min(p.N, lo + p.chunk_keys);
            const int nt = max(0, (hi - lo + TN - 1) / TN);
            const int* o = table_row(tab, u / units_per_prompt);
            const int sg = count_le_warp(o, p.S + 1, lo);  // segment of the first piece
            // end of the current piece, and of the one after it (fetched one piece ahead)
            const int* next = o + sg + 1;
            int pend = next[-1], pend_n = next[0];
            // this warp's flag of the item: set when a sum leaves the range (the item is then recomputed below)
            if (lane == 0) reinterpret_cast<unsigned char*>(p.redo + it)[warp - 4] = 0;
            __syncwarp();
            float m_ref = SHOTKV_NEG_INF, neg = 0.f;       // reference exponent of this (row, item); neg = -m_ref
            uint64_t z[2] = {0ull, 0ull};                  // four running sums of the current piece, as two packed pairs
            const int plain_end = min(hi, p.N - p.W + 1);  // keys below this count for every window row
            float* out_z = p.part_z + ((size_t)u * p.P + sg + j) * p.Rpad + row;
            float zsum = 0.f;                              // sum of the item's pieces so far (they share m_ref)

            // the current piece is complete: write its partials and move on to the next piece
            auto flush = [&]() {
                float s0, s1, s2, s3;
                tc::unpack2(z[0], s0, s1);
                tc::unpack2(z[1], s2, s3);
                const float zz = (s0 + s1) + (s2 + s3);
                if (!SHORT && live && !(zz < tc::kRedoAbove)) {      // out of range, or not a number
                    reinterpret_cast<unsigned char*>(p.redo + it)[warp - 4] = 1;
                    *pp.repair_flag() = 1;
                }
                *out_z = live ? zz : 0.f;
                out_z += p.Rpad;
                zsum += zz;
                z[0] = z[1] = 0ull;
                pend = pend_n;
                pend_n = *++next;
            };

            // 32 columns starting at key kc that hold the end of the keys, the causal window, or a piece end
            auto chunk_slow = [&](uint32_t (&r)[32], int kc) {
                while (pend <= kc) flush();
                if (kc + 32 <= plain_end) {                              // every column counts; pieces end inside
                    tc::peel_chunk<PE>(r, scale, neg, mtab, kc, pend, z, flush);
                    return;
                }
                const int lim = min(hi, plim + 1) - kc;                  // columns of the chunk that count
                if (!__all_sync(0xffffffffu, lim >= 32)) tc::mask32(r, lim);
                tc::exp32(r, scale, neg);
                int start = 0;
                while (pend < kc + 32) {
                    const int e = pend - kc;
                    z[0] = tc::fadd2(z[0], tc::pack2(tc::range32(r, start, e), 0.f));
                    start = e;
                    flush();
                }
                z[0] = tc::fadd2(z[0], tc::pack2(tc::range32(r, start, 32), 0.f));
            };
            auto chunk = [&](uint32_t (&r)[32], int kc) {
                if (kc + 32 <= min(pend, plain_end)) tc::expacc32<PE>(r, scale, neg, z);
                else chunk_slow(r, kc);
            };
            // waits (bounded) until the accumulators of the tile in buffer `a` are complete
            auto wait_tile = [&](int a) {
                const uint32_t tph = (tfphase >> a) & 1u;
                // usually ready: one test by the whole warp, made uniform before anything depends on it
                if (!__all_sync(0xffffffffu, tc::mbar_try(pp.tfull(a, blk), tph))) {
                    bool w = lane == 0 ? tc::mbar_wait(pp.tfull(a, blk), tph, pp.abort_flag, p.err, p.wait_cycles) : true;   // one poller per warp
                    w = __shfl_sync(0xffffffffu, w, 0);
                    if (!w) ok = false;
                }
                tfphase ^= 1u << a;
                tc::fence_after_sync();
            };

            bool have_a = false;                            // chunk 0 of the next tile has been requested into ra
            if (nt > 0) {
                // the reference exponent: this thread's maximum over the item's first tile
                const int a = tiles_before & 1;
                wait_tile(a);
                if (ok) {
                    const uint32_t taddr = tlane + (uint32_t)(a * MB * TN);
                    float cm = SHOTKV_NEG_INF;
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        tc::tmem_ld32_sync(ra, taddr + c * 32);
                        const int lim = min(hi, plim + 1) - (lo + c * 32);
                        if (!__all_sync(0xffffffffu, lim >= 32)) tc::mask32(ra, lim);
                        cm = fmaxf(cm, tc::max32(ra));
                    }
                    if (cm != SHOTKV_NEG_INF) {
                        m_ref = fmaf(cm, scale, tc::kRefShift);
                        neg = -m_ref;
                    }
                    tc::tmem_ld32_issue(ra, taddr);
                    have_a = true;
                }
            }
            for (int t = 0; t < nt && ok; ++t) {
                const int a = (tiles_before + t) & 1;
                const int kc0 = lo + t * TN;
                const uint32_t taddr = tlane + (uint32_t)(a * MB * TN);
                if (!have_a) {                              // the barrier was not complete when the previous tile looked
                    wait_tile(a);
                    if (!ok) break;
                    tc::tmem_ld32_issue(ra, taddr);
                }
                tc::tmem_ld_wait(ra);
                tc::tmem_ld32_issue(rb, taddr + 32);
                chunk(ra, kc0);
                tc::tmem_ld_wait(rb);
                tc::tmem_ld32_issue(ra, taddr + 64);
                chunk(rb, kc0 + 32);
                tc::tmem_ld_wait(ra);
                tc::tmem_ld32_issue(rb, taddr + 96);
                chunk(ra, kc0 + 64);
                tc::tmem_ld_wait(rb);
                // all of this tile's accumulators are in registers: hand the buffer back
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(pp.tempty(a, blk));
                // request the first chunk of the next tile if its accumulators are complete already
                have_a = false;
                if (t + 1 < nt) {
                    const int an = a ^ 1;
                    const uint32_t tph = (tfphase >> an) & 1u;
                    if (__all_sync(0xffffffffu, tc::mbar_try(pp.tfull(an, blk), tph))) {
                        tfphase ^= 1u << an;
                        tc::fence_after_sync();
                        tc::tmem_ld32_issue(ra, tlane + (uint32_t)(an * MB * TN));
                        have_a = true;
                    }
                }
                chunk(rb, kc0 + 96);
            }
            if (!ok) break;
            flush();                                       // the piece that the item's end cuts
            if (SHORT && live && !(zsum < tc::kRedoAbove)) {
                reinterpret_cast<unsigned char*>(p.redo + it)[warp - 4] = 1;
                *pp.repair_flag() = 1;
            }
            // the row's statistics over the whole item: its reference and the sum of its pieces
            p.item_m[(size_t)it * p.Rpad + row] = live ? m_ref : 0.f;
            p.item_z[(size_t)it * p.Rpad + row] = live ? zsum : 0.f;
            tiles_before += nt;
        }
        // an abort may leave a requested chunk unread: nothing of tensor memory is in flight past here
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    }

    tc::fence_before_sync();
    __syncthreads();
    tc::stamp(p.clk, 1);
    if (*pp.repair_flag() && !*pp.abort_flag)
        tc::repair_items<D, MB, Cfg::kEpiWarps, Cfg>(smem_raw, &tmQ, &tmK, q_box_rows, k_box_rows, p, tab);
    if (warp == 0) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc(pp.tmem_base, 512);
    }
}

}  // namespace shotkv
