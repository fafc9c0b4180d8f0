// The small reductions that follow the scoring pass.
//
// What the scoring pass leaves per unit (unit = prompt x layer x kv head; an item = one of the
// unit's `nchunk` chunks of keys; a piece = a run of one item's keys inside one segment):
//   part_z [U][P][Rpad]       per (piece, window row) z = sum exp2(x - m) over the piece's keys
//   item_m, item_z [U*nchunk][Rpad]   per (item, row) the reference exponent m all of the item's
//                              pieces share, and the sum of their z -- written by the kernels that
//                              fix one reference per item (score_fast.cuh, score_stream.cuh)
//   part_m [U][P][Rpad]       per (piece, row) reference -- written only by the epilogue of
//                              score_tc.cuh, whose running maximum moves inside an item
//   redo   [U*nchunk]         not 0 for the items that were recomputed with a running maximum
// The piece of segment s (0 = before the first shot, i + 1 = shot i, S + 1 = the question) in item j
// of a unit has index s + j.
// An item is "exact" when every item is (`all_exact`: the kernel of score_tc.cuh did all the work) or when
// its redo flag is set; its rows' statistics are then rebuilt from its pieces.
// A row whose z is not a number in some piece (a query or a key that is none) has the pair (m, z) = (NaN, 0) there: its
// sum over the unit is then no number either, so the row gets weight 0, and its z may still be multiplied by it.
// row_stats_kernel, reduce_select_kernel, shot_score_from_tokens_kernel: fixed-order reductions of
// those partials, and of per-token importances.
#pragma once
#include "common.cuh"
#include "select_compact.cuh"

namespace shotkv {

struct PartialView {
    const float* part_m;      // [U][P][Rpad]
    const float* part_z;      // [U][P][Rpad]
    const float* item_m;      // [U * nchunk][Rpad]
    const float* item_z;      // [U * nchunk][Rpad]
    const unsigned long long* redo;   // [U * nchunk], or NULL
    int nchunk, chunk_keys;   // items of a unit, keys of an item
    int N, S, P, Rpad, all_exact;     // S = -1: the pieces are the items
};

__device__ __forceinline__ bool item_is_exact(const PartialView& v, int item) {
    return v.all_exact || (v.redo && v.redo[item]);
}
// First and last piece of item j of a unit whose prompt has the boundaries o.
__device__ __forceinline__ int first_piece(const PartialView& v, const int* o, int j) {
    return count_le(o, v.S + 1, j * v.chunk_keys) + j;
}
__device__ __forceinline__ int last_piece(const PartialView& v, const int* o, int j) {
    return count_le(o, v.S + 1, min(v.N, (j + 1) * v.chunk_keys) - 1) + j;
}
// (m, z) of two partial sums merged: z relative to the larger reference
__device__ __forceinline__ void merge_mz(float& m, float& z, float mq, float zq) {
    const float mn = fmaxf(m, mq);
    const float mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
    z = z * ex2f(m - mu) + zq * ex2f(mq - mu);
    m = mn;
}
// Row r of unit u over all of its keys: m = max reference, z = sum exp2(x - m).  Items in index
// order, an exact item's pieces in index order: the result does not depend on scheduling.
__device__ __forceinline__ void row_stats_of(const PartialView& v, const int* o, int u, int r, float& m, float& z) {
    m = SHOTKV_NEG_INF;
    z = 0.f;
    for (int j = 0; j < v.nchunk; ++j) {
        const int item = u * v.nchunk + j;
        if (item_is_exact(v, item)) {
            const float* pm = v.part_m + (size_t)u * v.P * v.Rpad + r;
            const float* pz = v.part_z + (size_t)u * v.P * v.Rpad + r;
            for (int q = first_piece(v, o, j), last = last_piece(v, o, j); q <= last; ++q) merge_mz(m, z, pm[(size_t)q * v.Rpad], pz[(size_t)q * v.Rpad]);
        } else {
            merge_mz(m, z, v.item_m[(size_t)item * v.Rpad + r], v.item_z[(size_t)item * v.Rpad + r]);
        }
    }
}

// Per (unit, row) of a scoring pass on plain chunks: m = max over the unit's keys, Z = sum exp2(x - m);
// stores m and 1/Z (0 for padding rows and rows without weight).  The maximum first, then the sum, so
// that the items' loads are in flight together (merged one by one: 4.8 and 6.4 us on 256 and 128 units).
__global__ void row_stats_kernel(const PartialView v, int R, float* __restrict__ row_m, float* __restrict__ row_invz) {
    const int u = blockIdx.x, r = threadIdx.x;                  // one thread per padded row
    grid_release();
    grid_wait();
    bool any = false;
    for (int j = r; j < v.nchunk; j += blockDim.x) any |= item_is_exact(v, u * v.nchunk + j);
    any = __syncthreads_or(any);
    float m = SHOTKV_NEG_INF, z = 0.f;
    if (r < R) {                                                // padding rows carry no weight; their partials may be anything
        if (any) {
            row_stats_of(v, nullptr, u, r, m, z);               // S = -1: the pieces are the items
        } else {
            const float* im = v.item_m + (size_t)u * v.nchunk * v.Rpad + r;
            const float* iz = v.item_z + (size_t)u * v.nchunk * v.Rpad + r;
#pragma unroll 8
            for (int j = 0; j < v.nchunk; ++j) m = fmaxf(m, im[(size_t)j * v.Rpad]);
            const float mu = m == SHOTKV_NEG_INF ? 0.f : m;
#pragma unroll 8
            for (int j = 0; j < v.nchunk; ++j) z += iz[(size_t)j * v.Rpad] * ex2f(im[(size_t)j * v.Rpad] - mu);
        }
    }
    row_m[(size_t)u * v.Rpad + r] = (r < R && m != SHOTKV_NEG_INF) ? m : 0.f;
    row_invz[(size_t)u * v.Rpad + r] = (r < R && z > 0.f) ? 1.f / z : 0.f;
}

// One (b, l): the mass every window row puts on every shot, normalised and summed over the rows and the kv heads,
//   mass[h][i] = sum_r ( sum_{pieces q of shot i} z_q[r] * exp2(m_q[r] - m[r]) ) / Z[r]
//   Score(s_i) = (1/k_i) * sum_h mass[h][i]                             (prefill score equation)
// then the selection.  A cluster of CTAs shares the kv heads of a (b, l), CTA c taking heads c, c + cluster size,
// ...; each leaves its masses in the leader's shared memory and ends, and the leader adds them in a fixed order and
// selects.  In one kernel because the three steps are latency, not work: separate kernels for the masses (one CTA a
// unit, items and pieces one after the other), the sum over heads and the selection took 20 + 2.3 + 5.5 us on one
// layer of 4K and 38 + 2.6 + 8.4 us on 4 x 32 layers of 32K, where reading the partials (115 MB) is 18 us of memory
// time.
//
// Per head: (1) a thread (two, with 128 rows) per row merges the item statistics into the row's (m, 1/Z), four items
// at a time, whose loads are in flight together; the weight exp2(m_item[r] - m[r]) / Z[r], the same for all pieces of
// an item, goes to a table of items and rows. (2) Every warp takes a run of consecutive pieces, its lanes the rows
// four at a time, and weights them from that table (an exact item's pieces carry their own references and pay one
// exp2 per row); the sums over the lanes of the pieces in flight go side by side.  (3) The pieces of each shot are
// added in index order.
// All sums have a fixed order.  What a warp does is wait for its pieces, so it has four in flight.  With 256 rows
// that takes registers of a fourth CTA on the SM: three in flight and four CTAs made 12 layers x 2 heads of 193 shots
// 114.6 us a call, four in flight 109.1; 4 layers x 8 heads of 400 shots 155.6 and 140.8.  Where three CTAs to an SM
// are more than one wave, three in flight are the better (this kernel with 256 shots and 8 heads: 48 layers 49.4 |
// 49.4 us, 56 layers 55.5 | 63.6, 64 layers 55.6 | 61.8, 128 layers 90 | 94.6).  The weights of an item kept in
// registers from piece to piece: 112.7 and 156.4.
constexpr int kReduceThreads = kSelectThreads;
constexpr int kReduceCluster = 8;                  // most CTAs that share the kv heads of a (b, l)

// Shared memory: boundaries; masses of the shots, one row per CTA of the cluster (the leader's copy is
// read); row statistics, the items' weights, piece masses and piece -> item (reused by the selection).
__host__ __device__ constexpr size_t reduce_smem_bytes(int Rpad, int P, int S, int nchunk, int ranks) {
    const size_t pieces = (size_t)(P + 3) / 4 * 4 * 4 + (size_t)(P + 15) / 16 * 16;
    const size_t work = (size_t)(4 + nchunk) * Rpad * 4 + pieces, select = select_smem_bytes(S);
    return bounds_smem_bytes(S) + ranks * ((size_t)(S + 3) / 4 * 4 * 4) + (work > select ? work : select);
}

template <int ROWS, int AHEAD>
__global__ void __launch_bounds__(kReduceThreads, ROWS == 128 || AHEAD < 4 ? 4 : 3)
    reduce_select_kernel(const PartialView v, const __grid_constant__ ShotTable tab, int R, int Hkv, int ranks, float* __restrict__ shot_scores,
                         const SelectArgs a, int* err, long long wait_cycles) {
    constexpr int NW = kReduceThreads / 32, NH = ROWS / 128, PARTS = kReduceThreads / ROWS;
    constexpr int FIRST = 4;                       // items whose statistics a thread has in flight (AHEAD: pieces whose z a warp has)
    constexpr unsigned char kNoItem = 255;
    static_assert(ROWS == 128 || ROWS == 256, "padded window rows");
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int exact[64];
    __shared__ unsigned long long arrived;         // leader: barrier of the other CTAs' masses
    const int S = v.S, np = v.P;
    const int s4 = (S + 3) / 4 * 4;
    int* o = reinterpret_cast<int*>(sm);
    float* masses = reinterpret_cast<float*>(sm + bounds_smem_bytes(S));   // [ranks][s4]
    unsigned char* work = reinterpret_cast<unsigned char*>(masses + (size_t)ranks * s4);
    float* row_m = reinterpret_cast<float*>(work); // [2][ROWS] maxima of the parts; where an item is exact, then [ROWS]
    float* row_w = row_m + 2 * ROWS;               // [2][ROWS] sums of the parts; then [ROWS] 1/Z (0 for rows without weight)
    float* weight = row_w + 2 * ROWS;              // [nchunk][ROWS] 2^(m_item - row's m) / Z
    float* piece_mass = weight + (size_t)v.nchunk * ROWS;   // [P]
    unsigned char* item_of = reinterpret_cast<unsigned char*>(piece_mass + (np + 3) / 4 * 4);   // [P]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bl = blockIdx.x / ranks, rank = blockIdx.x - bl * ranks;   // a cluster is the `ranks` CTAs of one (b, l)
    float* mass = masses + rank * s4;              // of this CTA's heads

    grid_release();
    if (ranks > 1) {
        if (rank == 0 && tid == 0) expect_messages(&arrived, (ranks - 1) * S * (int)sizeof(float));
        cluster_arrive();
    }
    if (tab.ptr) grid_wait();                      // boundaries among the launch parameters are there already
    {   // a segment's pieces are one an item it reaches into; the index after them belongs to none where it ends with an item
        const int* t = table_row(tab, bl / a.L);
#pragma unroll 1
        for (int s = tid; s <= S + 1; s += kReduceThreads) {
            const int lo = s > 0 ? t[s - 1] : 0, hi = s <= S ? t[s] : v.N;
            if (s <= S) o[s] = hi;
            if (lo == hi) continue;                // no token before the first shot
            int j = lo / v.chunk_keys, end = j * v.chunk_keys;
#pragma unroll 1
            do {
                item_of[s + j] = (unsigned char)j;
                ++j;
                end += v.chunk_keys;
            } while (end < hi);
            if (end == hi && s <= S) item_of[s + j] = kNoItem;
        }
    }
    grid_wait();
    const int q_first = table_row(tab, bl / a.L)[0] == 0, q_count = S + v.nchunk + 1 - q_first;

    for (int h = rank; h < Hkv; h += ranks) {
        const int u = bl * Hkv + h;
        // everything the common case needs is asked for at once: the items' flags, the first statistics of
        // this thread's row, and the first pieces of this warp
        const int r = tid % ROWS, part = tid / ROWS;
        const float* im = v.item_m + (size_t)u * v.nchunk * v.Rpad + r;
        const float* iz = v.item_z + (size_t)u * v.nchunk * v.Rpad + r;
        const float* pm = v.part_m + (size_t)u * v.P * v.Rpad;
        const float* pz = v.part_z + (size_t)u * v.P * v.Rpad;
        const int q0 = q_first + q_count * warp / NW, q1 = q_first + q_count * (warp + 1) / NW;
        float m_first[FIRST], z_first[FIRST];
        float4 z4[AHEAD][NH];
        auto load_items = [&](int j0) {
#pragma unroll
            for (int n = 0; n < FIRST; ++n) {
                const int j = j0 + n * PARTS;
                m_first[n] = j < v.nchunk ? im[(size_t)j * v.Rpad] : SHOTKV_NEG_INF;
                z_first[n] = j < v.nchunk ? iz[(size_t)j * v.Rpad] : 0.f;
            }
        };
        load_items(part);
        auto load_pieces = [&](int q) {
#pragma unroll
            for (int n = 0; n < AHEAD; ++n)
                if (q + n < q1)
#pragma unroll
                    for (int k = 0; k < NH; ++k) z4[n][k] = reinterpret_cast<const float4*>(pz + (size_t)(q + n) * v.Rpad)[k * 32 + lane];
        };
        load_pieces(q0);
        bool any = false;
#pragma unroll 1
        for (int j = tid; j < v.nchunk; j += kReduceThreads) {
            const bool e = item_is_exact(v, u * v.nchunk + j);
            exact[j] = e;
            any |= e;
        }
        // (m, z) of this thread's items, as many at a time as its loads ahead
        float m = SHOTKV_NEG_INF, z = 0.f;
#pragma unroll 1
        for (int j0 = part;; ) {
            float bm = SHOTKV_NEG_INF, bz = 0.f;
#pragma unroll
            for (int n = 0; n < FIRST; ++n) bm = fmaxf(bm, m_first[n]);
            const float mu = bm == SHOTKV_NEG_INF ? 0.f : bm;
#pragma unroll
            for (int n = 0; n < FIRST; ++n) bz += z_first[n] * ex2f(m_first[n] - mu);
            merge_mz(m, z, bm, bz);
            j0 += FIRST * PARTS;
            if (j0 >= v.nchunk) break;
            load_items(j0);
        }
        if (PARTS > 1) {
            row_m[part * ROWS + r] = m;
            row_w[part * ROWS + r] = z;
        }
        any = __syncthreads_or(any);
        if (any) {                                 // an item's statistics are those of its pieces
            m = SHOTKV_NEG_INF, z = 0.f;
            if (part == 0) row_stats_of(v, o, u, r, m, z);
            __syncthreads();
            row_m[part * ROWS + r] = m;
            row_w[part * ROWS + r] = z;
            __syncthreads();
        }
        if (PARTS > 1) {
            m = row_m[r];
            z = row_w[r];
            merge_mz(m, z, row_m[ROWS + r], row_w[ROWS + r]);
        }
        const float rm = m == SHOTKV_NEG_INF ? 0.f : m;
        const float rw = (r < R && z > 0.f) ? 1.f / z : 0.f;   // padding rows carry no weight
        // 2^(m_item - row's m) / Z of this row; a row without weight (padding, or nothing but underflow) gets
        // factor 0 whatever its reference
        auto factor = [](float ref, float m, float w) { return w > 0.f ? ex2f(ref - m) * w : 0.f; };
#pragma unroll 4
        for (int j = part; j < v.nchunk; j += PARTS) weight[j * ROWS + r] = factor(im[(size_t)j * v.Rpad], rm, rw);
        if (any) {                                 // for the pieces of exact items (the rows' statistics have been read)
            __syncthreads();
            if (part == 0) {
                row_m[r] = rm;
                row_w[r] = rw;
            }
        }
        __syncthreads();
        // rows 4*lane .. 4*lane+3 (and the same 128 further on when there are 256 rows)
        for (int q = q0; q < q1; q += AHEAD) {
            if (q != q0) load_pieces(q);
            float s[AHEAD];
#pragma unroll
            for (int n = 0; n < AHEAD; ++n) {
                s[n] = 0.f;
                const int j = q + n < q1 ? item_of[q + n] : kNoItem;
                if (j == kNoItem) continue;
                const bool e = any && exact[j] != 0;
#pragma unroll
                for (int k = 0; k < NH; ++k) {
                    float4 f;
                    if (e) {
                        const float4 ref = reinterpret_cast<const float4*>(pm + (size_t)(q + n) * v.Rpad)[k * 32 + lane];
                        const float4 m4 = reinterpret_cast<const float4*>(row_m)[k * 32 + lane];
                        const float4 w4 = reinterpret_cast<const float4*>(row_w)[k * 32 + lane];
                        f = make_float4(factor(ref.x, m4.x, w4.x), factor(ref.y, m4.y, w4.y), factor(ref.z, m4.z, w4.z), factor(ref.w, m4.w, w4.w));
                    } else {
                        f = reinterpret_cast<const float4*>(weight + j * ROWS)[k * 32 + lane];
                    }
                    s[n] = fmaf(z4[n][k].x, f.x, s[n]);
                    s[n] = fmaf(z4[n][k].y, f.y, s[n]);
                    s[n] = fmaf(z4[n][k].z, f.z, s[n]);
                    s[n] = fmaf(z4[n][k].w, f.w, s[n]);
                }
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1)
#pragma unroll
                for (int n = 0; n < AHEAD; ++n) s[n] += __shfl_xor_sync(0xffffffffu, s[n], d);
#pragma unroll
            for (int n = 0; n < AHEAD; ++n)
                if (lane == n && q + n < q1) piece_mass[q + n] = s[n];
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < S; i += kReduceThreads) {
            float s = 0.f;
#pragma unroll 1
            for (int j = o[i] / v.chunk_keys, last = (o[i + 1] - 1) / v.chunk_keys; j <= last; ++j) s += piece_mass[i + 1 + j];
            mass[i] = h == rank ? s : mass[i] + s;
        }
        if (h + ranks < Hkv) __syncthreads();
    }
    bool ok = true;
    if (ranks > 1) {
        cluster_wait();                            // all CTAs have begun
        if (rank != 0) {
#pragma unroll 1
            for (int i = tid; i < S; i += kReduceThreads) send(mass + i, 0, &arrived, mass[i]);
            return;
        }
        ok = await_messages(&arrived, err, wait_cycles);   // if not, the selection is one of whatever masses are there
    }
    float* scores = shot_scores + (size_t)bl * S;
    __syncthreads();                               // the selection takes the place of the work area
    select_body<kReduceThreads>(a, bl, o, work, [&](int i) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < kReduceCluster; ++c)
            if (c < ranks) s += masses[c * s4 + i];
        s /= (float)(o[i + 1] - o[i]);
        scores[i] = s;
        return s;
    });
    if (!ok) outlive_messages(&arrived, nullptr, err, wait_cycles);
}

// Score(s_i) from per-token importance.  Latency-bound while the importances come from L2, so what counts is how
// many loads are in flight, and how many warps where there are many shots.  Eight warps a CTA, in three forms:
//   kHeadsAbreast  short units, thousands of them: a warp a shot, a lane has up to eight heads' loads in flight
//   kTokensAhead   many long units: a warp a shot, head after head, four runs of 32 tokens in flight; few registers, so
//                  that twice the warps of the other forms fit an SM
//   kWholeCta      few long units: a CTA a shot, a warp takes every eighth head, and a lane up to eight tokens of it
// Every lane sums a fixed subset of the shot's (kv head, token) pairs; lanes are added by shuffles and
// warps in order.
enum TokenForm { kHeadsAbreast, kTokensAhead, kWholeCta };
constexpr int kTokenWarps = 8;
constexpr int kLongShot = 96;                  // mean length from which a unit is long
template <TokenForm FORM>
__global__ void __launch_bounds__(32 * kTokenWarps, FORM == kTokensAhead ? 8 : 4)
    shot_score_from_tokens_kernel(const float* imp, const __grid_constant__ ShotTable tab, int L, int Hkv, int N, int S, float* shot_scores) {
    constexpr int AHEAD = FORM == kTokensAhead ? 4 : 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, bl = blockIdx.y;
    const int i = FORM == kWholeCta ? blockIdx.x : blockIdx.x * kTokenWarps + warp;
    grid_release();
    if (i >= S) return;
    grid_wait();
    const int* o = table_row(tab, bl / L);
    const int lo = o[i], hi = o[i + 1];
    const float* base = imp + (size_t)bl * Hkv * N;
    float a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = 0.f;
    if (FORM == kHeadsAbreast) {
        for (int h0 = 0; h0 < Hkv; h0 += AHEAD)
            for (int t = lo + lane; t < hi; t += 32)
#pragma unroll
                for (int k = 0; k < AHEAD; ++k)
                    if (h0 + k < Hkv) a[k] += base[(size_t)(h0 + k) * N + t];
    } else if (FORM == kTokensAhead) {
        for (int h = 0; h < Hkv; ++h) {
            const float* row = base + (size_t)h * N;
            int t = lo + lane;
            for (; t + 32 * (AHEAD - 1) < hi; t += 32 * AHEAD) {
                float v[AHEAD];
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) v[k] = row[t + 32 * k];
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) a[k] += v[k];
            }
            for (; t < hi; t += 32) a[0] += row[t];
        }
    } else {
        for (int h = warp; h < Hkv; h += kTokenWarps)
            for (int t0 = lo; t0 < hi; t0 += 32 * AHEAD)
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) {
                    const int t = t0 + k * 32 + lane;
                    if (t < hi) a[k] += base[(size_t)h * N + t];
                }
    }
    float s = warp_sum(((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7])));
    if (FORM == kWholeCta) {
        __shared__ float part[kTokenWarps];
        if (lane == 0) part[warp] = s;
        __syncthreads();
        s = 0.f;
        for (int w = 0; w < kTokenWarps; ++w) s += part[w];
        if (threadIdx.x == 0) shot_scores[(size_t)bl * S + i] = s / (float)(hi - lo);
    } else if (lane == 0) {
        shot_scores[(size_t)bl * S + i] = s / (float)(hi - lo);
    }
}

}  // namespace shotkv
