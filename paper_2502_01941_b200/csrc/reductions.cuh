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

// One (b, l): the mass every window row puts on every shot, normalised and summed over the rows and
// the kv heads,
//   mass[h][i] = sum_r ( sum_{pieces q of shot i} z_q[r] * exp2(m_q[r] - m[r]) ) / Z[r]
//   Score(s_i) = (1/k_i) * sum_h mass[h][i]                             (prefill score equation)
// then the selection.  A cluster of CTAs shares the kv heads of a (b, l), CTA c taking heads c,
// c + cluster size, ...; each leaves its masses in the leader's shared memory and ends, and the leader
// adds them in a fixed order and selects.  In one kernel because the three steps are latency, not work:
// separate kernels for the masses (one CTA a unit, items and pieces one after the other), the sum
// over heads and the selection took 20 + 2.3 + 5.5 us on one layer of 4K and 38 + 2.6 + 8.4 us on
// 4 x 32 layers of 32K, where reading the partials (115 MB) is 18 us of memory time.
//
// Per head: (1) a thread (two, with 128 rows) per row merges the item statistics into the row's
// (m, 1/Z): the maximum first, then the sum, so that the items' loads are all in flight at once.
// (2) Every warp takes a run of consecutive pieces, its lanes the rows four at a time; the weight
// exp2(m_item[r] - m[r]) / Z[r] is the same for all pieces of an item and is formed when the run
// enters the item (an exact item's pieces carry their own references and pay one exp2 per row); one
// shuffle reduction gives the piece's mass.  (3) The pieces of each shot are added in index order.
// All sums have a fixed order.
constexpr int kReduceThreads = kSelectThreads;
constexpr int kReduceCluster = 8;                  // most CTAs that share the kv heads of a (b, l)

// Shared memory: boundaries; masses of the shots, one row per CTA of the cluster (the leader's copy is
// read); row statistics, piece masses and piece -> item (reused by the selection).
__host__ __device__ constexpr size_t reduce_smem_bytes(int Rpad, int P, int S, int ranks) {
    const size_t pieces = (size_t)(P + 3) / 4 * 4 * 4 + (size_t)(P + 15) / 16 * 16;
    const size_t work = (size_t)Rpad * 16 + pieces, select = select_smem_bytes(S);
    return bounds_smem_bytes(S) + ranks * ((size_t)(S + 3) / 4 * 4 * 4) + (work > select ? work : select);
}

template <int ROWS>
__global__ void __launch_bounds__(kReduceThreads, 4) reduce_select_kernel(const PartialView v, const __grid_constant__ ShotTable tab,
                                                                      int R, int Hkv, int ranks,
                                                                      float* __restrict__ shot_scores, const SelectArgs a) {
    constexpr int NW = kReduceThreads / 32, NH = ROWS / 128, PARTS = kReduceThreads / ROWS;
    constexpr int AHEAD = 4 / NH, FIRST = 4;       // pieces whose z a warp has in flight; items whose statistics a thread has
    constexpr unsigned char kNoItem = 255;
    static_assert(ROWS == 128 || ROWS == 256, "padded window rows");
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int2 range[64];                     // first and last piece of every item
    __shared__ int exact[64];
    const int S = v.S, np = v.P;
    const int s4 = (S + 3) / 4 * 4;
    int* o = reinterpret_cast<int*>(sm);
    float* masses = reinterpret_cast<float*>(sm + bounds_smem_bytes(S));   // [ranks][s4]
    unsigned char* work = reinterpret_cast<unsigned char*>(masses + (size_t)ranks * s4);
    float* row_m = reinterpret_cast<float*>(work); // [2][ROWS] maxima of the parts, then [ROWS]
    float* row_w = row_m + 2 * ROWS;               // [2][ROWS] sums of the parts, then [ROWS] 1/Z (0 for rows without weight)
    float* piece_mass = row_w + 2 * ROWS;          // [P]
    unsigned char* item_of = reinterpret_cast<unsigned char*>(piece_mass + (np + 3) / 4 * 4);   // [P]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bl = blockIdx.x / ranks, rank = blockIdx.x - bl * ranks;   // a cluster is the `ranks` CTAs of one (b, l)
    float* mass = masses + rank * s4;              // of this CTA's heads

    grid_release();
    if (tab.ptr) grid_wait();                      // boundaries among the launch parameters are there already
    copy_bounds(o, tab, bl / a.L, S);
    if (ranks > 1) cluster_arrive();               // (1) this CTA has begun: its shared memory may be written to
    __syncthreads();
#pragma unroll 1
    for (int j = tid; j < v.nchunk; j += kReduceThreads) range[j] = make_int2(first_piece(v, o, j), last_piece(v, o, j));
#pragma unroll 1
    for (int i = tid; i < S; i += kReduceThreads) mass[i] = 0.f;
#pragma unroll 1
    for (int q = tid; q < np; q += kReduceThreads) item_of[q] = kNoItem;   // an index no piece has (a boundary on a chunk end)
    __syncthreads();
#pragma unroll 1
    for (int j = warp; j < v.nchunk; j += NW)
#pragma unroll 1
        for (int q = range[j].x + lane; q <= range[j].y; q += 32) item_of[q] = (unsigned char)j;
    grid_wait();
    const int q_first = range[0].x, q_count = range[v.nchunk - 1].y + 1 - q_first;

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
#pragma unroll
        for (int n = 0; n < FIRST; ++n) {
            const int j = part + n * PARTS;
            m_first[n] = j < v.nchunk ? im[(size_t)j * v.Rpad] : SHOTKV_NEG_INF;
            z_first[n] = j < v.nchunk ? iz[(size_t)j * v.Rpad] : 0.f;
        }
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
        any = __syncthreads_or(any);
        {   // row statistics
            float m = SHOTKV_NEG_INF, z = 0.f;
            if (!any) {
#pragma unroll
                for (int n = 0; n < FIRST; ++n) m = fmaxf(m, m_first[n]);
#pragma unroll 4
                for (int j = part + FIRST * PARTS; j < v.nchunk; j += PARTS) m = fmaxf(m, im[(size_t)j * v.Rpad]);
            } else if (part == 0) {
                row_stats_of(v, o, u, r, m, z);
            }
            if (PARTS > 1) {
                row_m[part * ROWS + r] = m;
                __syncthreads();
                m = fmaxf(row_m[r], row_m[ROWS + r]);
            }
            const float mu = m == SHOTKV_NEG_INF ? 0.f : m;
            if (!any) {
#pragma unroll
                for (int n = 0; n < FIRST; ++n) z += z_first[n] * ex2f(m_first[n] - mu);
#pragma unroll 4
                for (int j = part + FIRST * PARTS; j < v.nchunk; j += PARTS) z += iz[(size_t)j * v.Rpad] * ex2f(im[(size_t)j * v.Rpad] - mu);
            }
            if (PARTS > 1) {
                row_w[part * ROWS + r] = z;
                __syncthreads();
                z = row_w[r] + row_w[ROWS + r];
                __syncthreads();
            }
            if (part == 0) {
                row_m[r] = mu;
                row_w[r] = (r < R && z > 0.f) ? 1.f / z : 0.f;   // padding rows carry no weight
            }
        }
        __syncthreads();
        // rows 4*lane .. 4*lane+3 (and the same 128 further on when there are 256 rows)
        float4 rm[NH], rw[NH], f[NH];
#pragma unroll
        for (int k = 0; k < NH; ++k) {
            rm[k] = reinterpret_cast<const float4*>(row_m)[k * 32 + lane];
            rw[k] = reinterpret_cast<const float4*>(row_w)[k * 32 + lane];
        }
        // 2^(m - row's m) / Z of this lane's rows; a row without weight (padding, or nothing but
        // underflow) gets factor 0 whatever its reference
        auto weights = [&](const float* ref) {
#pragma unroll
            for (int k = 0; k < NH; ++k) {
                const float4 mi = reinterpret_cast<const float4*>(ref)[k * 32 + lane];
                f[k].x = rw[k].x > 0.f ? ex2f(mi.x - rm[k].x) * rw[k].x : 0.f;
                f[k].y = rw[k].y > 0.f ? ex2f(mi.y - rm[k].y) * rw[k].y : 0.f;
                f[k].z = rw[k].z > 0.f ? ex2f(mi.z - rm[k].z) * rw[k].z : 0.f;
                f[k].w = rw[k].w > 0.f ? ex2f(mi.w - rm[k].w) * rw[k].w : 0.f;
            }
        };
        int item = kNoItem;
        for (int q = q0; q < q1; q += AHEAD) {
            if (q != q0) load_pieces(q);
#pragma unroll
            for (int n = 0; n < AHEAD; ++n) {
                const int j = q + n < q1 ? item_of[q + n] : kNoItem;
                if (j == kNoItem) continue;
                const bool e = exact[j] != 0;
                if (e || j != item) weights(e ? pm + (size_t)(q + n) * v.Rpad : v.item_m + ((size_t)u * v.nchunk + j) * v.Rpad);
                item = e ? kNoItem : j;
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < NH; ++k) {
                    s = fmaf(z4[n][k].x, f[k].x, s);
                    s = fmaf(z4[n][k].y, f[k].y, s);
                    s = fmaf(z4[n][k].z, f[k].z, s);
                    s = fmaf(z4[n][k].w, f[k].w, s);
                }
                s = warp_sum(s);
                if (lane == 0) piece_mass[q + n] = s;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < S; i += kReduceThreads) {
            float s = 0.f;
#pragma unroll 1
            for (int j = o[i] / v.chunk_keys, last = (o[i + 1] - 1) / v.chunk_keys; j <= last; ++j) s += piece_mass[i + 1 + j];
            mass[i] += s;
        }
        __syncthreads();
    }
    if (ranks > 1) {
        cluster_wait();                            // (1) the leader has begun
        if (rank != 0)
#pragma unroll 1
            for (int i = tid; i < S; i += kReduceThreads) cluster_store(mass + i, 0, mass[i]);
        cluster_arrive();                          // (2) this CTA's masses are with the leader
    }
    if (rank == 0) {
        if (ranks > 1) cluster_wait();             // (2)
        float* scores = shot_scores + (size_t)bl * S;
        select_body<kReduceThreads>(a, bl, o, work, [&](int i) {
            float s = 0.f;
#pragma unroll 1
            for (int c = 0; c < ranks; ++c) s += masses[c * s4 + i];
            s /= (float)(o[i + 1] - o[i]);
            scores[i] = s;
            return s;
        });
    }
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
