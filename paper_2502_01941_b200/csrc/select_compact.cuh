// Whole-shot selection under the token budget and K/V row compaction.
#pragma once
#include "common.cuh"

namespace shotkv {

constexpr int kSelectThreads = 256;

// Exclusive prefix sum over n ints in shared memory, in place; returns the total.  All NT threads
// of the CTA must call it.  Each thread sums a contiguous slice, a warp scans its slices by shuffles
// and every thread adds up the warps before its own (`tmp`: NT / 32 ints).
template <int NT = kSelectThreads>
__device__ __forceinline__ int block_exclusive_scan(int* a, int n, int* tmp) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int per = (n + NT - 1) / NT;
    const int lo = min(tid * per, n), hi = min(lo + per, n);
    int s = 0;
#pragma unroll 1
    for (int i = lo; i < hi; ++i) s += a[i];
    int inc = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += v;
    }
    if (lane == 31) tmp[warp] = inc;
    __syncthreads();
    int run = inc - s, total = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const int v = tmp[w];
        if (w < warp) run += v;
        total += v;
    }
#pragma unroll 1
    for (int i = lo; i < hi; ++i) {
        const int v = a[i];
        a[i] = run;
        run += v;
    }
    __syncthreads();
    return total;
}

// What one (b, l) selects from and where the result goes.
struct SelectArgs {
    int L, N, S, budget_tokens, mode, Mcap;
    uint8_t* keep;       // [B*L][S]
    int* kept_idx;       // [B*L][Mcap]
    int* kept_count;     // [B*L]
};

// Up to this many shots are ranked by counting the better ones, one thread a shot, four scores a
// shared-memory read; beyond it the S^2 comparisons weigh more than a bitonic sort, and the CTA has
// four times the threads.
constexpr int kRankByCount = kSelectThreads, kSortThreads = 1024;

__host__ __device__ constexpr int select_sort_size(int S) {
    int n = 2 * kRankByCount;
    while (n < S) n *= 2;
    return n;
}
// Shared memory of rank_all for n values, and of select_body for S shots, in bytes (multiples of 16).
__host__ __device__ constexpr size_t rank_smem_bytes(int n) {
    return n <= kRankByCount ? (size_t)(n + 3) / 4 * 4 * 4 : (size_t)select_sort_size(n) * 8;
}
__host__ __device__ constexpr size_t select_smem_bytes(int S) {
    return rank_smem_bytes(S) + 2 * ((size_t)(S + 3) / 4 * 4 * 4) + 128;
}

// Sort key of (value descending, index ascending); v is not NaN.
__device__ __forceinline__ unsigned long long rank_key(float v, int i) {
    const unsigned b = __float_as_uint(v + 0.f);                            // -0 and +0 are equal
    const unsigned up = b & 0x80000000u ? ~b : b | 0x80000000u;             // ascending with the value
    return (unsigned long long)~up << 32 | (unsigned)i;
}

// Bitonic sort of n = a power of two >= 64 keys in shared memory, ascending, by the NT threads of a
// CTA.  Exchanges over fewer than 32 places run inside a warp, on registers, so that only the longer
// ones cost a barrier each (1,024 keys: 21 barriers instead of 55).
template <int NT>
__device__ __forceinline__ void block_sort(unsigned long long* key, int n) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto in_warp = [&](int k_from, int k_to) {
        for (int x0 = warp * 32; x0 < n; x0 += NT) {
            const int x = x0 + lane;
            unsigned long long v = key[x];
            for (int k = k_from; k <= k_to; k <<= 1)
                for (int j = min(k >> 1, 16); j > 0; j >>= 1) {
                    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, j);
                    const bool low = (x & j) == 0, up = (x & k) == 0;
                    if ((w < v) == (low == up) && w != v) v = w;      // the lower place of an ascending pair takes the smaller
                }
            key[x] = v;
        }
        __syncthreads();
    };
    in_warp(2, 32);
    for (int k = 64; k <= n; k <<= 1) {
        for (int j = k >> 1; j >= 32; j >>= 1) {
            for (int t = threadIdx.x; t < n / 2; t += NT) {
                const int x = 2 * t - (t & (j - 1)), y = x + j;       // y has bit j, x has not
                const unsigned long long kx = key[x], ky = key[y];
                if ((kx > ky) == ((x & k) == 0)) {
                    key[x] = ky;
                    key[y] = kx;
                }
            }
            __syncthreads();
        }
        in_warp(k, k);
    }
}

// Ranks n values by (value descending, index ascending), NaN last: emit(rank, i) is called once for
// every i, by some thread of the CTA; value(i) is asked for once, by one thread.  NT threads (at least
// n of them where values are ranked by counting), all of which call; `sm` rank_smem_bytes(n) bytes,
// 16-byte aligned.  The caller puts the barrier behind it.
template <int NT, class Value, class Emit>
__device__ __forceinline__ void rank_all(int n, unsigned char* sm, Value&& value, Emit&& emit) {
    const int tid = threadIdx.x;
    if (n <= kRankByCount) {
        float* sc = reinterpret_cast<float*>(sm);
        if (tid < (n + 3) / 4 * 4) {
            const float v = tid < n ? value(tid) : SHOTKV_NEG_INF;
            sc[tid] = v == v ? v : SHOTKV_NEG_INF;     // a NaN ranks last instead of breaking the total order
        }
        __syncthreads();
        if (tid < n) {
            const float v = sc[tid];
            int rank = 0;
#pragma unroll 1
            for (int j = 0; j < n; j += 4) {           // the padding behind the last value never counts: -inf, larger index
                const float4 w = *reinterpret_cast<const float4*>(sc + j);
                rank += (w.x > v) || (w.x == v && j < tid);
                rank += (w.y > v) || (w.y == v && j + 1 < tid);
                rank += (w.z > v) || (w.z == v && j + 2 < tid);
                rank += (w.w > v) || (w.w == v && j + 3 < tid);
            }
            emit(rank, tid);
        }
    } else {
        unsigned long long* key = reinterpret_cast<unsigned long long*>(sm);
        const int ns = select_sort_size(n);
        for (int i = tid; i < ns; i += NT) {
            unsigned long long k = ~0ull;
            if (i < n) {
                const float v = value(i);
                k = rank_key(v == v ? v : SHOTKV_NEG_INF, i);
            }
            key[i] = k;
        }
        __syncthreads();
        block_sort<NT>(key, ns);
        for (int r = tid; r < n; r += NT) emit(r, (int)(unsigned)key[r]);
    }
}

// Ranks the S shots by (score descending, index ascending), keeps whole shots while they fit the
// budget left after the always-kept tokens, and writes the kept token positions in ascending order.
//   mode 0: the longest prefix of the ranking that fits;  mode 1: every shot that still fits.
// Run by a whole CTA of NT threads (at least S of them where shots are ranked by counting); score(i)
// gives shot i's score (each i is asked for once, by one thread); `o` the prompt's boundaries, in
// shared memory; `sm` select_smem_bytes(S) bytes, 16-byte aligned.  What bounds it is latency: every
// step is a handful of barriers and shared-memory round trips, so none of them may be serial in S; and code
// that runs once is fetched once, so loops of a few turns are not unrolled (here and in reduce_select_kernel:
// one small layer of 512 tokens 13.5 -> 12.3 us a call, one layer of a 4K prompt 18.0 -> 16.9 us).
template <int NT, class Score>
__device__ __forceinline__ void select_body(const SelectArgs& a, int bl, const int* o, unsigned char* sm, Score&& score) {
    const int S = a.S, s4 = (S + 3) / 4 * 4, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int* order = reinterpret_cast<int*>(sm + rank_smem_bytes(S));           // rank -> shot
    int* cum = order + s4;                                                  // rank -> length, then scanned
    int* kl = reinterpret_cast<int*>(sm);                                   // shot -> kept length, then destination (once ranked)
    int* tmp = cum + s4;
    const int pre = o[0], qst = o[S];
    const int always = pre + (a.N - qst);
    const int shot_budget = a.budget_tokens - always;

    int kept_shot_tokens;
    if (a.mode == 0 && S <= kRankByCount) {
        // What the better shots take of the budget is added up while they are counted, so
        // neither the ranks nor a scan over them is needed, and the destinations are a scan over registers:
        // three barriers instead of eight (8 shots 2.3 -> 1.7 us).  Four lanes a shot, or two, share the counting
        // where there are threads for it.
        float* sc = reinterpret_cast<float*>(sm);
        int* ln = order;
        if (tid < s4) {
            float v = SHOTKV_NEG_INF;
            int l = 0;
            if (tid < S) {
                v = score(tid);
                v = v == v ? v : SHOTKV_NEG_INF;       // as in rank_all
                l = o[tid + 1] - o[tid];
            }
            sc[tid] = v;
            ln[tid] = l;
        }
        __syncthreads();
        const int sh = S <= NT / 4 ? 2 : S <= NT / 2 ? 1 : 0, i = tid >> sh, share = tid & ((1 << sh) - 1);
        int before = 0, len = 0;
        if (i < S) {
            const float v = sc[i];
            len = ln[i];
#pragma unroll 1
            for (int j = 4 * share; j < S; j += 4 << sh) {
                const float4 w = *reinterpret_cast<const float4*>(sc + j);
                const int4 l = *reinterpret_cast<const int4*>(ln + j);
                before += (w.x > v) || (w.x == v && j < i) ? l.x : 0;
                before += (w.y > v) || (w.y == v && j + 1 < i) ? l.y : 0;
                before += (w.z > v) || (w.z == v && j + 2 < i) ? l.z : 0;
                before += (w.w > v) || (w.w == v && j + 3 < i) ? l.w : 0;
            }
        }
        if (sh > 0) before += __shfl_xor_sync(0xffffffffu, before, 1);
        if (sh > 1) before += __shfl_xor_sync(0xffffffffu, before, 2);
        if (share != 0 || before + len > shot_budget) len = 0;
        if (i < S && share == 0) a.keep[(size_t)bl * S + i] = len > 0;
        int inc = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += x;
        }
        if (lane == 31) tmp[warp] = inc;
        __syncthreads();
        int dst = inc - len;
        kept_shot_tokens = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) {
            const int x = tmp[w];
            if (w < warp) dst += x;
            kept_shot_tokens += x;
        }
        if (i < S && share == 0) kl[i] = dst;
        __syncthreads();
    } else {
        rank_all<NT>(S, sm, score, [&](int rank, int i) {
            order[rank] = i;
            cum[rank] = o[i + 1] - o[i];
        });
        __syncthreads();
        if (a.mode == 0) {
            block_exclusive_scan<NT>(cum, S, tmp);
#pragma unroll 1
            for (int r = tid; r < S; r += NT) {
                const int i = order[r];
                const int len = o[i + 1] - o[i];
                kl[i] = (cum[r] + len <= shot_budget) ? len : 0;
            }
        } else if (warp == 0) {
            // one warp walks the ranking, 32 shots at a time, and hops from one that fits to the next
            int left = shot_budget;
            for (int r0 = 0; r0 < S; r0 += 32) {
                const int r = r0 + lane;
                const int len = r < S ? cum[r] : 0x7fffffff;
                unsigned ahead = 0xffffffffu, kept = 0;                          // shots not passed yet; shots kept
                for (;;) {
                    const unsigned fit = __ballot_sync(0xffffffffu, len <= left) & ahead;
                    if (!fit) break;
                    const int f = __ffs(fit) - 1;
                    kept |= 1u << f;
                    ahead = f == 31 ? 0u : ~0u << (f + 1);
                    left -= __shfl_sync(0xffffffffu, len, f);
                }
                if (r < S) kl[order[r]] = (kept >> lane) & 1u ? len : 0;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < S; i += NT) a.keep[(size_t)bl * S + i] = kl[i] > 0;
        __syncthreads();
        kept_shot_tokens = block_exclusive_scan<NT>(kl, S, tmp);
    }
    const int total = always + kept_shot_tokens;
    int* out = a.kept_idx + (size_t)bl * a.Mcap;
    if (tid == 0) a.kept_count[bl] = total;
#pragma unroll 1
    for (int t = tid; t < pre && t < a.Mcap; t += NT) out[t] = t;
#pragma unroll 1
    for (int i = warp; i < S; i += NT / 32) {
        const int at = kl[i], len = (i + 1 < S ? kl[i + 1] : kept_shot_tokens) - at;   // 0 unless the shot is kept
        const int dst = pre + at, lo = o[i];
#pragma unroll 1
        for (int t = lane; t < len; t += 32)
            if (dst + t < a.Mcap) out[dst + t] = lo + t;
    }
    const int qdst = pre + kept_shot_tokens;
#pragma unroll 1
    for (int t = tid; t < a.N - qst; t += NT)
        if (qdst + t < a.Mcap) out[qdst + t] = qst + t;
#pragma unroll 1
    for (int t = total + tid; t < a.Mcap; t += NT) out[t] = -1;
}

// The boundaries of a prompt, copied to shared memory by the whole CTA (the caller puts the barrier).
__device__ __forceinline__ void copy_bounds(int* to, const ShotTable& tab, int b, int S) {
    const int* o = table_row(tab, b);
#pragma unroll 1
    for (int i = threadIdx.x; i <= S; i += blockDim.x) to[i] = o[i];
}
__host__ __device__ constexpr size_t bounds_smem_bytes(int S) { return (size_t)(S + 4) / 4 * 4 * 4; }

// Selection from scores already in memory: one CTA per (b, l), NT = kSelectThreads where shots are
// ranked by counting, kSortThreads beyond; bounds_smem_bytes(S) + select_smem_bytes(S) of shared memory.
template <int NT>
__global__ void __launch_bounds__(NT) select_shots_kernel(const float* shot_scores, const __grid_constant__ ShotTable tab,
                                                         const SelectArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int bl = blockIdx.x;
    int* o = reinterpret_cast<int*>(sm);
    grid_release();
    grid_wait();
    copy_bounds(o, tab, bl / a.L, a.S);
    __syncthreads();
    const float* scores = shot_scores + (size_t)bl * a.S;
    select_body<NT>(a, bl, o, sm + bounds_smem_bytes(a.S), [&](int i) { return scores[i]; });
}

// Row gather: Kc[u][j] = K[u][kept_idx[bl][j]], same for V.  Rows are D bf16 = D/8 16-byte
// vectors; consecutive lanes move consecutive vectors of a row, each thread keeps four
// independent loads in flight.  grid = (row blocks, Hkv, B*L).
template <int D>
__global__ void __launch_bounds__(256) compact_kv_kernel(const uint4* K, const uint4* V, const int* kept_idx, const int* kept_count,
                                                        int Hkv, int N, int Mcap, uint4* Kc, uint4* Vc) {
    constexpr int VPR = D / 8;                 // 16-byte vectors per row
    constexpr int ROWS = 256 / VPR * 4;        // rows per CTA per pass
    const int bl = blockIdx.z, h = blockIdx.y;
    grid_release();
    grid_wait();
    const int* idx = kept_idx + (size_t)bl * Mcap;
    const int row_in = threadIdx.x / VPR, v = threadIdx.x % VPR;
    // the first pass's indices and the count are asked for together (the index rows hold Mcap entries)
    int src[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = blockIdx.x * ROWS + q * (256 / VPR) + row_in;
        src[q] = j < Mcap ? idx[j] : -1;
    }
    const int count = min(kept_count[bl], Mcap);
    const size_t u = (size_t)bl * Hkv + h;
    const uint4* Ku = K + u * N * VPR;
    const uint4* Vu = V + u * N * VPR;
    uint4* Kcu = Kc + u * Mcap * VPR;
    uint4* Vcu = Vc + u * Mcap * VPR;
    for (int j0 = blockIdx.x * ROWS; j0 < count; j0 += gridDim.x * ROWS) {
        uint4 kk[4], vv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = j0 + q * (256 / VPR) + row_in;
            if (j0 != blockIdx.x * ROWS) src[q] = j < count ? idx[j] : -1;
            if (j >= count || src[q] >= N) src[q] = -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            kk[q] = load_if(Ku + (size_t)src[q] * VPR + v, src[q] >= 0);
            vv[q] = load_if(Vu + (size_t)src[q] * VPR + v, src[q] >= 0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (src[q] >= 0) {
                const int j = j0 + q * (256 / VPR) + row_in;
                Kcu[(size_t)j * VPR + v] = kk[q];
                Vcu[(size_t)j * VPR + v] = vv[q];
            }
    }
}

}  // namespace shotkv
