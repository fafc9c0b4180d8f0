// Decode phase: per-step attention-score accumulation over the decode-side entries and
// periodic top-k eviction.
#pragma once
#include "common.cuh"
#include "select_compact.cuh"

namespace shotkv {

struct DecodeParams {
    const __nv_bfloat16* q;       // [B][L][H][d]
    const __nv_bfloat16* k_new;   // [B][L][Hkv][d]
    const __nv_bfloat16* v_new;   // [B][L][Hkv][d]
    const __nv_bfloat16* Kc;      // [U][Mcap][d]
    const int* kept_count;        // [B*L]
    __nv_bfloat16* Kd;            // [U][Dcap][d]
    __nv_bfloat16* Vd;            // [U][Dcap][d]
    float* partial;               // [U][Dcap]
    int H, Hkv, G, Mcap, Dcap, n_old;
    int nsplit;                   // CTAs (a cluster) that share a unit's keys
    float scale_log2;
    const __nv_bfloat16* Vc;      // [U][Mcap][d]   (attention-output variant only)
    float* out;                   // [B][L][H][d]   (attention-output variant only)
    int* err;                     // error word (host-visible); set to 1 when a bounded wait gave up
    long long wait_cycles;        // its limit
};

// The rest of a step for one (b, l): acc[j] += sum over kv heads of the entries' weights (fixed order,
// a new entry starts from 0), and, every so many steps, the eviction: the k entries greatest in (acc
// descending, index ascending) are kept, acc, born and the K and V rows moved up in place.  Entries
// born at or after `protect_from` rank before all others (an option beyond the paper's rule; a value
// above every step number protects nothing).
struct DecodeFinishParams {
    const float* partial;         // [U][Dcap]
    float* acc;                   // [B*L][Dcap]
    int* born;                    // [B*L][Dcap]
    __nv_bfloat16* Kd;            // [U][Dcap][d]
    __nv_bfloat16* Vd;            // [U][Dcap][d]
    int Hkv, Dcap, n, T_old;      // n entries, the new one included
    int k, protect_from;          // entries to keep
    int ranks;                    // CTAs (a cluster) per (b, l), heads rank, rank + ranks, ... each
};
__device__ __forceinline__ float accumulated(const DecodeFinishParams& p, int bl, int j) {
    const float* part = p.partial + (size_t)bl * p.Hkv * p.Dcap + j;
    float s = 0.f;
#pragma unroll 8
    for (int h = 0; h < p.Hkv; ++h) s += part[(size_t)h * p.Dcap];
    return (j == p.n - 1 ? 0.f : p.acc[(size_t)bl * p.Dcap + j]) + s;
}

// A step without eviction.
constexpr int kAccumulateThreads = 128;         // one entry a thread
__global__ void __launch_bounds__(kAccumulateThreads) decode_accumulate_kernel(const DecodeFinishParams p) {
    const int bl = blockIdx.x, j = blockIdx.y * kAccumulateThreads + threadIdx.x;
    grid_wait();
    grid_release();
    if (j < p.n) {
        p.acc[(size_t)bl * p.Dcap + j] = accumulated(p, bl, j);
        if (j == p.n - 1) p.born[(size_t)bl * p.Dcap + j] = p.T_old;
    }
}

// A step with eviction.  Every CTA of the cluster adds up and ranks all entries for itself (a few
// hundred: cheaper than handing the ranking round), so one barrier is all the cluster needs: nobody
// writes acc and born before all have read them.  Then each moves the rows of its heads, as many at a
// time as a thread keeps 16-byte vectors in flight; the source of row j is at or after j, so a pass
// that first loads its rows and then, after a barrier, stores them never overwrites a later source.
// Latency-bound: as three kernels (sum, ranking, rows) the end of a cycle took 2.5 + 4.8 + 2.4 us on one
// small layer and 5 + 6.4 + 39 us on 8 sequences x 32 layers.
// Shared memory: decode_evict_smem_bytes(n).  `value(j)`: entry j's accumulated score.  CTA `rank` of the `ranks` that share the
// (b, l)'s heads; clustered: they are a cluster.  At most NT entries, or more than kRankByCount.
__host__ __device__ constexpr size_t decode_evict_smem_bytes(int n) {
    return rank_smem_bytes(n) + 5 * ((size_t)(n + 3) / 4 * 4 * 4) + 128;
}
template <int D, int NT, class Value>
__device__ __forceinline__ void evict_entries(const DecodeFinishParams& p, int bl, int rank, int ranks, bool clustered,
                                              unsigned char* sm, Value&& value) {
    constexpr int VPR = D / 8, RPP = NT / VPR, Q = 4;   // 16-byte vectors a row, rows a pass per vector in flight
    const int n = p.n, n4 = (n + 3) / 4 * 4;
    float* a = reinterpret_cast<float*>(sm + rank_smem_bytes(n));   // accumulated scores
    int* bs = reinterpret_cast<int*>(a + n4);      // born
    int* kf = bs + n4;                             // kept?
    int* ds = kf + n4;                             // its exclusive scan = destination
    int* kp = ds + n4;                             // destination -> source
    int* tmp = kp + n4;
    int* first_gone = tmp + 31;
    const int tid = threadIdx.x;
    if (tid == 0) *first_gone = n;
#pragma unroll 1
    for (int j = tid; j < n; j += NT) {
        const float v = value(j);
        a[j] = v == v ? v : SHOTKV_NEG_INF;        // keep the order total even if a score is NaN
        bs[j] = j < n - 1 ? p.born[(size_t)bl * p.Dcap + j] : p.T_old;
    }
    if (clustered) cluster_arrive();
    __syncthreads();
    const float top = __int_as_float(0x7f800000);
    rank_all<NT>(n, sm, [&](int j) { return bs[j] >= p.protect_from ? top : a[j]; },
                 [&](int r, int j) {
                     kf[j] = ds[j] = r < p.k;
                     if (r >= p.k) atomicMin(first_gone, j);
                 });
    __syncthreads();
    block_exclusive_scan<NT>(ds, n, tmp);
#pragma unroll 1
    for (int j = tid; j < n; j += NT)
        if (kf[j]) kp[ds[j]] = j;
    if (clustered) cluster_wait();                 // all CTAs have read acc and born
    __syncthreads();
    if (rank == 0)
#pragma unroll 1
        for (int j = tid; j < p.k; j += NT) {
            p.acc[(size_t)bl * p.Dcap + j] = a[kp[j]];
            p.born[(size_t)bl * p.Dcap + j] = bs[kp[j]];
        }
    const int row_in = tid / VPR, vec = tid % VPR;
    for (int h = rank; h < p.Hkv; h += ranks) {
        uint4* Ku = reinterpret_cast<uint4*>(p.Kd + ((size_t)bl * p.Hkv + h) * p.Dcap * D);
        uint4* Vu = reinterpret_cast<uint4*>(p.Vd + ((size_t)bl * p.Hkv + h) * p.Dcap * D);
        for (int c = *first_gone; c < p.k; c += RPP * Q) {      // the rows before the first evicted entry stay
            uint4 kk[Q], vv[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = c + q * RPP + row_in;
                kk[q] = vv[q] = make_uint4(0, 0, 0, 0);
                if (j < p.k) {
                    const size_t at = (size_t)kp[j] * VPR + vec;
                    kk[q] = Ku[at];
                    vv[q] = Vu[at];
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = c + q * RPP + row_in;
                if (j < p.k) {
                    Ku[(size_t)j * VPR + vec] = kk[q];
                    Vu[(size_t)j * VPR + vec] = vv[q];
                }
            }
            __syncthreads();
        }
    }
}
template <int D>
__global__ void __launch_bounds__(kSelectThreads) decode_evict_kernel(const DecodeFinishParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int bl = blockIdx.x / p.ranks, rank = blockIdx.x - bl * p.ranks;
    grid_wait();
    grid_release();
    evict_entries<D, kSelectThreads>(p, bl, rank, p.ranks, p.ranks > 1, sm, [&](int j) { return accumulated(p, bl, j); });
}

// ---- a unit's keys shared by a cluster -------------------------------------------------------
// A unit (sequence, layer, kv head) whose batch is too small to fill the GPU is shared by a cluster of
// p.nsplit CTAs: blocks of 16 keys go round the warps of all of them.  Every CTA sends its (m, z) per
// query row to all others and each then knows the whole row's maximum and sum.
constexpr int kMaxSplit = 16;

// (m, z) of row r over the NW warps' sums in `sred`, [NW][8 rows], and the warps' factors (negative: nothing to add).
template <int NW>
__device__ __forceinline__ float2 row_of_cta(const float2* sred, int r, float (&f)[NW]) {
    float2 w[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) w[i] = sred[i * 8 + r];
    float m = SHOTKV_NEG_INF, z = 0.f;
#pragma unroll
    for (int i = 0; i < NW; ++i) m = fmaxf(m, w[i].x);
    const float mu = m == SHOTKV_NEG_INF ? 0.f : m;        // a CTA of a cluster may have had no keys
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const float e = ex2f(w[i].x - mu);
        z += w[i].y * e;
        f[i] = w[i].x == SHOTKV_NEG_INF ? -1.f : e;
    }
    return make_float2(m, z);
}
// Row lane / 4 over `parts` sums (those of the warps, or of the cluster's CTAs) in `table`, [parts][8 rows]: its maximum m and
// 1 / its sum, the same in the four lanes of the row, of which each takes every fourth.
__device__ __forceinline__ void row_of_unit(const float2* table, int parts, float& m, float& iz) {
    const int lane = threadIdx.x & 31;
    float2 part[kMaxSplit / 4];
    m = SHOTKV_NEG_INF;
#pragma unroll
    for (int i = 0; i < kMaxSplit / 4; ++i) {
        const int c = (lane & 3) + 4 * i;
        part[i] = c < parts ? table[c * 8 + (lane >> 2)] : make_float2(SHOTKV_NEG_INF, 0.f);
        m = fmaxf(m, part[i].x);
    }
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const float mu = m == SHOTKV_NEG_INF ? 0.f : m;        // a row without a finite logit has no weight anywhere
    float z = 0.f;
#pragma unroll
    for (int i = 0; i < kMaxSplit / 4; ++i) z += part[i].y * ex2f(part[i].x - mu);
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    iz = z > 0.f ? 1.f / z : 0.f;
}
// Weights of the decode entries begin + lane, begin + step + lane, ... below `end`, of the lanes below `lanes`, summed over
// the G query rows in order, from their logits in `sdec`, [G or 8][Dcap]; (m, iz) from row_of_unit.  A warp's lanes call
// together.  The rows' logits are read side by side, the last row's in place of those past it, which get no weight: one
// after the other, each behind its row's branch, they made a chain (768 units of 608 keys and 390 entries, d = 64, eight query heads
// to a KV head: 45.7 -> 41 us a step; one unit of 600 keys and 400 entries 5.9 -> 5.6, with eight query heads 6.3 -> 5.9).
template <class Emit>
__device__ __forceinline__ void entry_weights(const float* sdec, int Dcap, int G, float m, float iz, int begin, int end, int step, int lanes,
                                              Emit&& emit) {
    if (begin >= end) return;
    const int lane = threadIdx.x & 31;
    float mr[8], izr[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        mr[r] = __shfl_sync(0xffffffffu, m, r * 4);
        izr[r] = __shfl_sync(0xffffffffu, iz, r * 4);
    }
#pragma unroll 1
    for (int j = begin + lane; j - lane < end; j += step) {
        if (lane >= lanes || j < 0 || j >= end) continue;
        float s = 0.f;
#pragma unroll
        for (int half = 0; half < 8; half += 4) {
            if (half >= G) break;
            float x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) x[r] = sdec[min(half + r, G - 1) * Dcap + j];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float more = fmaf(ex2f(x[r] - mr[half + r]), izr[half + r], s);
                s = half + r < G ? more : s;
            }
        }
        emit(j, s);
    }
}

// ---- a step that ends in the kernel it begins in -----------------------------------------------
// Where all CTAs of a (sequence, layer) fit one cluster, its heads' and their shares', the end of the step needs no kernel of
// its own: every CTA sends the weights of its decode entries to the CTA that adds them up, or to all where the step
// evicts, and goes on as the kernels above do, in the same order of additions.  (One kernel boundary and one launch less: see
// decode_step_impl.)
constexpr int kFusedWeights = 4096;                // most weights, heads x entries, that a CTA is sent
struct FusedEnd {
    float* weights;               // [Hkv][n]  in shared memory
    unsigned long long* arrived;
    unsigned char* scratch;       // decode_evict_smem_bytes(n), where the step evicts
};
__host__ __device__ constexpr size_t fused_end_smem_bytes(int Hkv, int n, bool evicts) {
    return 16 + ((size_t)Hkv * n + 3) / 4 * 16 + (evicts ? decode_evict_smem_bytes(n) : 0);
}
// By one thread, ahead of the cluster_arrive at the start; `c`: this CTA's number in the cluster.
__device__ __forceinline__ FusedEnd fused_end_at(unsigned char* sm, const DecodeFinishParams& f) {
    float* w = reinterpret_cast<float*>(sm + 16);
    return FusedEnd{w, reinterpret_cast<unsigned long long*>(sm), reinterpret_cast<unsigned char*>(w + (f.Hkv * f.n + 3) / 4 * 4)};
}
__device__ __forceinline__ void fused_expect(const FusedEnd& e, const DecodeFinishParams& f, int c) {
    if (f.k < f.n || c == 0) expect_messages(e.arrived, f.Hkv * f.n * (int)sizeof(float));
}
__device__ __forceinline__ void fused_send(const FusedEnd& e, const DecodeFinishParams& f, int hk, int j, float w, int ctas) {
    float* to = e.weights + hk * f.n + j;
    const int receivers = f.k < f.n ? ctas : 1;
#pragma unroll 1
    for (int c = 0; c < receivers; ++c) send(to, c, e.arrived, w);
}
// All threads of all CTAs, once a CTA has sent its weights and made its other outputs.  False: the wait gave up,
// and the end was made with whatever weights are there; every index stays in range, and the state is no longer a valid one anyhow.
template <int D, int NT>
__device__ __forceinline__ bool fused_finish(const FusedEnd& e, const DecodeFinishParams& f, int bl, int c, int ctas,
                                             const DecodeParams& p) {
    const bool evicts = f.k < f.n;
    if (!evicts && c != 0) return true;
    const bool ok = await_messages(e.arrived, p.err, p.wait_cycles);
    const auto value = [&](int j) {
        float s = 0.f;
#pragma unroll 1
        for (int h = 0; h < f.Hkv; ++h) s += e.weights[h * f.n + j];
        return (j == f.n - 1 ? 0.f : f.acc[(size_t)bl * f.Dcap + j]) + s;
    };
    if (evicts) {
        evict_entries<D, NT>(f, bl, c, ctas, true, e.scratch, value);
    } else {
#pragma unroll 1
        for (int j = threadIdx.x; j < f.n; j += NT) {
            f.acc[(size_t)bl * f.Dcap + j] = value(j);
            if (j == f.n - 1) f.born[(size_t)bl * f.Dcap + j] = f.T_old;
        }
    }
    return ok;
}

__host__ __device__ constexpr size_t score_smem_bytes(int Dcap, bool split) {
    return ((size_t)8 * Dcap + 8 * 8 * 2 + (split ? kMaxSplit * 16 + 4 : 0)) * 4;
}

// One CTA, or a cluster of p.nsplit, per (sequence, layer, kv head).  Each warp takes 16 keys at a
// time straight from global memory: thread (g, t) of a warp reads 16 contiguous bytes of key rows g
// and g+8 per 32-dim block, which serve as the A fragments of two m16n8k16 MMAs whose B operand is
// the group's (up to 8) query rows held in registers with the same k-index permutation.  The logits
// of the decode entries are parked in shared memory until the softmax statistics over all keys
// (kept prefill keys + decode keys) are known.
// A shared unit leaves few warps to an SM, so each asks for its next block before it computes this one.
// SPLIT = false is the same for whole units, nsplit = 1: with the stride of the loop a constant it is
// unrolled DEPTH times and more loads are in flight (left to itself the compiler chose 1 to 4 by what stood around the
// loop: 8 sequences x 32 layers 301 to 259 us a step, 1 sequence 56 to 43; two or four deep 255 and 39.5).  Four deep takes
// the registers of a CTA on the SM: three there instead of four with d = 128, four instead of five with d = 64.
// FUSED (with SPLIT): the cluster is all CTAs of a (sequence, layer), and the step ends here.
constexpr int kDeep = 4, kShallow = 2;
template <int D, bool SPLIT, bool FUSED, int DEPTH>
__global__ void __launch_bounds__(256) decode_score_kernel(const DecodeParams p, const DecodeFinishParams f) {
    constexpr int NB = D / 32;     // 32-dim blocks
    constexpr int VPR = D / 8;     // 16-byte vectors per row
    extern __shared__ __align__(128) unsigned char dsm[];
    float* sdec = reinterpret_cast<float*>(dsm);             // [8][Dcap]
    float2* sred = reinterpret_cast<float2*>(sdec + 8 * p.Dcap);   // [8 warps][8 rows]  (m, z)
    float2* stab = sred + 8 * 8;                             // [kMaxSplit][8 rows]  (m, z) of the cluster's CTAs
    // of a cluster: barrier of what they send here
    unsigned long long* arrived = reinterpret_cast<unsigned long long*>(stab + kMaxSplit * 8);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int nsplit = SPLIT ? p.nsplit : 1;
    const int u = blockIdx.x / nsplit, rank = blockIdx.x - u * nsplit;
    const int bl = u / p.Hkv, hk = u - bl * p.Hkv;
    const int first_cta = FUSED ? hk * nsplit : 0, ctas = p.Hkv * nsplit;    // in the cluster: the unit's first; FUSED: all
    FusedEnd end{};
    if (FUSED) end = fused_end_at(dsm + score_smem_bytes(p.Dcap, true), f);
    if (SPLIT) {
        if (tid == 0) {
            expect_messages(arrived, nsplit * 8 * (int)sizeof(float2));
            if (FUSED) fused_expect(end, f, first_cta + rank);
        }
        cluster_arrive();
    }
    grid_wait();
    grid_release();
    const uint4* Kc_u = reinterpret_cast<const uint4*>(p.Kc + (size_t)u * p.Mcap * D);
    uint4* Kd_u = reinterpret_cast<uint4*>(p.Kd + (size_t)u * p.Dcap * D);
    uint4* Vd_u = reinterpret_cast<uint4*>(p.Vd + (size_t)u * p.Dcap * D);
    const uint4* knew_u = reinterpret_cast<const uint4*>(p.k_new + (size_t)u * D);
    const uint4* vnew_u = reinterpret_cast<const uint4*>(p.v_new + (size_t)u * D);
    // the kept count, the queries and the new token's rows are asked for at once
    const int kept = p.kept_count[bl];
    // query rows of this group as B fragments (row g of the fragment = query head hk*G+g)
    uint4 qf[NB];
    {
        const uint4* qrow = reinterpret_cast<const uint4*>(p.q + ((size_t)bl * p.H + (size_t)hk * p.G + g) * D);
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) qf[kb] = g < p.G ? qrow[kb * 4 + t4] : make_uint4(0, 0, 0, 0);
    }
    const bool appends = rank == 0 && tid < 2 * VPR;         // the CTA that appends the new token's rows
    uint4 fresh_row = make_uint4(0, 0, 0, 0);
    if (appends) fresh_row = (tid < VPR ? knew_u + tid : vnew_u + (tid - VPR))[0];
    const int M = min(kept, p.Mcap);
    const int n = p.n_old + 1;
    const int Ktot = M + n;
    if (SPLIT) cluster_wait();                               // all CTAs of the cluster have begun: their memory may be written to
    if (appends)                                             // decode entry n_old
        (tid < VPR ? Kd_u + (size_t)p.n_old * VPR + tid : Vd_u + (size_t)p.n_old * VPR + (tid - VPR))[0] = fresh_row;

    auto row_ptr = [&](int i, bool valid) -> const uint4* {
        if (!valid) return knew_u;                         // any readable row; the result is masked
        if (i < M) return Kc_u + (size_t)i * VPR;
        const int j = i - M;
        return j == p.n_old ? knew_u : Kd_u + (size_t)j * VPR;
    };
    // a block's 16 key rows: this lane's 16-byte pieces of rows base + g and base + 8 + g
    uint4 a_lo[NB], a_hi[NB], n_lo[NB], n_hi[NB];          // this block and, where units are shared, the next
    auto load = [&](int base, uint4 (&lo)[NB], uint4 (&hi)[NB]) {
        const uint4 *pa, *pb;
        if (SPLIT && base + 16 <= M) {                     // all of it kept prefill rows: one run of memory (whole
            pa = Kc_u + (size_t)(base + g) * VPR;          // units: the branch would cost the unrolled loop 2.6 %)
            pb = pa + 8 * VPR;
        } else {
            pa = row_ptr(base + g, base + g < Ktot);
            pb = row_ptr(base + 8 + g, base + 8 + g < Ktot);
        }
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
            lo[kb] = pa[kb * 4 + t4];
            hi[kb] = pb[kb * 4 + t4];
        }
    };
    float m0 = SHOTKV_NEG_INF, m1 = SHOTKV_NEG_INF, z0 = 0.f, z1 = 0.f;   // query rows 2*t4, 2*t4+1
    const int first = (rank * 8 + warp) * 16;
    if (SPLIT && first < Ktot) load(first, n_lo, n_hi);
#pragma unroll DEPTH
    for (int base = first; base < Ktot; base += nsplit * 8 * 16) {
        const int ia = base + g, ib = base + g + 8;
        const bool va = ia < Ktot, vb = ib < Ktot;
        if (SPLIT) {
#pragma unroll
            for (int kb = 0; kb < NB; ++kb) {
                a_lo[kb] = n_lo[kb];
                a_hi[kb] = n_hi[kb];
            }
            if (base + nsplit * 8 * 16 < Ktot) load(base + nsplit * 8 * 16, n_lo, n_hi);
        } else {
            load(base, a_lo, a_hi);
        }
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
            const uint32_t f0[4] = {a_lo[kb].x, a_hi[kb].x, a_lo[kb].y, a_hi[kb].y};
            const uint32_t f1[4] = {a_lo[kb].z, a_hi[kb].z, a_lo[kb].w, a_hi[kb].w};
            mma_bf16_16816(c, f0, qf[kb].x, qf[kb].y);
            mma_bf16_16816(c, f1, qf[kb].z, qf[kb].w);
        }
        const float xa0 = va ? c[0] * p.scale_log2 : SHOTKV_NEG_INF;
        const float xa1 = va ? c[1] * p.scale_log2 : SHOTKV_NEG_INF;
        const float xb0 = vb ? c[2] * p.scale_log2 : SHOTKV_NEG_INF;
        const float xb1 = vb ? c[3] * p.scale_log2 : SHOTKV_NEG_INF;
        if (va && ia >= M) {
            sdec[(2 * t4) * p.Dcap + (ia - M)] = xa0;
            sdec[(2 * t4 + 1) * p.Dcap + (ia - M)] = xa1;
        }
        if (vb && ib >= M) {
            sdec[(2 * t4) * p.Dcap + (ib - M)] = xb0;
            sdec[(2 * t4 + 1) * p.Dcap + (ib - M)] = xb1;
        }
        {
            const float mn = fmaxf(m0, fmaxf(xa0, xb0));
            const float mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
            z0 = z0 * ex2f(m0 - mu) + ex2f(xa0 - mu) + ex2f(xb0 - mu);
            m0 = mn;
        }
        {
            const float mn = fmaxf(m1, fmaxf(xa1, xb1));
            const float mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
            z1 = z1 * ex2f(m1 - mu) + ex2f(xa1 - mu) + ex2f(xb1 - mu);
            m1 = mn;
        }
    }
    // combine the (m, z) pairs of the 8 lanes that share t4, then of the 8 warps
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) {
        const float om0 = __shfl_xor_sync(0xffffffffu, m0, o), oz0 = __shfl_xor_sync(0xffffffffu, z0, o);
        const float om1 = __shfl_xor_sync(0xffffffffu, m1, o), oz1 = __shfl_xor_sync(0xffffffffu, z1, o);
        {
            const float mn = fmaxf(m0, om0), mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
            z0 = z0 * ex2f(m0 - mu) + oz0 * ex2f(om0 - mu);
            m0 = mn;
        }
        {
            const float mn = fmaxf(m1, om1), mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
            z1 = z1 * ex2f(m1 - mu) + oz1 * ex2f(om1 - mu);
            m1 = mn;
        }
    }
    if (g == 0) {
        sred[warp * 8 + 2 * t4] = make_float2(m0, z0);
        sred[warp * 8 + 2 * t4 + 1] = make_float2(m1, z1);
    }
    __syncthreads();
    bool ok = true;
    if (SPLIT) {
        if (tid < 8 * nsplit) {                            // every CTA's rows to every CTA
            float fac[8];
            send(stab + rank * 8 + (tid & 7), first_cta + (tid >> 3), arrived, row_of_cta(sred, tid & 7, fac));
        }
        ok = await_messages(arrived, p.err, p.wait_cycles);
    }
    float rm, riz;                                         // of row lane / 4, over all keys of the unit
    row_of_unit(SPLIT ? stab : sred, SPLIT ? nsplit : 8, rm, riz);
    if (SPLIT) {                                           // the decode entries among this warp's blocks
        const int stride = nsplit * 8 * 16;
        const int begin = first + max(0, (M - 15 - first + stride - 1) / stride) * stride;
        entry_weights(sdec, p.Dcap, p.G, rm, riz, begin - M, n, stride, 16, [&](int j, float s) {
            if (FUSED) fused_send(end, f, hk, j, s, ctas);
            else p.partial[(size_t)u * p.Dcap + j] = s;
        });
        const bool all = !FUSED || fused_finish<D, 256>(end, f, bl, first_cta + rank, ctas, p);
        if (!(ok && all)) outlive_messages(ok ? nullptr : arrived, all ? nullptr : end.arrived, p.err, p.wait_cycles);
    } else {
        // (entry_weights here takes registers of a CTA on the SM: 448 units of 3,276 keys, d = 128, 61.5 -> 83.9 us a step)
        for (int j0 = warp * 32; j0 < n; j0 += 256) {
            const int j = j0 + lane;
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float mr = __shfl_sync(0xffffffffu, rm, r * 4), izr = __shfl_sync(0xffffffffu, riz, r * 4);
                if (j < n && r < p.G) s += ex2f(sdec[r * p.Dcap + j] - mr) * izr;
            }
            if (j < n) p.partial[(size_t)u * p.Dcap + j] = s;
        }
    }
}

// ---- helpers of the fused step ---------------------------------------------------------------
// 16 bytes global -> shared without a register stage; `bytes` = 16 copies, 0 writes zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// Four 8x8 bf16 matrices from shared memory, transposed: register i of lane (g, t4) holds
// elements [2*t4][g] and [2*t4 + 1][g] of the matrix whose row addresses lanes 8i..8i+7 supplied.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// Two floats as a bf16 pair (round to nearest even), low half = a.
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Shared-memory staging of the fused step: every warp owns a ring of kStages stages, a stage
// holding the 16 key rows and the 16 value rows of one block, unpadded, with the 16-byte chunks of a
// row permuted so that the reads are free of bank conflicts: keys (read back as 16 bytes per lane,
// two rows per quarter-warp) with chunk ^ 4*(row & 1), values (read by ldmatrix, eight rows per
// matrix) with chunk ^ (row & 7).
template <int D>
struct AttendCfg {
    static constexpr int kWarps = 4;                              // warps per CTA
    static constexpr int kStages = 2;                             // blocks in the ring: one in use, one in flight (three CTAs fit an SM)
    static constexpr int kRowBytes = D * 2;
    static constexpr int kTileBytes = 16 * kRowBytes;             // 16 rows of keys (or of values)
    static constexpr int kStageBytes = 2 * kTileBytes;
    static constexpr int kRingBytes = kWarps * kStages * kStageBytes;
    static constexpr int kOutPitch = D + 4;                       // floats a row of a warp's outputs
    static_assert(8 * kOutPitch * 4 <= kStages * kStageBytes, "a warp's outputs take the place of its ring");
};

// Dynamic shared memory of the decode kernels for decode regions of Dcap rows, multiples of 16 bytes.
template <int D>
__host__ __device__ constexpr size_t attend_smem_bytes(int G, int Dcap, int nsplit) {
    const size_t shares = nsplit > 1 ? (size_t)nsplit * (16 + (G * D / 4 / nsplit + 1) * 4) : 0;   // (m, z) of 8 rows, and a share of the quads
    return AttendCfg<D>::kRingBytes + 16 + ((size_t)AttendCfg<D>::kWarps * 16 + ((size_t)G * Dcap + 3) / 4 * 4 + shares) * 4;
}

// The same step with the attention output fused in: o_h = sum_t alpha_{t,h} v_t over the kept prefill entries and the
// decode entries, with the very weights the decoding score sums, so that scoring adds no pass over K to a decode step
// that has to read K and V anyway.
//
// HBM-bound, and what it takes to stay there is bytes in flight: a warp that loads a block's keys into registers and
// then waits for them is idle for the whole (loaded) memory latency, and the accumulators of the output leave too few
// registers for enough such warps.  So nothing is loaded into registers from global memory here: key and value rows
// go global -> shared by cp.async one block ahead of their use, into a per-warp ring (measured: two stages with three
// CTAs on an SM beat three stages with two). The ring comes first in shared memory, which is declared so: its rows
// lie on 128-byte boundaries as they do in global memory, or a warp's copy of 512 bytes takes five lines of it and
// part of its sectors from L2 twice (40 % more of them with the ring 16 bytes off a boundary; 8 sequences x 32 layers
// 580 us a step there, 511 at 64 bytes, 495 at 128).
//
// Both products run on the tensor cores, transposed so that the few query rows of a group are the narrow N = 8 side.
// Per block of 16 keys a warp computes S^T[rows x keys] = Q . K^T with the group's query rows as the A operand (held
// in registers) and the key rows as B fragments (16 contiguous bytes per lane and 32-dim block; the same k-index
// permutation on both operands).
// The accumulator fragment of that product -- lane (g, t4) holds row g, keys 2*t4, 2*t4+1, 8+2*t4, 9+2*t4 -- is,
// after the exponential, exactly the B fragment of O^T[dims x rows] = V^T . P^T, so the weights never leave their
// registers; they enter as a bf16 pair (high part plus remainder: relative error 2^-17) in two MMAs per 16
// dimensions, and ldmatrix.trans turns the value rows into the A fragments of V^T.  Online softmax per warp with a
// running maximum per query row (lanes that share g); the warps' (m, z, O) are merged at the end in warp order.
// With few CTAs on an SM what bounds it is the chain of one block in one warp (0.7 us before, 0.5 now): the copies of
// a block that is all prefill rows take their addresses from one pointer and immediate offsets, masks and parked
// logits are left to the blocks that need them, and the first product runs as four chains of MMAs.  32 steps of 8
// sequences x 32 layers 16.25 -> 15.93 ms, a step of 4 sequences x 1 layer 17.0 -> 15.9 us, one unit of 8,000 keys
// 20.0 -> 15.5 us.
// Of a step of few units (13 us: 4 sequences x 1 layer, 3,276 keys) less than half was blocks of keys.  The rest is a
// chain of latencies: everything the first two blocks need is now asked for in one go, each warp's outputs take the
// place of its own ring (no barrier before they are written), every thread merges the rows it needs for itself, and
// the CTAs of a cluster send each other their rows and the quads of output each adds up (12.9 -> 11.1 us; 2 sequences
// 12.2 -> 9.2). FUSED: the cluster is all CTAs of a (sequence, layer), and the step ends here.
template <int D, bool FUSED>
__global__ void __launch_bounds__(AttendCfg<D>::kWarps * 32, 3) decode_attend_kernel(const DecodeParams p, const DecodeFinishParams f) {
    using Cfg = AttendCfg<D>;
    constexpr int NB = D / 32;     // 32-dim blocks
    constexpr int VPR = D / 8;     // 16-byte chunks per row
    constexpr int MT = D / 16;     // 16-dim tiles of the output
    constexpr int NW = Cfg::kWarps, NS = Cfg::kStages, NT = NW * 32;
    extern __shared__ __align__(128) unsigned char dsm[];
    // [NW][NS][keys | values][16 rows][D bf16]; later each warp's outputs [8 rows][PITCH]
    unsigned char* ring = dsm;
    float2* sred = reinterpret_cast<float2*>(ring + Cfg::kRingBytes + 16);   // [NW warps][8 rows]  (m, z)
    float* sdec = reinterpret_cast<float*>(sred + NW * 8);   // [G][Dcap]  logits of the decode entries
    // of a cluster: [nsplit][8 rows] (m, z) of its CTAs, [nsplit][share] their outputs, of which this CTA has its share of the
    // quads, and the barrier of what they send here
    float2* stab = reinterpret_cast<float2*>(sdec + ((p.G * p.Dcap + 3) & ~3));
    float4* sin = reinterpret_cast<float4*>(stab + p.nsplit * 8);
    unsigned long long* arrived = reinterpret_cast<unsigned long long*>(sred) - 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int u = blockIdx.x / p.nsplit, rank = blockIdx.x - u * p.nsplit;
    // The group's output rows are handed round in quads of four elements: quad q is added up by CTA q % nsplit, as its
    // quad number q / nsplit (256 quads and 16 CTAs at most: the product is exact).
    const int quads = p.G * (D / 4), over = 65536 / p.nsplit + 1;
    const int share = (quads * over) >> 16, owned = share + (rank < quads - share * p.nsplit);
    const int bl = u / p.Hkv, hk = u - bl * p.Hkv;
    const int first_cta = FUSED ? hk * p.nsplit : 0, ctas = p.Hkv * p.nsplit;   // in the cluster: the unit's first; FUSED: all
    FusedEnd end{};
    if (FUSED) end = fused_end_at(dsm + attend_smem_bytes<D>(p.G, p.Dcap, p.nsplit), f);
    if (FUSED || p.nsplit > 1) {
        if (tid == 0) {
            if (p.nsplit > 1) expect_messages(arrived, p.nsplit * (8 * (int)sizeof(float2) + owned * (int)sizeof(float4)));
            if (FUSED) fused_expect(end, f, first_cta + rank);
        }
        cluster_arrive();
    }
    grid_wait();
    grid_release();
    uint4* Kd_u = reinterpret_cast<uint4*>(p.Kd + (size_t)u * p.Dcap * D);
    uint4* Vd_u = reinterpret_cast<uint4*>(p.Vd + (size_t)u * p.Dcap * D);
    const uint4* knew_u = reinterpret_cast<const uint4*>(p.k_new + (size_t)u * D);
    const uint4* vnew_u = reinterpret_cast<const uint4*>(p.v_new + (size_t)u * D);
    // what the first block needs is asked for at once: the kept count, the queries, the new token's rows and the block itself
    const int kept = p.kept_count[bl];
    // query row g of the group as A fragments (rows 8..15 of the 16-row operand are zero)
    uint4 qf[NB];
    {
        const uint4* qrow = reinterpret_cast<const uint4*>(p.q + ((size_t)bl * p.H + (size_t)hk * p.G + g) * D);
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) qf[kb] = g < p.G ? qrow[kb * 4 + t4] : make_uint4(0, 0, 0, 0);
    }
    const bool appends = rank == 0 && tid < 2 * VPR;         // the CTA that appends the new token's rows
    uint4 fresh_row = make_uint4(0, 0, 0, 0);
    if (appends) fresh_row = (tid < VPR ? knew_u + tid : vnew_u + (tid - VPR))[0];
    const uint4* Kc_u = reinterpret_cast<const uint4*>(p.Kc + (size_t)u * p.Mcap * D);
    const uint4* Vc_u = reinterpret_cast<const uint4*>(p.Vc + (size_t)u * p.Mcap * D);
    // this warp's ring.  A lane copies chunk (lane % VPR) of rows lane / VPR + k * (32 / VPR) of a block;
    // kdst and vdst are its first copies' offsets in a stage, permuted as above (the row's low bits of later
    // copies enter the values' permutation by exclusive or)
    constexpr int RPI = 32 / VPR;                            // rows per warp-wide copy
    const uint32_t wring = smem_u32(ring) + (uint32_t)(warp * NS * Cfg::kStageBytes);
    const uint32_t kdst = (uint32_t)((lane / VPR) * Cfg::kRowBytes + (((lane % VPR) ^ (((lane / VPR) & 1) << 2)) << 4));
    const uint32_t vdst = (uint32_t)(Cfg::kTileBytes + (lane / VPR) * Cfg::kRowBytes + (((lane % VPR) ^ ((lane / VPR) & 7)) << 4));
    auto fetch_prefill = [&](int base, int stage) {          // 16 prefill rows: one run of memory
        const uint32_t st = wring + (uint32_t)(stage * Cfg::kStageBytes);
        const uint4* ks = Kc_u + (size_t)base * VPR + lane;
        const uint4* vs = Vc_u + (size_t)base * VPR + lane;
#pragma unroll
        for (int k = 0; k < 16 / RPI; ++k) {
            cp_async16(st + kdst + (uint32_t)(k * RPI * Cfg::kRowBytes), ks + k * 32);
            cp_async16(st + (vdst ^ (uint32_t)(((k * RPI) & 7) << 4)) + (uint32_t)(k * RPI * Cfg::kRowBytes), vs + k * 32);
        }
        cp_async_commit();
    };
    // the first blocks are asked for before the kept count is there: rows below Mcap can be read, and where the
    // count turns out to end before them they are fetched again
    const int first = (rank * NW + warp) * 16, STRIDE = p.nsplit * NW * 16;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        if (first + k * STRIDE + 16 <= p.Mcap) fetch_prefill(first + k * STRIDE, k);
        else cp_async_commit();
    }
    const int M = min(kept, p.Mcap);
    const int n = p.n_old + 1;
    const int Ktot = M + n;
    if (FUSED || p.nsplit > 1) cluster_wait();               // all CTAs of the cluster have begun: their memory may be written to
    if (appends)                                             // decode entry n_old
        (tid < VPR ? Kd_u + (size_t)p.n_old * VPR + tid : Vd_u + (size_t)p.n_old * VPR + (tid - VPR))[0] = fresh_row;

    // a block with decode entries in it, or past the end: rows past the end are filled with zeros (a weight of
    // zero must not meet a stray NaN)
    auto fetch_block = [&](int base, int stage) {
        if (base + 16 <= M) {
            fetch_prefill(base, stage);
            return;
        }
        const int c = lane % VPR;
        const uint32_t st = wring + (uint32_t)(stage * Cfg::kStageBytes);
#pragma unroll
        for (int k = 0; k < 16 / RPI; ++k) {
            const int rr = lane / VPR + k * RPI;
            const int i = base + rr;
            const bool valid = i < Ktot;
            const bool fresh = i - M == p.n_old;            // the token appended by this very step
            const uint4* ksrc = i < M ? Kc_u + (size_t)i * VPR : (fresh ? knew_u : Kd_u + (size_t)(i - M) * VPR);
            const uint4* vsrc = i < M ? Vc_u + (size_t)i * VPR : (fresh ? vnew_u : Vd_u + (size_t)(i - M) * VPR);
            cp_async16(st + (uint32_t)(rr * Cfg::kRowBytes + ((c ^ ((rr & 1) << 2)) << 4)), valid ? ksrc + c : knew_u, valid ? 16 : 0);
            cp_async16(st + (uint32_t)(Cfg::kTileBytes + rr * Cfg::kRowBytes + ((c ^ (rr & 7)) << 4)), valid ? vsrc + c : vnew_u, valid ? 16 : 0);
        }
        cp_async_commit();
    };
    // ldmatrix row of this lane: matrix lane/8 = (keys 0-7 | 8-15) x (dims +0 | +8), row lane%8
    const int ldm_row = ((lane >> 4) & 1) * 8 + (lane & 7), ldm_hi = (lane >> 3) & 1;

    float O[MT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) O[mt][q] = 0.f;
    // running maximum of query row g over this warp's keys (the same in the 4 lanes that share g);
    // z: this lane's part of the row sum relative to it
    float m = SHOTKV_NEG_INF, z = 0.f;
    // One copy group per block, empty past the end, so that "at most NS - 1 groups pending" always means this
    // block's rows have landed.  Of the blocks asked for above, those that are not all prefill rows are fetched now.
    bool landed = false;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int base = first + k * STRIDE;
        if (base + 16 > M) {
            if (!landed) {
                cp_async_wait<0>();
                __syncwarp();
                landed = true;
            }
            if (base < Ktot) fetch_block(base, k);
            else cp_async_commit();
        }
    }
    int stage = 0;
    for (int base = first; base < Ktot; base += STRIDE) {
        cp_async_wait<NS - 1>();                            // this block's rows have landed (later blocks' may be in flight)
        __syncwarp();
        const uint32_t st = wring + (uint32_t)(stage * Cfg::kStageBytes);
        // keys base+g and base+8+g as B fragments
        // keys base+0..7 and base+8..15, each in two chains of MMAs so that none is longer than NB
        float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f}, s3[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
            const uint32_t off = (uint32_t)(((kb * 4 + t4) ^ ((g & 1) << 2)) << 4);
            uint4 ka, kb8;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(ka.x), "=r"(ka.y), "=r"(ka.z), "=r"(ka.w) : "r"(st + (uint32_t)(g * Cfg::kRowBytes) + off));
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(kb8.x), "=r"(kb8.y), "=r"(kb8.z), "=r"(kb8.w) : "r"(st + (uint32_t)((g + 8) * Cfg::kRowBytes) + off));
            const uint32_t a0[4] = {qf[kb].x, 0u, qf[kb].y, 0u};
            const uint32_t a1[4] = {qf[kb].z, 0u, qf[kb].w, 0u};
            mma_bf16_16816(s0, a0, ka.x, ka.y);
            mma_bf16_16816(s1, a0, kb8.x, kb8.y);
            mma_bf16_16816(s2, a1, ka.z, ka.w);
            mma_bf16_16816(s3, a1, kb8.z, kb8.w);
        }
        // this lane: row g, keys base + {2*t4, 2*t4+1, 8+2*t4, 9+2*t4}
        const int k0 = base + 2 * t4;
        float x[4] = {(s0[0] + s2[0]) * p.scale_log2, (s0[1] + s2[1]) * p.scale_log2, (s1[0] + s3[0]) * p.scale_log2,
                      (s1[1] + s3[1]) * p.scale_log2};
        if (base + 16 > M) {                                // decode entries, or the end of the keys
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int key = k0 + (q & 1) + (q >> 1) * 8;
                if (key >= Ktot) x[q] = SHOTKV_NEG_INF;
                else if (g < p.G && key >= M) sdec[g * p.Dcap + (key - M)] = x[q];
            }
        }
        float bm = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
        bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
        const float mn = fmaxf(m, bm);
        const float mu = mn == SHOTKV_NEG_INF ? 0.f : mn;
        const float al = ex2f(m - mu);                      // rescale of what was summed so far
        float pw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) pw[q] = ex2f(x[q] - mu);
        z = z * al + (pw[0] + pw[1]) + (pw[2] + pw[3]);
        const bool changed = __any_sync(0xffffffffu, mn != m);
        m = mn;
        if (changed) {
            // the output fragments hold rows 2*t4 and 2*t4+1: their factors live in lanes 8*t4 and 8*t4+4
            const float f0 = __shfl_sync(0xffffffffu, al, 8 * t4), f1 = __shfl_sync(0xffffffffu, al, 8 * t4 + 4);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                O[mt][0] *= f0; O[mt][1] *= f1; O[mt][2] *= f0; O[mt][3] *= f1;
            }
        }
        // weights as B fragments of the second product: high bf16 part and remainder
        const uint32_t h0 = pack_bf16(pw[0], pw[1]), h1 = pack_bf16(pw[2], pw[3]);
        const uint32_t l0 = pack_bf16(pw[0] - __uint_as_float(h0 << 16), pw[1] - __uint_as_float(h0 & 0xffff0000u));
        const uint32_t l1 = pack_bf16(pw[2] - __uint_as_float(h1 << 16), pw[3] - __uint_as_float(h1 & 0xffff0000u));
        const uint32_t vrow = st + (uint32_t)(Cfg::kTileBytes + ldm_row * Cfg::kRowBytes);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            uint32_t a[4];
            ldmatrix_x4_trans(a, vrow + (uint32_t)((((2 * mt + ldm_hi) ^ (ldm_row & 7))) << 4));
            mma_bf16_16816(O[mt], a, h0, h1);
            mma_bf16_16816(O[mt], a, l0, l1);
        }
        __syncwarp();                                       // every lane has read the stage the next copy overwrites
        if (base + NS * STRIDE < Ktot) fetch_block(base + NS * STRIDE, stage);
        else cp_async_commit();
        stage = stage + 1 == NS ? 0 : stage + 1;
    }
    cp_async_wait<0>();
    // row sums over the 4 lanes that share g
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    if (t4 == 0) sred[warp * 8 + g] = make_float2(m, z);
    __syncwarp();                                           // all lanes are done with the warp's ring: its outputs take its place
    constexpr int PITCH = Cfg::kOutPitch, kWarpRing = NS * Cfg::kStageBytes / 4;    // floats
    float* sO = reinterpret_cast<float*>(ring);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        float* o = sO + warp * kWarpRing + 2 * t4 * PITCH + mt * 16 + g;
        o[0] = O[mt][0];
        o[PITCH] = O[mt][1];
        o[8] = O[mt][2];
        o[PITCH + 8] = O[mt][3];
    }
    __syncthreads();
    float* out = p.out + ((size_t)bl * p.H + (size_t)hk * p.G) * D;
    if (p.nsplit > 1 && tid < 8 * p.nsplit) {                // every CTA's rows to every CTA
        float fac[NW];
        send(stab + rank * 8 + (tid & 7), first_cta + (tid >> 3), arrived, row_of_cta(sred, tid & 7, fac));
    }
    // the warps' outputs relative to the CTA's maximum: alone, the CTA has the rows' whole sums
#pragma unroll 1
    for (int q = tid; q < quads; q += NT) {
        const int r = q / (D / 4), c = q % (D / 4) * 4;
        float fac[NW];
        const float2 row = row_of_cta(sred, r, fac);
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float4 v = *reinterpret_cast<const float4*>(sO + w * kWarpRing + r * PITCH + c);
            if (fac[w] >= 0.f) o.x += v.x * fac[w], o.y += v.y * fac[w], o.z += v.z * fac[w], o.w += v.w * fac[w];
        }
        if (p.nsplit > 1) {
            const int slot = (q * over) >> 16, to = q - slot * p.nsplit;
            send(sin + rank * (share + 1) + slot, first_cta + to, arrived, o);
        } else {
            const float iz = row.y > 0.f ? 1.f / row.y : 0.f;
            float* d = out + 4 * q;
            d[0] = o.x * iz;
            d[1] = o.y * iz;
            d[2] = o.z * iz;
            d[3] = o.w * iz;
        }
    }
    const bool ok = p.nsplit <= 1 || await_messages(arrived, p.err, p.wait_cycles);
    float rm, riz;                                           // of row lane / 4, over all keys of the unit
    row_of_unit(p.nsplit > 1 ? stab : sred, p.nsplit > 1 ? p.nsplit : NW, rm, riz);
    const float rmu = rm == SHOTKV_NEG_INF ? 0.f : rm;
    // the CTA's own quads, four lanes each of which adds up every fourth CTA's
    if (p.nsplit > 1) {
#pragma unroll 1
        for (int x = tid; x < (owned * 4 + 31) / 32 * 32; x += NT) {
            const int slot = x >> 2, q = slot * p.nsplit + rank;
            const int r = slot < owned ? q / (D / 4) : 0;
            const float mu = __shfl_sync(0xffffffffu, rmu, r * 4), iz = __shfl_sync(0xffffffffu, riz, r * 4);
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < kMaxSplit / 4; ++i) {
                const int c = t4 + 4 * i;
                if (slot < owned && c < p.nsplit) {
                    const float4 v = sin[c * (share + 1) + slot];
                    const float e = ex2f(stab[c * 8 + r].x - mu);
                    o.x += v.x * e, o.y += v.y * e, o.z += v.z * e, o.w += v.w * e;
                }
            }
#pragma unroll
            for (int d = 1; d <= 2; d <<= 1) {
                o.x += __shfl_xor_sync(0xffffffffu, o.x, d);
                o.y += __shfl_xor_sync(0xffffffffu, o.y, d);
                o.z += __shfl_xor_sync(0xffffffffu, o.z, d);
                o.w += __shfl_xor_sync(0xffffffffu, o.w, d);
            }
            if (slot < owned) out[4 * q + t4] = (t4 == 0 ? o.x : t4 == 1 ? o.y : t4 == 2 ? o.z : o.w) * iz;
        }
    }
    // the decode entries, their weights summed over the query rows: of a shared unit those among this warp's blocks, 16 lanes
    // at a time; whole units have them all here, and a lane each (768 units of 608 keys and 390 decode entries, d = 64: 46.3
    // -> 43.2 us a step, eight query heads to a KV head 50.8 -> 45.7)
    const bool whole = p.nsplit == 1;
    const int begin = whole ? warp * 32 : first + max(0, (M - 15 - first + STRIDE - 1) / STRIDE) * STRIDE - M;
    entry_weights(sdec, p.Dcap, p.G, rm, riz, begin, n, whole ? NT : STRIDE, whole ? 32 : 16, [&](int j, float s) {
        if (FUSED) fused_send(end, f, hk, j, s, ctas);
        else p.partial[(size_t)u * p.Dcap + j] = s;
    });
    const bool all = !FUSED || fused_finish<D, NT>(end, f, bl, first_cta + rank, ctas, p);
    if (!(ok && all)) outlive_messages(ok ? nullptr : arrived, all ? nullptr : end.arrived, p.err, p.wait_cycles);
}

}  // namespace shotkv
