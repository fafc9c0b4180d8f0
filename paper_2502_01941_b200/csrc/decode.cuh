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
};

// ---- a unit's keys shared by a cluster -------------------------------------------------------
// A unit (sequence, layer, kv head) whose batch is too small to fill the GPU is shared by a cluster of
// p.nsplit CTAs: blocks of 16 keys go round the warps of all of them.  Every CTA sends its (m, z) per
// query row to all others and each then knows the whole row's maximum and sum.
constexpr int kMaxSplit = 8;

// Every CTA's (m, z) of the 8 query rows (`own`, [8][2], in shared memory behind a barrier) to all
// CTAs' `table` [nsplit][8][2]; returns when all have arrived.  Preceded by a cluster_arrive at the
// start of the kernel (a CTA's memory may be written once it has begun).  What the CTA wrote to its own
// shared memory before may be read by the others afterwards; they must be done before it ends.
__device__ __forceinline__ void exchange_stats(const float* own, float* table, int rank, int nsplit) {
    cluster_wait();
#pragma unroll 1
    for (int i = threadIdx.x; i < 16 * nsplit; i += blockDim.x) cluster_store(table + rank * 16 + (i & 15), i >> 4, own[i & 15]);
    cluster_arrive();
    cluster_wait();
}
// The row's maximum and 1 / sum over the whole cluster.
__device__ __forceinline__ void merge_stats(const float* table, int nsplit, int row, float& m, float& iz) {
    m = SHOTKV_NEG_INF;
    for (int c = 0; c < nsplit; ++c) m = fmaxf(m, table[c * 16 + row * 2]);
    float z = 0.f;
    for (int c = 0; c < nsplit; ++c) z += table[c * 16 + row * 2 + 1] * ex2f(table[c * 16 + row * 2] - m);
    iz = z > 0.f ? 1.f / z : 0.f;
}

// One CTA, or a cluster of p.nsplit, per (sequence, layer, kv head).  Each warp takes 16 keys at a
// time straight from global memory: thread (g, t) of a warp reads 16 contiguous bytes of key rows g
// and g+8 per 32-dim block, which serve as the A fragments of two m16n8k16 MMAs whose B operand is
// the group's (up to 8) query rows held in registers with the same k-index permutation.  The logits
// of the decode entries are parked in shared memory until the softmax statistics over all keys
// (kept prefill keys + decode keys) are known.
// A shared unit leaves few warps to an SM, so each asks for its next block before it computes this one.
// SPLIT = false is the same for whole units, nsplit = 1: with the stride of the loop a constant the
// compiler unrolls it and keeps more loads in flight (8 sequences x 32 layers: 245 us a step against 273).
template <int D, bool SPLIT>
__global__ void __launch_bounds__(256) decode_score_kernel(const DecodeParams p) {
    constexpr int NB = D / 32;     // 32-dim blocks
    constexpr int VPR = D / 8;     // 16-byte vectors per row
    extern __shared__ __align__(16) unsigned char dsm[];
    float* sdec = reinterpret_cast<float*>(dsm);             // [8][Dcap]
    float* sred = sdec + 8 * p.Dcap;                         // [8 warps][8 rows][2]
    float* sfin = sred + 8 * 8 * 2;                          // [8 rows][2]  (m, z) of this CTA, then (m, 1/Z)
    float* stab = sfin + 16;                                 // [nsplit][8 rows][2]  (m, z) of the cluster's CTAs

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int nsplit = SPLIT ? p.nsplit : 1;
    const int u = blockIdx.x / nsplit, rank = blockIdx.x - u * nsplit;
    if (SPLIT) cluster_arrive();
    grid_wait();
    grid_release();
    const int bl = u / p.Hkv, hk = u - bl * p.Hkv;
    const int M = min(p.kept_count[bl], p.Mcap);
    const int n = p.n_old + 1;
    const int Ktot = M + n;
    const uint4* Kc_u = reinterpret_cast<const uint4*>(p.Kc + (size_t)u * p.Mcap * D);
    uint4* Kd_u = reinterpret_cast<uint4*>(p.Kd + (size_t)u * p.Dcap * D);
    uint4* Vd_u = reinterpret_cast<uint4*>(p.Vd + (size_t)u * p.Dcap * D);
    const uint4* knew_u = reinterpret_cast<const uint4*>(p.k_new + (size_t)u * D);
    const uint4* vnew_u = reinterpret_cast<const uint4*>(p.v_new + (size_t)u * D);

    // append the new token's key and value as decode entry n_old
    if (rank != 0) {
    } else if (tid < VPR) Kd_u[(size_t)p.n_old * VPR + tid] = knew_u[tid];
    else if (tid < 2 * VPR) Vd_u[(size_t)p.n_old * VPR + (tid - VPR)] = vnew_u[tid - VPR];

    // query rows of this group as B fragments (row g of the fragment = query head hk*G+g)
    uint4 qf[NB];
    {
        const uint4* qrow = reinterpret_cast<const uint4*>(p.q + ((size_t)bl * p.H + (size_t)hk * p.G + g) * D);
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) qf[kb] = g < p.G ? qrow[kb * 4 + t4] : make_uint4(0, 0, 0, 0);
    }

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
        sred[(warp * 8 + 2 * t4) * 2 + 0] = m0;
        sred[(warp * 8 + 2 * t4) * 2 + 1] = z0;
        sred[(warp * 8 + 2 * t4 + 1) * 2 + 0] = m1;
        sred[(warp * 8 + 2 * t4 + 1) * 2 + 1] = z1;
    }
    __syncthreads();
    if (tid < 8) {
        float m = SHOTKV_NEG_INF;
        for (int w = 0; w < 8; ++w) m = fmaxf(m, sred[(w * 8 + tid) * 2]);
        const float mu = m == SHOTKV_NEG_INF ? 0.f : m;      // a CTA of a cluster may have had no keys
        float z = 0.f;
        for (int w = 0; w < 8; ++w) z += sred[(w * 8 + tid) * 2 + 1] * ex2f(sred[(w * 8 + tid) * 2] - mu);
        sfin[tid * 2] = m;
        sfin[tid * 2 + 1] = SPLIT ? z : (z > 0.f ? 1.f / z : 0.f);
    }
    __syncthreads();
    if (SPLIT) {
        exchange_stats(sfin, stab, rank, nsplit);
        if (tid < 8) merge_stats(stab, nsplit, tid, sfin[tid * 2], sfin[tid * 2 + 1]);
        __syncthreads();
    }
    auto weight = [&](int j) {
        float s = 0.f;
        for (int r = 0; r < p.G; ++r) s += ex2f(sdec[r * p.Dcap + j] - sfin[r * 2]) * sfin[r * 2 + 1];
        p.partial[(size_t)u * p.Dcap + j] = s;
    };
    if (SPLIT) {                                           // the decode entries among this warp's blocks
        const int stride = nsplit * 8 * 16;
        for (int base = first + max(0, (M - 15 - first + stride - 1) / stride) * stride; base < Ktot; base += stride) {
            const int j = base + lane - M;
            if (lane < 16 && j >= 0 && j < n) weight(j);
        }
    } else {
        for (int j = tid; j < n; j += 256) weight(j);
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
    static constexpr int kOBytes = kWarps * 8 * D * 4;            // the warps' outputs for the final merge (reuses the ring)
    static_assert(kOBytes <= kRingBytes, "the merge area must fit into the ring");
};

// The same step with the attention output fused in: o_h = sum_t alpha_{t,h} v_t over the kept
// prefill entries and the decode entries, with the very weights the decoding score sums, so that
// scoring adds no pass over K to a decode step that has to read K and V anyway.
//
// HBM-bound, and what it takes to stay there is bytes in flight: a warp that loads a block's keys
// into registers and then waits for them is idle for the whole (loaded) memory latency, and the
// accumulators of the output leave too few registers for enough such warps.  So nothing is loaded
// into registers from global memory here: key and value rows go global -> shared by cp.async one
// block ahead of their use, into a per-warp ring (measured: two stages with three CTAs on an SM beat three stages with two).
//
// Both products run on the tensor cores, transposed so that the few query rows of a group are the
// narrow N = 8 side.  Per block of 16 keys a warp computes S^T[rows x keys] = Q . K^T with the
// group's query rows as the A operand (held in registers) and the key rows as B fragments (16
// contiguous bytes per lane and 32-dim block; the same k-index permutation on both operands).
// The accumulator fragment of that product -- lane (g, t4) holds row g, keys 2*t4, 2*t4+1,
// 8+2*t4, 9+2*t4 -- is, after the exponential, exactly the B fragment of O^T[dims x rows] =
// V^T . P^T, so the weights never leave their registers; they enter as a bf16 pair (high part plus
// remainder: relative error 2^-17) in two MMAs per 16 dimensions, and ldmatrix.trans turns the
// value rows into the A fragments of V^T.  Online softmax per warp with a running maximum per
// query row (lanes that share g); the warps' (m, z, O) are merged at the end in warp order.
// With few CTAs on an SM what bounds it is the chain of one block in one warp (0.7 us before, 0.5 now): the
// copies of a block that is all prefill rows take their addresses from one pointer and immediate offsets,
// masks and parked logits are left to the blocks that need them, and the first product runs as four chains
// of MMAs.  32 steps of 8 sequences x 32 layers 16.25 -> 15.93 ms, a step of 4 sequences x 1 layer 17.0 -> 15.9 us,
// one unit of 8,000 keys 20.0 -> 15.5 us.
// What follows the blocks runs once and its loops are not unrolled: code that runs once is fetched cold (32 steps
// of one layer 439.2 -> 435.8 us).
template <int D>
__global__ void __launch_bounds__(AttendCfg<D>::kWarps * 32, 3) decode_attend_kernel(const DecodeParams p) {
    using Cfg = AttendCfg<D>;
    constexpr int NB = D / 32;     // 32-dim blocks
    constexpr int VPR = D / 8;     // 16-byte chunks per row
    constexpr int MT = D / 16;     // 16-dim tiles of the output
    constexpr int NW = Cfg::kWarps, NS = Cfg::kStages, NT = NW * 32;
    extern __shared__ __align__(16) unsigned char dsm[];
    float* sdec = reinterpret_cast<float*>(dsm);             // [8][Dcap]
    float* sred = sdec + 8 * p.Dcap;                         // [NW warps][8 rows][2]
    float* sfin = sred + NW * 8 * 2;                         // [8 rows][2]  (m, z) of this CTA, then (m, 1/Z)
    float* stab = sfin + 16;                                 // [kMaxSplit][8 rows][2]  (m, z) of the cluster's CTAs
    unsigned char* ring = reinterpret_cast<unsigned char*>(stab + kMaxSplit * 16);   // [NW][NS][keys | values][16 rows][D bf16]; later [NW][8 rows][D] floats
    float* sO = reinterpret_cast<float*>(ring);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int u = blockIdx.x / p.nsplit, rank = blockIdx.x - u * p.nsplit;
    if (p.nsplit > 1) cluster_arrive();
    grid_wait();
    grid_release();
    const int bl = u / p.Hkv, hk = u - bl * p.Hkv;
    const int kept = p.kept_count[bl];
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
    // the first block is asked for before the kept count is there: rows below Mcap can be read, and where the
    // count turns out to end before them they are fetched again
    const int first = (rank * NW + warp) * 16;
    const bool ahead = first + 16 <= p.Mcap;
    if (ahead) fetch_prefill(first, 0);
    const int M = min(kept, p.Mcap);
    const int n = p.n_old + 1;
    const int Ktot = M + n;
    uint4* Kd_u = reinterpret_cast<uint4*>(p.Kd + (size_t)u * p.Dcap * D);
    uint4* Vd_u = reinterpret_cast<uint4*>(p.Vd + (size_t)u * p.Dcap * D);
    const uint4* knew_u = reinterpret_cast<const uint4*>(p.k_new + (size_t)u * D);
    const uint4* vnew_u = reinterpret_cast<const uint4*>(p.v_new + (size_t)u * D);

    // append the new token's key and value as decode entry n_old
    if (rank != 0) {
    } else if (tid < VPR) Kd_u[(size_t)p.n_old * VPR + tid] = knew_u[tid];
    else if (tid < 2 * VPR) Vd_u[(size_t)p.n_old * VPR + (tid - VPR)] = vnew_u[tid - VPR];

    // query row g of the group as A fragments (rows 8..15 of the 16-row operand are zero)
    uint4 qf[NB];
    {
        const uint4* qrow = reinterpret_cast<const uint4*>(p.q + ((size_t)bl * p.H + (size_t)hk * p.G + g) * D);
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) qf[kb] = g < p.G ? qrow[kb * 4 + t4] : make_uint4(0, 0, 0, 0);
    }

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
    // blocks are requested NS - 1 ahead; one copy group per block, empty past the end, so that
    // "at most NS - 1 groups pending" always means this block's rows have landed
    const int STRIDE = p.nsplit * NW * 16;
    int stage = 0;
    if (ahead && first + 16 > M) {                          // not all prefill rows after all
        cp_async_wait<0>();
        __syncwarp();
    }
    if (!ahead || first + 16 > M) {
        if (first < Ktot) fetch_block(first, 0);
        else cp_async_commit();
    }
#pragma unroll
    for (int k = 1; k < NS - 1; ++k) {
        if (first + k * STRIDE < Ktot) fetch_block(first + k * STRIDE, k);
        else cp_async_commit();
    }
    for (int base = first; base < Ktot; base += STRIDE) {
        __syncwarp();                                       // every lane has read the stage the next copy overwrites
        {
            const int nb = base + (NS - 1) * STRIDE;
            if (nb < Ktot) fetch_block(nb, stage == 0 ? NS - 1 : stage - 1);
            else cp_async_commit();
        }
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
        stage = stage + 1 == NS ? 0 : stage + 1;
    }
    cp_async_wait<0>();
    // row sums over the 4 lanes that share g
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    if (t4 == 0) {
        sred[(warp * 8 + g) * 2 + 0] = m;
        sred[(warp * 8 + g) * 2 + 1] = z;
    }
    __syncthreads();                                        // all warps are done with their rings
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        sO[(warp * 8 + 2 * t4) * D + mt * 16 + g] = O[mt][0];
        sO[(warp * 8 + 2 * t4 + 1) * D + mt * 16 + g] = O[mt][1];
        sO[(warp * 8 + 2 * t4) * D + mt * 16 + 8 + g] = O[mt][2];
        sO[(warp * 8 + 2 * t4 + 1) * D + mt * 16 + 8 + g] = O[mt][3];
    }
    if (tid < 8) {
        float mm = SHOTKV_NEG_INF;
        for (int w = 0; w < NW; ++w) mm = fmaxf(mm, sred[(w * 8 + tid) * 2]);
        const float mu = mm == SHOTKV_NEG_INF ? 0.f : mm;    // a CTA of a cluster may have had no keys
        float zz = 0.f;
        for (int w = 0; w < NW; ++w) zz += sred[(w * 8 + tid) * 2 + 1] * ex2f(sred[(w * 8 + tid) * 2] - mu);
        sfin[tid * 2] = mm;
        sfin[tid * 2 + 1] = p.nsplit > 1 ? zz : (zz > 0.f ? 1.f / zz : 0.f);
    }
    __syncthreads();
    float* out = p.out + ((size_t)bl * p.H + (size_t)hk * p.G) * D;
    // the warps' outputs, relative to the CTA's maximum; alone, the CTA has the rows' whole sums already
#pragma unroll 1
    for (int idx = tid; idx < p.G * D; idx += NT) {
        const int r = idx / D;
        const float mm = sfin[r * 2];
        float o = 0.f;
        for (int w = 0; w < NW; ++w) {
            const float mw = sred[(w * 8 + r) * 2];
            if (mw != SHOTKV_NEG_INF) o += sO[w * 8 * D + idx] * ex2f(mw - mm);
        }
        if (p.nsplit > 1) sO[idx] = o;                       // read above by this thread alone
        else out[idx] = o * sfin[r * 2 + 1];
    }
    if (p.nsplit > 1) {
        __syncthreads();
        exchange_stats(sfin, stab, rank, p.nsplit);          // and all CTAs' outputs may be read
        if (tid < 8) merge_stats(stab, p.nsplit, tid, sfin[tid * 2], sfin[tid * 2 + 1]);
        __syncthreads();
        // each CTA adds up its share of the output elements
#pragma unroll 1
        for (int idx = rank * NT + tid; idx < p.G * D; idx += p.nsplit * NT) {
            const int r = idx / D;
            const float mm = sfin[r * 2];
            const float mu = mm == SHOTKV_NEG_INF ? 0.f : mm;    // a row without a finite logit has no weight anywhere
            float o = 0.f;
            for (int c = 0; c < p.nsplit; ++c) o += cluster_load(sO + idx, c) * ex2f(stab[c * 16 + r * 2] - mu);
            out[idx] = o * sfin[r * 2 + 1];
        }
        cluster_arrive();                                    // done with the others' memory
    }
    // the decode entries among this warp's blocks: their weights summed over the query rows
    for (int base = first + max(0, (M - 15 - first + STRIDE - 1) / STRIDE) * STRIDE; base < Ktot; base += STRIDE) {
        const int j = base + lane - M;
        if (lane < 16 && j >= 0 && j < n) {
            float s = 0.f;
#pragma unroll 1
            for (int r = 0; r < p.G; ++r) s += ex2f(sdec[r * p.Dcap + j] - sfin[r * 2]) * sfin[r * 2 + 1];
            p.partial[(size_t)u * p.Dcap + j] = s;
        }
    }
    if (p.nsplit > 1) cluster_wait();                        // the others are done with this CTA's
}

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
// Shared memory: decode_evict_smem_bytes(n).
__host__ __device__ constexpr size_t decode_evict_smem_bytes(int n) {
    return rank_smem_bytes(n) + 5 * ((size_t)(n + 3) / 4 * 4 * 4) + 128;
}
template <int D>
__global__ void __launch_bounds__(kSelectThreads) decode_evict_kernel(const DecodeFinishParams p) {
    constexpr int NT = kSelectThreads, VPR = D / 8, RPP = NT / VPR, Q = 4;   // 16-byte vectors a row, rows a pass per vector in flight
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int first_gone;
    const int n = p.n, n4 = (n + 3) / 4 * 4;
    float* a = reinterpret_cast<float*>(sm + rank_smem_bytes(n));   // accumulated scores
    int* bs = reinterpret_cast<int*>(a + n4);      // born
    int* kf = bs + n4;                             // kept?
    int* ds = kf + n4;                             // its exclusive scan = destination
    int* kp = ds + n4;                             // destination -> source
    int* tmp = kp + n4;
    const int tid = threadIdx.x;
    const int bl = blockIdx.x / p.ranks, rank = blockIdx.x - bl * p.ranks;
    if (tid == 0) first_gone = n;
    grid_wait();
    grid_release();
#pragma unroll 1
    for (int j = tid; j < n; j += NT) {
        const float v = accumulated(p, bl, j);
        a[j] = v == v ? v : SHOTKV_NEG_INF;        // keep the order total even if a score is NaN
        bs[j] = j < n - 1 ? p.born[(size_t)bl * p.Dcap + j] : p.T_old;
    }
    if (p.ranks > 1) cluster_arrive();
    __syncthreads();
    const float top = __int_as_float(0x7f800000);
    rank_all<NT>(n, sm, [&](int j) { return bs[j] >= p.protect_from ? top : a[j]; },
                 [&](int r, int j) {
                     kf[j] = ds[j] = r < p.k;
                     if (r >= p.k) atomicMin(&first_gone, j);
                 });
    __syncthreads();
    block_exclusive_scan<NT>(ds, n, tmp);
#pragma unroll 1
    for (int j = tid; j < n; j += NT)
        if (kf[j]) kp[ds[j]] = j;
    if (p.ranks > 1) cluster_wait();               // all CTAs have read acc and born
    __syncthreads();
    if (rank == 0)
#pragma unroll 1
        for (int j = tid; j < p.k; j += NT) {
            p.acc[(size_t)bl * p.Dcap + j] = a[kp[j]];
            p.born[(size_t)bl * p.Dcap + j] = bs[kp[j]];
        }
    const int row_in = tid / VPR, vec = tid % VPR;
    for (int h = rank; h < p.Hkv; h += p.ranks) {
        uint4* Ku = reinterpret_cast<uint4*>(p.Kd + ((size_t)bl * p.Hkv + h) * p.Dcap * D);
        uint4* Vu = reinterpret_cast<uint4*>(p.Vd + ((size_t)bl * p.Hkv + h) * p.Dcap * D);
        for (int c = first_gone; c < p.k; c += RPP * Q) {      // the rows before the first evicted entry stay
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

}  // namespace shotkv
