// Shared device helpers for the ShotKV kernels (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace shotkv {

constexpr int kWarp = 32;
constexpr float kLog2e = 1.4426950408889634f;

#define SHOTKV_NEG_INF (__int_as_float(0xff800000))

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// D(16x8,f32) += A(16x16,bf16,row) * B(16x8,bf16,col)
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The shot boundaries off[B][S+1] as kernels get them, a row of `stride` entries per prompt.  For the
// scoring pass three entries of kNoBound follow the S + 1 boundaries of every row, so that it can
// walk along a row one boundary ahead without comparing indices (and a row without boundaries is
// these three alone).  A table of up to kTableArgs entries (three kilobytes: 8 prompts of 92 shots, or
// one of 764) travels in the launch's own parameters; a larger one is copied to the workspace and `ptr` is
// its address.  A copy of a small table costs a host-to-device transfer of 1.5 us and a gap of 2 to
// 5 us on either side of it.
constexpr int kTableArgs = 768;
constexpr int kNoBound = 0x7fffffff;
constexpr int kTableEnd = 3;
struct ShotTable {
    const int* ptr;            // device table, or NULL: the entries are in `data`
    int stride;
    int data[kTableArgs];
};
// Boundaries of prompt b.
__device__ __forceinline__ const int* table_row(const ShotTable& t, int b) {
    return (t.ptr ? t.ptr : t.data) + (size_t)b * t.stride;
}
// Number of the n ascending entries o[0..n) that are <= x.
__device__ __forceinline__ int count_le(const int* o, int n, int x) {
    int lo = 0;
    while (lo < n) {
        const int mid = (lo + n) >> 1;
        if (o[mid] <= x) lo = mid + 1; else n = mid;
    }
    return lo;
}
// The same by a whole warp, 32 probes a round: at most three rounds for 8,193 entries.
__device__ __forceinline__ int count_le_warp(const int* o, int n, int x) {
    const int lane = threadIdx.x & 31;
    int lo = 0;
    while (n > 0) {
        const int step = (n + 31) >> 5;
        const int first = lane * step;
        const bool le = first < n && o[lo + min(first + step, n) - 1] <= x;
        const int skip = min(__popc(__ballot_sync(0xffffffffu, le)) * step, n);   // whole blocks that are <= x
        lo += skip;
        n = min(step, n - skip) - 1;                                                // the next block's last entry is > x
    }
    return lo;
}

// Programmatic dependent launch: a kernel launched with that attribute may begin while the one before
// it on the stream still runs.  Every such kernel passes grid_wait before it touches global memory:
// it returns when the kernel before has finished and its writes are visible (and, that kernel having
// waited too, everything before it).  grid_release lets the next kernel's CTAs begin, once all CTAs of
// this one have called it or ended.  What such a kernel reads may still be written when it begins, so no
// pointer it reads through is __restrict__ and no load takes the read-only path: either would let the compiler
// move a load above the wait.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// 16 bytes at p, or zeros.  Written as one predicated instruction: a branch around each plain load of a row kept
// the next one waiting behind it.
__device__ __forceinline__ uint4 load_if(const uint4* p, bool valid) {
    uint4 v = make_uint4(0, 0, 0, 0);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t@q ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
                 : "l"(p), "r"((int)valid));
    return v;
}

// Barrier of a thread-block cluster in two halves, for all threads of its CTAs.
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared memory of CTA `rank` of the cluster: `p` is the address of the same variable in this CTA.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}

// What the CTAs of a cluster tell one another goes as messages: a store counts its bytes on the receiver's barrier,
// which is complete when as many as the receiver expects are there.  That is one way across the cluster, where a
// barrier of all its threads is two (1.7 us of a step of 4 sequences x 1 layer).  expect_messages: by one thread,
// ahead of the cluster_arrive at the start; nobody sends before a cluster_wait (a CTA's memory may be written once it
// has begun), and a CTA that has been sent everything may end.
__device__ __forceinline__ void expect_messages(unsigned long long* bar, int bytes) {
    const uint32_t b = smem_u32(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ void send(float* to, int rank, unsigned long long* bar, float v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(cluster_addr(to, rank)), "f"(v),
                 "r"(cluster_addr(bar, rank))
                 : "memory");
}
__device__ __forceinline__ void send(float2* to, int rank, unsigned long long* bar, float2 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(cluster_addr(to, rank)),
                 "f"(v.x), "f"(v.y), "r"(cluster_addr(bar, rank))
                 : "memory");
}
__device__ __forceinline__ void send(float4* to, int rank, unsigned long long* bar, float4 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(cluster_addr(to, rank)),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(cluster_addr(bar, rank))
                 : "memory");
}
// Waits, `limit` cycles at most, until all bytes expected are there.  False: it gave up and has set the error word; what it
// waited for may still come, so the thread passes outlive_messages before it ends.
__device__ __forceinline__ bool await_messages(unsigned long long* bar, int* err, long long limit) {
    const uint32_t b = smem_u32(bar);
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}"
            : "=r"(done)
            : "r"(b)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > limit) {
            atomicExch(err, 1);
            return false;
        }
    }
}
// For single threads whose wait gave up, at their end: keeps their CTA, whose memory the others write to, until all
// other threads of the cluster have ended or are here too (every wait of theirs ends), and until what they sent has
// landed, if it does within the limit.  `bar`, `more`: the barriers waited for in vain, or NULL.
__device__ __forceinline__ void outlive_messages(unsigned long long* bar, unsigned long long* more, int* err, long long limit) {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (bar) await_messages(bar, err, limit);
    if (more) await_messages(more, err, limit);
}

// Self-test of that, for the host to run on demand: a cluster of two CTAs of one warp.  The first expects two words;
// the second sends one at once and the other well after the limit, when the first has given up.  Lane 0 of the first
// waits on behalf of its warp, as a thread of a cluster's CTA does.  report[0..1] = {that wait succeeded, the late
// word was there before the CTA ended}.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(32) message_wait_selftest_kernel(long long limit, int* err, int* report) {
    __shared__ __align__(8) unsigned long long arrived;
    __shared__ float words[2];
    const int lane = threadIdx.x;
    if (lane == 0) {
        words[0] = words[1] = 0.f;
        if (blockIdx.x == 0) expect_messages(&arrived, 2 * (int)sizeof(float));
    }
    cluster_arrive();
    cluster_wait();
    if (lane != 0) return;
    if (blockIdx.x != 0) {
        send(words, 0, &arrived, 1.f);
        for (const long long t0 = clock64(); clock64() - t0 < 4 * limit + 1000000;) __nanosleep(100);
        send(words + 1, 0, &arrived, 2.f);
        return;
    }
    const bool ok = await_messages(&arrived, err, limit);
    report[0] = ok;
    if (!ok) outlive_messages(&arrived, nullptr, err, limit);
    report[1] = *(volatile float*)&words[0] == 1.f && *(volatile float*)&words[1] == 2.f;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
}  // namespace shotkv
