// Pieces shared by the split-KV decode-attention kernels (bf16 cache and int8 cache): the tiling
// constants, the work-item table every CTA builds from the sequence lengths, and the named barrier
// of the consumer warps.
#pragma once
#include "common.cuh"

namespace prsv {

constexpr int kTileKeys = 64;
constexpr int kConsumerWarps = 4;
constexpr int kAttnThreads = (kConsumerWarps + 1) * 32;
constexpr int kMaxStreams = 2048;                      // (sequence, kv head) pairs per launch

__device__ __forceinline__ void consumer_barrier()
{
    asm volatile("bar.sync 1, %0;" ::"n"(kConsumerWarps * 32) : "memory");
}

__device__ __forceinline__ int tiles_of(int ctx) { return (ctx + 1 + kTileKeys - 1) / kTileKeys; }

// (Loops that run a few times per kernel or item are kept rolled: unrolled by default they were 6 KB of each attention
// kernel's 33-48, and what a layer's kernels execute competes for the instruction caches.  Not the loops over the streams,
// here and in the merge kernel, up to 64 dependent rounds: rolled, three layers of hidden 4096 with 16 kv heads at
// batch 128 and 40 tokens took 286.3 us instead of 268.2, at batch 64 185.1 instead of 176.6, 8 kv heads at batch 64 and 200 tokens 200.0
// instead of 194.1; int8 cache 314.1 / 295.8, 232.7 / 225.1 and 198.4 / 194.2; up to 128 streams the same.)

// First item index of every stream, computed identically by every CTA: the lengths are
// fetched by all threads at once (one memory round trip), then warp 0 scans them.
template <typename Params>
__device__ __forceinline__ void build_item_table(const Params &p, int *item_base)
{
    const int streams = p.B * p.nkv;
#pragma unroll 4
    for (int i = threadIdx.x; i < streams; i += blockDim.x) {
        const int nt = tiles_of(p.ctx_len[i / p.nkv]);
        item_base[i + 1] = (nt + p.tiles_per_item - 1) / p.tiles_per_item;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int carry = 0;
#pragma unroll 4
        for (int base = 0; base < streams; base += 32) {
            const int i = base + threadIdx.x;
            int v = i < streams ? item_base[i + 1] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, v, o);
                if ((int)threadIdx.x >= o)
                    v += n;
            }
            if (i < streams)
                item_base[i + 1] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
        if (threadIdx.x == 0)
            item_base[0] = 0;
    }
}

__device__ __forceinline__ int find_stream(const int *item_base, int streams, int item)
{
    int lo = 0, hi = streams;     // item_base[lo] <= item < item_base[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (item_base[mid] <= item) lo = mid; else hi = mid;
    }
    return lo;
}

// ---- Short caches: one cluster per (sequence, kv head) instead of work items and a merge kernel.  Rank r of
// the cluster takes the r-th of `cl` equal runs of the sequence's tiles; the ranks' partials meet by one-sided
// stores (rank q finishes elements [q L, (q + 1) L) of the group's G x 128 outputs, L = G * 128 / cl), and the
// result leaves the kernel merged.
constexpr int kMaxAttnCluster = 8;
constexpr int kMaxClusterGroup = 8;
struct ClusterRecv {
    float o[kMaxClusterGroup * 128];                          // [source rank][L]
    float ml[kMaxAttnCluster * kMaxClusterGroup][2];          // [source rank][head]
    uint64_t bar;
    int gave_up;
};
// (by one thread, before the CTA's barrier; `more` bytes are expected that nobody sends: a test hook)
__device__ __forceinline__ void cluster_recv_init(ClusterRecv &rc, int G, int cl, uint32_t more)
{
    mbar_init(&rc.bar, 1);
    mbar_fence_init();
    mbar_expect_tx(&rc.bar, (uint32_t)(G * 128 * 4 + cl * G * 8) + more);
    rc.gave_up = 0;
}
// balanced runs, the longer ones first (rank 0 is never empty)
__device__ __forceinline__ int cluster_first_tile(int nt, int rank, int cl) { return (nt * rank + cl - 1) / cl; }
// head dims 2 * d2, 2 * d2 + 1 of head r, relative to this rank's maximum M with weight sum l
__device__ __forceinline__ void cluster_send(ClusterRecv &rc, int G, int cl, int rank, int r, int d2, float2 acc, float M, float l)
{
    const int L = G * 128 / cl, e = r * 128 + 2 * d2, q = e / L;
    st_async_v2(cluster_map(&rc.o[rank * L + e - q * L], q), acc, cluster_map(&rc.bar, q));
    if (d2 < cl)
        st_async_v2(cluster_map(rc.ml[rank * G + r], d2), make_float2(M, l), cluster_map(&rc.bar, d2));
}
// Waits for every rank's share of this rank's elements, adds them in rank order and hands each finished pair to
// store(head, first dim, value, value).  Called by all consumer threads (tid < 128).  In the timeline this part is the
// merge: the attention's slots end where it begins.
template <typename Store>
__device__ __forceinline__ void cluster_finish(ClusterRecv &rc, int G, int cl, int rank, int tid, int *status, long long *trace, Store store)
{
    long long *tr = trace ? trace + kTraceSlots : nullptr;
    trace_end(trace);
    trace_start(tr);
    if (!mbar_wait(&rc.bar, 0, status, ST_TIMEOUT_FULL)) {
        *reinterpret_cast<volatile int *>(&rc.gave_up) = 1;
        trace_waited(tr);
    } else {
        trace_waited(tr);
        const int L = G * 128 / cl;
#pragma unroll 1
        for (int i = 2 * tid; i < L; i += 2 * kConsumerWarps * 32) {
            const int e = rank * L + i, r = e >> 7;
            float M = -INFINITY;
#pragma unroll 4
            for (int c = 0; c < cl; ++c)
                M = fmaxf(M, rc.ml[c * G + r][0]);
            float2 acc = make_float2(0.f, 0.f);
            float l = 0.f;
#pragma unroll 4
            for (int c = 0; c < cl; ++c) {                    // rank order
                const float mc = rc.ml[c * G + r][0];
                const float w = mc == -INFINITY ? 0.f : exp2f(mc - M);
                const float2 v = *reinterpret_cast<const float2 *>(&rc.o[c * L + i]);
                acc.x += v.x * w;
                acc.y += v.y * w;
                l += rc.ml[c * G + r][1] * w;
            }
            store(r, e & 127, acc.x / l, acc.y / l);
        }
    }
    // A CTA that gave up may be about to leave before every peer has stored into it, and a store into the shared
    // memory of a CTA that has exited is a fault: it stays until every peer has left or reached this point
    // too, then gives the stores in flight a bounded time to land.  (The barrier counts only threads that have
    // not exited; a CTA that received everything simply leaves.)
    consumer_barrier();
    if (*reinterpret_cast<volatile int *>(&rc.gave_up)) {
        cluster_arrive_relaxed();
        cluster_wait();
        if (tid == 0)
            mbar_wait(&rc.bar, 0, status, ST_TIMEOUT_FULL);
        consumer_barrier();
    }
    trace_end(tr);
}
// The overflow report of the item form: device lengths that need more items than the plan has room for are
// reported although this form has no buffer they could overrun.  (One warp of one CTA.)
__device__ __forceinline__ void cluster_check_items(const int *ctx_len, int B, int nkv, int tiles_per_item, int max_items, int *status)
{
    int n = 0;
#pragma unroll 1
    for (int b = threadIdx.x & 31; b < B; b += 32)
        n += nkv * ((tiles_of(ctx_len[b]) + tiles_per_item - 1) / tiles_per_item);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        n += __shfl_xor_sync(0xffffffffu, n, o);
    if (n > max_items && (threadIdx.x & 31) == 0)
        atomicCAS(status, ST_OK, ST_ITEMS_OVERFLOW);
}

}  // namespace prsv
