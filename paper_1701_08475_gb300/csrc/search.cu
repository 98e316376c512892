// search.cu -- the enhanced hill-climbing search over a kNN graph (Sec. 3.2,
// Alg. 2) for a batch of queries.
//
// The rank list R matters only through its first ks entries by (d, id): they
// are what each iteration expands and what the search returns, and an entry
// outside them never re-enters them (R only grows).  So a query keeps those
// ks keys (ks <= 32, entry e in lane e).  An entry's neighbours are all
// visited once it has been expanded, so each entry is expanded once (a flag in
// its key), and the search ends when every entry is: later iterations could
// add nothing.
//
// An iteration collects the unvisited neighbours of its entries in a queue and
// computes their canonical FP32 distances 32 at a time: cp.async brings the
// rows' next 128 dims into shared memory, every lane's pieces in flight at
// once, and then each lane walks one row.  (A lane that walks its row in
// global memory waits for a few 16-byte pieces at a time.)  The distances
// merge into the list in any order: a key enters at most once and the
// collected ids do not depend on the order.
//
// Visited ids are kept in a shared-memory hash table.  It is exact until it is
// three quarters full; from then on it is a cache: an id is looked for in eight
// slots, and takes the place of another there when it is new.  So an id may be
// visited again, which the merge drops when it is in the list, and which cannot
// enter the list when it was turned away before (the ks-th key only falls).  The
// ids met again are mostly recent ones: with the table frozen when it was full,
// every later id went through long probes and was visited anew each time
// (300,000 x 128, k = 20, ks = 32, 1,000 queries 0.85 ms, 0.46 so; 40,000 x 48,
// k = 64, 305 queries 6.3 and 0.91; one query per warp with exact tables of twice
// the visits in global memory 1.1).
//
// One CTA per query: one warp, or, for few queries, kSearchGroup warps, which
// share the collecting and take a batch of rows each.  Rows of at least
// kSearchWide dims are staged 128 dims at a time with one warp too (fewer round
// trips to memory; the query then comes with each stage): 20,000 x 960, k = 16,
// ks = 32, 305 queries 1.95 -> 1.25 ms, 10,000 queries 6.10 -> 5.88; at 512 dims
// 10,000 queries 3.67 -> 3.88, at 256 2.21 -> 2.70.
//
// Measured (GB300), 1M x 128 integers, k = 20, 10,000 queries, t0 = 12, ks = 20:
// the call took 2.54 ms with a lane per row in global memory, the visited
// tables in global memory and every entry expanded in every iteration; 1.57
// with entries expanded once, staged rows and shared tables (128 dims, two
// queries per CTA: 10 warps per SM), 0.97 with one query per CTA and 32 dims,
// 0.86 with far rows dropped, 0.80 with a warp's ids queued by one atomic.  What
// is left is issue slots and latency about equally.  One query, 100,000 x 96: the
// kernel 115 -> 28 us.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace knng {

namespace {

constexpr int kSearchGroup = 4;  // warps of a query when there are few
// floats per staged row: the 16-byte reads of 8 lanes cover all banks
__host__ __device__ constexpr int search_stride(int dims) { return dims + 4; }
// slots of the visited table (log2): one warp's is small, so that many queries
// fit an SM; all layouts are compile-time constants (table sizes chosen at run
// time cost 30 % of the bulk search)
__host__ __device__ constexpr int search_tab(int W) { return W > 1 ? 12 : 10; }
constexpr int kSearchNear = 8;     // slots that a full table is asked for an id
constexpr int kSearchQueue = 256;
constexpr int kSearchWide = 640;

__host__ __device__ constexpr bool search_by_stage(int W, int dims) { return W == 1 && dims > 32; }

struct SearchSmem {
    size_t stage, tab, queue, keys, entry, misc, total;
};
__host__ __device__ inline SearchSmem search_smem(int D, int W, int dims) {
    SearchSmem L;
    // the query first; with one warp and wide stages, the dims of one stage
    L.stage = ((size_t)(search_by_stage(W, dims) ? dims : D) * 4 + 15) & ~(size_t)15;
    L.tab = L.stage + (size_t)W * 32 * search_stride(dims) * 4;
    L.queue = L.tab + ((size_t)4 << search_tab(W));
    L.keys = L.queue + kSearchQueue * 4;
    L.entry = L.keys + (size_t)W * 32 * 8;
    L.misc = L.entry + 32 * 4;
    L.total = L.misc + 16;
    return L;
}

// A list key: order-preserving distance, then id, then whether the entry has
// been expanded (ids are below 2^31).
__device__ __forceinline__ uint64_t list_key(float d, uint32_t id) {
    return ((uint64_t)ord32(d) << 32) | ((uint64_t)id << 1);
}
__device__ __forceinline__ uint32_t list_id(uint64_t k) { return (uint32_t)k >> 1; }

// W: warps of the CTA; DIMS: dims staged at once.
template <bool VEC, int W, int DIMS>
__global__ void __launch_bounds__(32 * W) k8_search(
    const float* __restrict__ X, int64_t n, int D, const int32_t* __restrict__ G, int k, const float* __restrict__ Q,
    const int32_t* __restrict__ S, int s, int t0, int ks, int32_t* __restrict__ out_ids,
    float* __restrict__ out_d) {
    constexpr int kDims = DIMS, kStride = search_stride(DIMS);
    constexpr int tab_log2 = search_tab(W), full = 3 << (tab_log2 - 2);
    constexpr uint32_t mask = (1u << tab_log2) - 1u;
    extern __shared__ __align__(16) uint8_t se_smem[];
    const int gt = threadIdx.x, gw = gt >> 5, lane = gt & 31;
    const int64_t qi = blockIdx.x;
    const SearchSmem L = search_smem(D, W, DIMS);
    uint8_t* base = se_smem;
    float* q = reinterpret_cast<float*>(base);
    float* stage = reinterpret_cast<float*>(base + L.stage) + (size_t)gw * 32 * kStride;
    int32_t* tab = reinterpret_cast<int32_t*>(base + L.tab);
    int32_t* queue = reinterpret_cast<int32_t*>(base + L.queue);
    uint64_t* keys = reinterpret_cast<uint64_t*>(base + L.keys);
    int32_t* entry = reinterpret_cast<int32_t*>(base + L.entry);
    int* misc = reinterpret_cast<int*>(base + L.misc);  // queued, visited, entries to expand
    float* bound = reinterpret_cast<float*>(misc + 3);  // the list's ks-th distance
    auto sync = [&] {
        if (W > 1) __syncthreads();
        else __syncwarp();
    };
    constexpr bool kByStage = search_by_stage(W, DIMS);
    for (int j = gt; j < D && !kByStage; j += 32 * W) q[j] = Q[qi * D + j];
    for (int j = gt; j < (1 << tab_log2) / 4; j += 32 * W) reinterpret_cast<int4*>(tab)[j] = make_int4(-1, -1, -1, -1);
    if (gt < 3) misc[gt] = 0;
    if (gt == 0) *bound = __int_as_float(0x7f800000);
    sync();
    uint64_t list = kEmptyKey;  // entry `lane` of the list (in warp 0)

    // queues the lanes' ids (-1: none) that have not been visited; by whole warps
    auto collect = [&](int32_t id) {
        const uint32_t h = ((uint32_t)id * 2654435761u) >> (32 - tab_log2);
        const bool room = __shfl_sync(0xffffffffu, *(volatile int*)(misc + 1), 0) < full;
        bool fresh = false;
        if (id >= 0 && id < n) {
            if (room) {
                uint32_t at = h;
                for (uint32_t probe = 0; probe <= mask; ++probe) {
                    const int32_t old = atomicCAS(tab + at, -1, id);
                    fresh = old == -1;
                    if (fresh || old == id) break;
                    at = (at + 1u) & mask;
                }
            } else {
                fresh = true;
#pragma unroll
                for (int e = 0; e < kSearchNear; ++e) fresh &= *(volatile int32_t*)(tab + ((h + e) & mask)) != id;
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, fresh);
        if (bal == 0) return;
        int at = 0;
        if (lane == 0) {
            at = atomicAdd(misc, __popc(bal));
            if (room) atomicAdd(misc + 1, __popc(bal));
        }
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
        if (fresh) {
            queue[at] = id;
            // full: the id takes the place of an older one near its own
            if (!room) *(volatile int32_t*)(tab + ((h + at % kSearchNear) & mask)) = id;
        }
    };
    // distances of the queued ids, merged into the list; empties the queue
    auto process = [&] {
        sync();
        const int nq = misc[0];
        for (int b = 0; b < nq; b += 32 * W) {
            const int at = b + 32 * gw + lane;
            const int cnt = min(32, nq - (b + 32 * gw));  // this warp's rows (may be <= 0)
            const int32_t id = at < nq ? queue[at] : -1;
            float acc = 0.f;
            // a distance only grows along its chain: a row already past the
            // list's ks-th distance is dropped, its further dims are not read
            const float far = *bound;
            unsigned open = cnt >= 32 ? 0xFFFFFFFFu : cnt > 0 ? (1u << cnt) - 1u : 0u;
            for (int d0 = 0; d0 < D && open; d0 += kDims) {
                const int dl = min(kDims, D - d0);
                __syncwarp();
                // P pieces per row: a warp's lanes take 32 / P rows side by side
                constexpr int P = VEC ? kDims / 4 : 32, R = 32 / P;
                const int32_t* ids = queue + b + 32 * gw;
                if (kByStage)
                    for (int c = lane; c < dl; c += 32)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                                         (uint32_t)__cvta_generic_to_shared(q + c)),
                                     "l"(Q + qi * D + d0 + c)
                                     : "memory");
                for (int r = lane / P; r < cnt; r += R) {
                    if (!((open >> r) & 1u)) continue;
                    const float* src = X + (int64_t)ids[r] * D + d0;
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage + r * kStride);
                    if (VEC) {
                        const int c = lane % P * 4;
                        if (c < dl)
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 4 * c), "l"(src + c)
                                         : "memory");
                    } else {
                        for (int c = lane; c < dl; c += 32)
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst + 4 * c), "l"(src + c)
                                         : "memory");
                    }
                }
                asm volatile("cp.async.wait_all;\n" ::: "memory");
                __syncwarp();
                if ((open >> lane) & 1u) {  // the canonical chain: dims ascending, t = x_j - q_j, acc = fmaf(t, t, acc)
                    const float* x = stage + lane * kStride;
                    const float* y = kByStage ? q : q + d0;
                    if (VEC) {
#pragma unroll 4
                        for (int j = 0; j < dl; j += 4) {
                            const float4 u = *reinterpret_cast<const float4*>(x + j);
                            const float4 v = *reinterpret_cast<const float4*>(y + j);
                            float t = __fsub_rn(u.x, v.x);
                            acc = __fmaf_rn(t, t, acc);
                            t = __fsub_rn(u.y, v.y);
                            acc = __fmaf_rn(t, t, acc);
                            t = __fsub_rn(u.z, v.z);
                            acc = __fmaf_rn(t, t, acc);
                            t = __fsub_rn(u.w, v.w);
                            acc = __fmaf_rn(t, t, acc);
                        }
                    } else {
                        for (int j = 0; j < dl; ++j) {
                            const float t = __fsub_rn(x[j], y[j]);
                            acc = __fmaf_rn(t, t, acc);
                        }
                    }
                }
                open = __ballot_sync(0xffffffffu, ((open >> lane) & 1u) && acc <= far);
            }
            keys[32 * gw + lane] = ((open >> lane) & 1u) ? list_key(acc, (uint32_t)id) : kEmptyKey;
            sync();
            if (gw == 0) {
                for (int v = 0; v < W && b + 32 * v < nq; ++v) {
                    uint64_t cand[1] = {keys[32 * v + lane]}, out;
                    if (misc[1] >= full) {
                        // the table is no longer exact: of the ids that could
                        // enter drop those that the list holds, and repeats
                        const uint64_t kth = shfl64(list, ks - 1);
                        const bool in = cand[0] < kth;
                        unsigned left = __ballot_sync(0xffffffffu, in);
                        if (left == 0) continue;
                        const uint32_t cid = in ? list_id(cand[0]) : 0x80000000u | (uint32_t)lane;  // ids are below 2^31
                        bool drop = (__match_any_sync(0xffffffffu, cid) & ((1u << lane) - 1u)) != 0;
                        const uint32_t have = list == kEmptyKey ? 0xFFFFFFFFu : list_id(list);
                        for (; left; left &= left - 1) {
                            const int src = __ffs(left) - 1;
                            const bool held = __any_sync(0xffffffffu, have == __shfl_sync(0xffffffffu, cid, src));
                            drop |= held && lane == src;
                        }
                        if (drop || !in) cand[0] = kEmptyKey;
                    }
                    __syncwarp();
                    bool changed;
                    // the keys are distinct and at most 64, so this never declines
                    if (warp_merge_few<1>(cand, list, ks, keys + 32 * v, out, changed))
                        list = lane < ks ? out : kEmptyKey;
                    __syncwarp();
                }
                if (lane == ks - 1 && list != kEmptyKey) *bound = key_dist(list);
            }
            sync();
        }
        if (gt == 0) misc[0] = 0;
        sync();
    };
    // the queue takes one more round of every thread's id
    auto make_room = [&] {
        sync();
        const bool full = *(volatile int*)misc > kSearchQueue - 32 * W;
        sync();  // every thread has read it before one appends
        if (full) process();
    };
    for (int a0 = 0; a0 < s; a0 += 32 * W) {
        make_room();
        collect(a0 + gt < s ? S[qi * s + a0 + gt] : -1);
    }
    process();
    for (int t = 0; t < t0; ++t) {
        if (gw == 0) {  // the entries not expanded yet
            const bool open = list != kEmptyKey && (list & 1) == 0;
            const unsigned bal = __ballot_sync(0xffffffffu, open);
            if (open) {
                entry[__popc(bal & ((1u << lane) - 1u))] = (int32_t)list_id(list);
                list |= 1;
            }
            if (lane == 0) misc[2] = __popc(bal);
        }
        sync();
        const int slots = misc[2] * k;
        if (slots == 0) break;  // every entry's neighbours are visited: nothing can change any more
        for (int u0 = 0; u0 < slots; u0 += 32 * W) {
            make_room();
            const int u = u0 + gt, e = u / k;
            collect(u < slots ? G[(int64_t)entry[e] * k + (u - e * k)] : -1);
        }
        process();
    }
    if (gw == 0 && lane < ks) {
        const bool real = list != kEmptyKey;
        out_ids[qi * ks + lane] = real ? (int32_t)list_id(list) : -1;
        out_d[qi * ks + lane] = real ? key_dist(list) : __int_as_float(0x7f800000);
    }
}

template <bool VEC, int W, int DIMS>
void launch_search_t(const float* X, int64_t n, int D, const int32_t* G, int k, const float* Q, int64_t m,
                     const int32_t* S, int s, int t0, int ks, int32_t* out_ids, float* out_d, cudaStream_t st) {
    const size_t smem = search_smem(D, W, DIMS).total;
    allow_smem(k8_search<VEC, W, DIMS>);
    k8_search<VEC, W, DIMS><<<(unsigned)m, 32 * W, smem, st>>>(X, n, D, G, k, Q, S, s, t0, ks, out_ids, out_d);
}

}  // namespace

void launch_search(const float* X, int64_t n, int D, const int32_t* G, int k, const float* Q, int64_t m,
                   const int32_t* S, int s, int t0, int ks, int32_t* out_ids, float* out_d, cudaStream_t st) {
    if (m <= 0) return;
    // algorithmic bytes: every possible visit reads a row and every expansion a
    // list (an upper bound; the visits actually made are fewer)
    const double visits = (double)s + (double)t0 * ks * k;
    LaunchScope ls("k8_search", st, (double)m * (visits * (D * 4.0 + 8.0) + (double)t0 * ks * k * 4.0 + D * 4.0),
                   (double)m * visits * 3.0 * D);
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    // with less than two queries per SM the chip is idle anyway: four warps on each
    const bool few = m <= 2 * 152;
    const bool wide = D >= kSearchWide;
    for (int64_t q0 = 0; q0 < m; q0 += (int64_t)1 << 30) {  // one CTA per query
        const int64_t c = std::min(m - q0, (int64_t)1 << 30);
        const float* Qc = Q + q0 * D;
        const int32_t* Sc = S ? S + q0 * s : nullptr;
        int32_t* ic = out_ids + q0 * ks;
        float* dc = out_d + q0 * ks;
        const auto launch = few ? (vec ? launch_search_t<true, kSearchGroup, 128> : launch_search_t<false, kSearchGroup, 128>)
                          : wide ? (vec ? launch_search_t<true, 1, 128> : launch_search_t<false, 1, 128>)
                                 : (vec ? launch_search_t<true, 1, 32> : launch_search_t<false, 1, 32>);
        launch(X, n, D, G, k, Qc, c, Sc, s, t0, ks, ic, dc, st);
    }
}

}  // namespace knng
