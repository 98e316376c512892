// join.cu -- neighbour-of-neighbour refinement (the nearest-neighbour-descent
// prior art cited in Sec. 1), in Jacobi form: every offer of a round is made
// from the graph as it stood before the round, so the result does not depend
// on the order in which offers arrive.
//
//   K6 reverse lists  R[i] = the k closest j with i in G[j], by (d, j)
//   K5 local join     for every node i and every pair {u, v} of
//                     N_i = G[i] (+ R[i]), u != v: offer v to u and u to v
//                     with the canonical distance; an offer that cannot beat
//                     the target's k-th entry is dropped at the source (it
//                     could never enter the target's list)
//   scatter           group the offers by target (counts, prefix sum)
//   K4 merge          G_new[u] = first k unique of G_old[u] + offers to u
#include <algorithm>
#include <cstdlib>
#include <utility>

#include "common.cuh"
#include "kernels.h"

namespace knng {

namespace {

constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanBlock * kScanItems;

__device__ __forceinline__ int warp_incl_scan(int x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_partial(const int32_t* __restrict__ cnt, int64_t n,
                                                             int32_t* __restrict__ bsum) {
    __shared__ int wt[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int s = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        const int64_t e = base + (int64_t)threadIdx.x * kScanItems + t;
        if (e < n) s += cnt[e];
    }
    s = warp_incl_scan(s);
    if ((threadIdx.x & 31) == 31) wt[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        int w = warp_incl_scan(wt[threadIdx.x]);
        if (threadIdx.x == 31) bsum[blockIdx.x] = w;
    }
}

__global__ void __launch_bounds__(kScanBlock) k_scan_blocks(int32_t* __restrict__ bsum, int nb) {
    __shared__ int wt[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += kScanBlock) {
        const int e = base + threadIdx.x;
        const int v = e < nb ? bsum[e] : 0;
        int x = warp_incl_scan(v);
        if ((threadIdx.x & 31) == 31) wt[threadIdx.x >> 5] = x;
        __syncthreads();
        if (threadIdx.x < 32) wt[threadIdx.x] = warp_incl_scan(wt[threadIdx.x]);
        __syncthreads();
        const int before = (threadIdx.x >= 32 ? wt[(threadIdx.x >> 5) - 1] : 0) + carry;
        if (e < nb) bsum[e] = before + x - v;
        __syncthreads();
        if (threadIdx.x == kScanBlock - 1) carry = before + x;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kScanBlock) k_scan_final(const int32_t* __restrict__ cnt, int64_t n,
                                                           const int32_t* __restrict__ bsum,
                                                           int32_t* __restrict__ off) {
    __shared__ int wt[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int v[kScanItems];
    int s = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        const int64_t e = base + (int64_t)threadIdx.x * kScanItems + t;
        v[t] = e < n ? cnt[e] : 0;
        s += v[t];
    }
    const int x = warp_incl_scan(s);
    if ((threadIdx.x & 31) == 31) wt[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) wt[threadIdx.x] = warp_incl_scan(wt[threadIdx.x]);
    __syncthreads();
    int run = bsum[blockIdx.x] + (threadIdx.x >= 32 ? wt[(threadIdx.x >> 5) - 1] : 0) + x - s;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        const int64_t e = base + (int64_t)threadIdx.x * kScanItems + t;
        if (e < n) off[e] = run;
        run += v[t];
        if (e == n - 1) off[n] = run;
    }
}

__global__ void k_fill_empty(uint64_t* __restrict__ G, int64_t count) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        G[e] = kEmptyKey;
}

__global__ void k_pack(const int32_t* __restrict__ ids, const float* __restrict__ d, uint64_t* __restrict__ G,
                       int64_t count, int64_t n, int* __restrict__ status) {
    bool bad = false;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t id = ids[e];
        bad |= id < -1 || id >= n;
        G[e] = (id < 0 || id >= n) ? kEmptyKey : make_key(__fadd_rn(d[e], 0.f), (uint32_t)id);
    }
    if (bad) atomicOr(status, kStatusBadInput);
}

__global__ void k_check_ids(const int32_t* __restrict__ ids, int64_t count, int64_t lo, int64_t hi,
                            int* __restrict__ status) {
    bool bad = false;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        bad |= ids[e] < lo || ids[e] >= hi;
    if (bad) atomicOr(status, kStatusBadInput);
}

__global__ void k_unpack(const uint64_t* __restrict__ G, int32_t* __restrict__ ids, float* __restrict__ d,
                         int64_t count, int64_t id_offset) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = G[e];
        if (key == kEmptyKey) {
            ids[e] = -1;
            d[e] = __int_as_float(0x7f800000);
        } else {
            ids[e] = (int32_t)((int64_t)key_id(key) - id_offset);
            d[e] = key_dist(key);
        }
    }
}

// ---------------------------------------------------------------- K6
__global__ void k6_count(const uint64_t* __restrict__ G, int64_t nk, int32_t* __restrict__ deg) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nk; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = G[e];
        if (key != kEmptyKey) atomicAdd(&deg[key_id(key)], 1);
    }
}

// Writes every list entry into its target's reverse list: cur starts as the
// lists' offsets, so one returning atomic gives the slot.  Bound by those
// atomics and the scattered writes; the sources come in the order of the last
// tree pass's leaves (when it is known), so a target's entries are written close
// together and meet in L2.  10M x 16 entries: 9.7 ms in id order with the offset
// read beside the atomic, 6.2 so; 1M x 20: 0.42 -> 0.30.
__global__ void k6_fill(const uint64_t* __restrict__ G, uint32_t nk, uint32_t k, int64_t n,
                        const int32_t* __restrict__ order, int32_t* __restrict__ cur, uint64_t* __restrict__ rbuf) {
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < nk; e += gridDim.x * blockDim.x) {
        const uint32_t p = e / k;
        const int64_t j = order ? (int64_t)order[p] : (int64_t)p;
        // a permutation of the nodes; a stray id (a failed partition, which the
        // status word reports) writes nothing outside the buffer
        if (j < 0 || j >= n) continue;
        const uint64_t key = G[j * k + (e - p * k)];
        if (key == kEmptyKey) continue;
        const uint32_t pos = (uint32_t)atomicAdd(&cur[key_id(key)], 1);
        if (pos < nk) rbuf[pos] = (key & 0xFFFFFFFF00000000ull) | (uint32_t)j;
    }
}

// k best keys of list[beg, end) merged with `run` (NO slots per lane, sorted
// list of k keys spread lane-major); duplicates merged.  Warp-wide.
template <int NO>
__device__ __forceinline__ void warp_merge_list(const uint64_t* __restrict__ list, int beg, int end, int k,
                                                uint64_t (&run)[NO]) {
    const int lane = threadIdx.x & 31;
    constexpr int NC = 4;
    for (int c = beg; c < end; c += 32 * NC) {
        uint64_t a[NC + NO];
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            const int e = c + lane + 32 * s;
            a[s] = e < end ? list[e] : kEmptyKey;
        }
        // skip the merge when nothing can enter: compare with the k-th key
        uint64_t mine = run[0];
#pragma unroll
        for (int o = 1; o < NO; ++o)
            if (o == ((k - 1) >> 5)) mine = run[o];
        const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)mine, (k - 1) & 31);
        const uint32_t hi = __shfl_sync(0xffffffffu, (uint32_t)(mine >> 32), (k - 1) & 31);
        const uint64_t last = ((uint64_t)hi << 32) | lo;
        bool any = false;
#pragma unroll
        for (int s = 0; s < NC; ++s) any |= a[s] < last;
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int o = 0; o < NO; ++o) a[NC + o] = run[o];
        sort_regs<NC + NO>(a);
        warp_select_unique<NC + NO, NO>(a, k, run);
    }
}

template <int NO>
__global__ void __launch_bounds__(256) k6_select(const uint64_t* __restrict__ rbuf, const int32_t* __restrict__ roff,
                                                 int64_t n, int k, uint64_t* __restrict__ R) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const int lane = threadIdx.x & 31;
    const int beg = roff[i], deg = roff[i + 1] - beg;
    if (deg <= 32) {
        // the usual case: every candidate fits a lane; the keys are distinct
        // (one per source list), so the sorted run's first k are the list.
        // With k <= 32 the list's order is not used (the flags look ids up
        // in a hash set and the join takes members in any order): up to k
        // candidates are the list as they come.
        uint64_t v = lane < deg ? rbuf[beg + lane] : kEmptyKey;
        if (NO > 1 || deg > k) v = warp_sort32(v);
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            const int e = lane + 32 * o;
            if (e < k) R[i * k + e] = o == 0 ? v : kEmptyKey;
        }
        return;
    }
    uint64_t run[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) run[o] = kEmptyKey;
    warp_merge_list<NO>(rbuf, roff[i], roff[i + 1], k, run);
#pragma unroll
    for (int o = 0; o < NO; ++o)
        if (lane + 32 * o < k) R[i * k + lane + 32 * o] = run[o];
}

// Whether `key` is one of the sorted keys list[0 .. k).
__device__ __forceinline__ bool sorted_has(const uint64_t* list, int k, uint64_t key) {
    int lo = 0, len = k;
    while (len > 0) {
        const int half = len >> 1;
        if (list[lo + half] < key) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return lo < k && list[lo] == key;
}

// Member flags of one round.  A member of node i (an entry of G_old[i] or of
// R[i]) is old when the same key was a member of i in the previous round
// (in G_prev[i] or R_prev[i]): both directions of a pair of old members were
// offered then, and such an offer is now either in its target's list already
// or beaten by the target's k-th entry (which never gets worse), so the join
// may skip the pair without changing the result.  One warp per node; bit e of
// fnew[i] (rnew[i]) marks entry e of G_old[i] (R[i]) new; nodes with a new
// member are appended to `active` (one atomic per block), unless `active` is
// NULL: then k6_active lists them afterwards in a given order.
constexpr int kFlagWarps = 16;
template <int NO>
__global__ void __launch_bounds__(32 * kFlagWarps) k6_flags(const uint64_t* __restrict__ Gcur,
                                                            const uint64_t* __restrict__ Rcur,
                                                            const uint64_t* __restrict__ Gprev,
                                                            const uint64_t* __restrict__ Rprev, int64_t n, int k,
                                                            uint64_t* __restrict__ fnew, uint64_t* __restrict__ rnew,
                                                            int32_t* __restrict__ active,
                                                            int32_t* __restrict__ nactive) {
    __shared__ uint64_t prev[kFlagWarps][2][32 * NO];
    __shared__ int act[kFlagWarps];
    __shared__ int base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kFlagWarps + w;
    int on = 0;
    if (i < n) {
        uint64_t fb = 0, rb = 0;
        if (NO == 1) {
            // k <= 32: by id (a pair always has the same canonical distance,
            // the same both ways), in a hash set of the previous members'
            // ids (at most 64 in 128 slots, linear probing); no list needs
            // to be sorted
            uint32_t* tab = reinterpret_cast<uint32_t*>(prev[w]);
            constexpr uint32_t kFree = 0xFFFFFFFFu;
            const uint64_t gk = lane < k ? Gcur[i * k + lane] : kEmptyKey;
            const uint64_t rk = (Rcur && lane < k) ? Rcur[i * k + lane] : kEmptyKey;
            const uint64_t pgk = lane < k ? Gprev[i * k + lane] : kEmptyKey;
            const uint64_t prk = (Rprev && lane < k) ? Rprev[i * k + lane] : kEmptyKey;
            for (int t = lane; t < 128; t += 32) tab[t] = kFree;
            __syncwarp();
            auto home = [](uint32_t id) { return (id * 2654435761u) >> 25; };
            for (int src = 0; src < 2; ++src) {
                const uint64_t key = src == 0 ? pgk : prk;
                if (key == kEmptyKey) continue;
                const uint32_t id = key_id(key);
                for (uint32_t h = home(id), t = 0; t < 128; ++t, h = (h + 1) & 127) {
                    const uint32_t old = atomicCAS(&tab[h], kFree, id);
                    if (old == kFree || old == id) break;
                }
            }
            __syncwarp();
            auto seen = [&](uint64_t key) {
                const uint32_t id = key_id(key);
                for (uint32_t h = home(id), t = 0; t < 128; ++t, h = (h + 1) & 127) {
                    const uint32_t v = tab[h];
                    if (v == id) return true;
                    if (v == kFree) return false;
                }
                return false;
            };
            fb = __ballot_sync(0xffffffffu, gk != kEmptyKey && !seen(gk));
            if (Rcur) rb = __ballot_sync(0xffffffffu, rk != kEmptyKey && !seen(rk));
        } else {
            uint64_t* pg = prev[w][0];
            uint64_t* pr = prev[w][1];
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const int e = lane + 32 * o;
                pg[e] = e < k ? Gprev[i * k + e] : kEmptyKey;
                pr[e] = (Rprev && e < k) ? Rprev[i * k + e] : kEmptyKey;
            }
            __syncwarp();
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const int e = lane + 32 * o;
                uint64_t key = e < k ? Gcur[i * k + e] : kEmptyKey;
                bool nw = key != kEmptyKey && !sorted_has(pg, k, key) && !(Rprev && sorted_has(pr, k, key));
                fb |= (uint64_t)__ballot_sync(0xffffffffu, nw) << (32 * o);
                if (Rcur) {
                    key = e < k ? Rcur[i * k + e] : kEmptyKey;
                    nw = key != kEmptyKey && !sorted_has(pg, k, key) && !(Rprev && sorted_has(pr, k, key));
                    rb |= (uint64_t)__ballot_sync(0xffffffffu, nw) << (32 * o);
                }
            }
        }
        if (lane == 0) {
            fnew[i] = fb;
            if (Rcur) rnew[i] = rb;
        }
        on = (fb | rb) != 0;
    }
    if (active == nullptr) return;  // the nodes are listed by k6_active (uniform over the CTA)
    if (lane == 0) act[w] = on;
    __syncthreads();
    if (threadIdx.x == 0) {
        int c = 0;
        for (int q = 0; q < kFlagWarps; ++q) c += act[q];
        base = c > 0 ? atomicAdd(nactive, c) : 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int at = base;
        for (int q = 0; q < kFlagWarps; ++q)
            if (act[q]) active[at++] = (int32_t)((int64_t)blockIdx.x * kFlagWarps + q);
    }
}

// The nodes with a new member listed in the order of `order` (position p
// listed when node order[p] has a new member in fnew / rnew, as k6_flags
// wrote them): positions keep their order inside a CTA, one atomic per CTA.
__global__ void __launch_bounds__(256) k6_active(const int32_t* __restrict__ order,
                                                 const uint64_t* __restrict__ fnew,
                                                 const uint64_t* __restrict__ rnew, int64_t n,
                                                 int32_t* __restrict__ active, int32_t* __restrict__ nactive) {
    __shared__ int wbefore[8];
    __shared__ int base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    int32_t i = 0;
    bool on = false;
    if (p < n) {
        i = order[p];
        // a permutation of the nodes; a stray id (a failed partition, which
        // the status word reports) lists nothing
        on = i >= 0 && i < n && (fnew[i] | (rnew ? rnew[i] : 0ull)) != 0;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    if (lane == 0) wbefore[w] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        int c = 0;
        for (int q = 0; q < 8; ++q) {
            const int t = wbefore[q];
            wbefore[q] = c;
            c += t;
        }
        base = c > 0 ? atomicAdd(nactive, c) : 0;
    }
    __syncthreads();
    if (on) active[base + wbefore[w] + __popc(bal & ((1u << lane) - 1u))] = i;
}

// ---------------------------------------------------------------- K5
// The FP32 local join with the pairs of several nodes spread over one CTA.
// A node's member pairs are cut into the 4 x 4 blocks of the upper triangle
// of its (mcap / 4)-group member grid: NB = RGN (RGN + 1) / 2 blocks, RGN =
// mcap / 4; a CTA of 256 threads takes G = 256 / NB nodes at a time.  Block
// (rg, cg) holds members {4 rg + a} x {4 cg + b}.  Distances are canonical
// (dims ascending, fmaf); surviving offers are appended to the chunk's buffer.
// A pair of members that shared a leaf in one of the build's last tree passes
// makes none (the leaf stage offered it already).
//
// Only blocks that can make an offer are computed: both groups hold members,
// one holds a new one (members are new first), and, in the first round, some
// pair shared no leaf (there the members come in the order of the leaf they
// share with the node, which makes whole blocks of leaf-mates).  1M x 96,
// k = 16: 8.7 of the 21 blocks in the first round, then 11.1, 8.2 and 5.7.
// They are listed in shared memory and dealt one per thread, so full warps
// compute and the others go on to wait; co-resident CTAs start at different
// warps.
//
// Bound by issue slots and the barriers between gather and sums.  So the
// differences and sums are paired FP32 instructions, two pairs of members
// each: members 4 g + 2 h and 4 g + 2 h + 1 are staged interleaved dim by dim
// in row h RGN + g, (r0, r1) - (c0, c1) and (r0, r1) - (c1, c0) give all four
// differences of two such rows, and every sum keeps its chain.  Lanes of
// consecutive cg read consecutive rows (an odd number of 16-byte pieces apart:
// different banks), lanes of one rg the same.  The gather's indices are
// stepped without divisions and two pieces are in flight per thread (one or
// three: 16.7 and 16.3 ms against 15.9 below); offers are a bit mask per
// thread, so that only the pairs that make one are visited again.  128 threads
// a CTA: 20.5.
// Four rounds on 1M x 96, k = 16: 31.8 ms with every block and scalar
// instructions, 27.1 paired, 21.3 with the live blocks dealt densely, 19.8
// with the stepped gather, 15.9 with the mask.  A form with one node per warp
// is gone: with the same gains it would idle the lanes past a node's blocks
// (100,000 x 960, k = 20: 17.8 against 11.6 ms; 300,000 x 96, k = 32: 24.0
// against 12.7; forward lists of 64: 40.6 against 23.8; none was faster).
constexpr int kJ2Threads = 256;
constexpr int kJ2Dist = 20;  // floats of a thread's 16 distances in shared memory (16 plus padding)
constexpr int kJ2Ahead = 2;  // pieces of the gather in flight per thread

struct J2Layout {
    int RGN, NB, G, dch, stride;
    size_t thr, lid, rows, mem, cnt, live, total;
};

__host__ __device__ inline J2Layout j2_layout(int D, int mcap, bool leafids) {
    J2Layout L;
    L.RGN = mcap / 4;
    L.NB = L.RGN * (L.RGN + 1) / 2;
    L.G = kJ2Threads / L.NB;  // mcap <= 64: NB <= 136
    const int slots = L.G * mcap;
    const int d4 = (D + 3) & ~3;
    int cap = (kJ2Threads * 176 / (slots * 4) - 4) & ~3;
    if (cap < 4) cap = 4;
    const int nch = (d4 + cap - 1) / cap;
    L.dch = ((d4 + nch - 1) / nch + 3) & ~3;
    L.stride = 2 * L.dch + 4;  // an odd number of 16-byte pieces
    L.thr = 0;
    L.lid = L.thr + (size_t)slots * 8;
    L.rows = L.lid + (leafids ? (size_t)slots * 16 : 0);
    const size_t rows = (size_t)(slots / 2) * L.stride * 4, dist = (size_t)kJ2Threads * kJ2Dist * 4;
    L.mem = L.rows + (rows > dist ? rows : dist);
    L.cnt = L.mem + (size_t)slots * 4;
    L.live = L.cnt + (size_t)L.G * 2 * 4;
    L.total = L.live + (size_t)(1 + kJ2Threads) * 4;
    return L;
}

__device__ __forceinline__ int j2_slot(int m, int RGN) { return (m & 3) * RGN + (m >> 2); }
// Where member m's id lies: pair row p's two ids are neighbours.
__device__ __forceinline__ int j2_mem(int m, int RGN) { return 2 * ((m & 2) / 2 * RGN + (m >> 2)) + (m & 1); }

__global__ void __launch_bounds__(kJ2Threads, 1024 / kJ2Threads) k5_join_cta(const float* __restrict__ X, int D, int k, int rev,
                                                         int mcap, const uint64_t* __restrict__ Gold,
                                                         const uint64_t* __restrict__ R,
                                                         const int32_t* __restrict__ list,
                                                         const uint64_t* __restrict__ fnew,
                                                         const uint64_t* __restrict__ rnew, int64_t node0,
                                                         int64_t node1, uint32_t* __restrict__ counter, int64_t cap,
                                                         uint32_t* __restrict__ ptgt, uint64_t* __restrict__ pkey,
                                                         int32_t* __restrict__ pcnt, int* __restrict__ status,
                                                         const int* __restrict__ skip_if_exact,
                                                         const int32_t* __restrict__ count_dev,
                                                         const int32_t* __restrict__ leafid, int npass,
                                                         int32_t* __restrict__ ovf_list,
                                                         int32_t* __restrict__ ovf_count) {
    extern __shared__ float4 smem4[];
    if (*status & kStatusStop) return;
    if (count_dev && (int64_t)*count_dev < node1) node1 = *count_dev;
    if (skip_if_exact) {  // the tensor-core join does this round when the 16-bit copy is exact
        const int f = *skip_if_exact;
        if ((f & 1) == 0 && !((f & 2) && (f & 4))) return;
    }
    const bool lids = leafid != nullptr && npass > 0;
    const J2Layout L = j2_layout(D, mcap, lids);
    char* base = reinterpret_cast<char*>(smem4);
    uint64_t* thr = reinterpret_cast<uint64_t*>(base + L.thr);  // [G][mcap] by slot
    int4* slid = reinterpret_cast<int4*>(base + L.lid);         // [G][mcap] by slot
    float* rows = reinterpret_cast<float*>(base + L.rows);      // [G][mcap / 2][stride] by pair row
    int32_t* mem = reinterpret_cast<int32_t*>(base + L.mem);    // [G][mcap / 2][2] by pair row, -1: none
    int* cnt = reinterpret_cast<int*>(base + L.cnt);            // [G] members, then [G] new members
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int RGN = L.RGN, NB = L.NB, G = L.G, dch = L.dch, stride = L.stride;
    int* nlive = reinterpret_cast<int*>(base + L.live);  // blocks to compute, then the blocks
    uint32_t* items = reinterpret_cast<uint32_t*>(nlive + 1);  // node | rg << 8 | cg << 16
    // the block this thread lists, fixed for the launch
    uint32_t own = 0u;
    if (tid < G * NB) {
        const int j = tid / NB;
        int b = tid - j * NB, g = 0;
        while (b >= RGN - g) {
            b -= RGN - g;
            ++g;
        }
        own = (uint32_t)(j | g << 8 | (g + b) << 16);
    }
    // every member is new in a build's first round: then most pairs are leaf-mates
    const bool by_leaf = lids && fnew == nullptr && rnew == nullptr;
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    // the gather's pieces: piece c4 of pair row pr, stepped without divisions
    const int q4 = dch >> 2, half = mcap / 2;
    const int pr0 = tid / q4, c40 = tid - pr0 * q4, dpr = kJ2Threads / q4, dc = kJ2Threads - dpr * q4;
    const int64_t ngroups = (node1 - node0 + G - 1) / G;
    for (int64_t grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
        const int64_t first = node0 + grp * G;
        if (tid == 0) *nlive = 0;
        // members of the group's nodes (warp w collects nodes w, w + 8, ...):
        // the new ones first, then the old ones; each takes ids of G_old[i],
        // then of R[i] (by_leaf: in the order of the first pass in which they
        // share i's leaf)
        for (int j = warp; j < G; j += kJ2Threads / 32) {
            const int64_t pos = first + j;
            int M = 0, nn = 0;
            if (pos < node1) {
                const int64_t i = list ? (int64_t)list[pos] : pos;
                const uint64_t fbits = fnew ? fnew[i] : ~0ull, rbits = rnew ? rnew[i] : ~0ull;
                auto take_member = [&](uint64_t key, bool take) {
                    const unsigned bal = __ballot_sync(0xffffffffu, take);
                    if (take) {
                        const int m = M + __popc(bal & ((1u << lane) - 1u));
                        const uint32_t u = key_id(key);
                        const int sl = j * mcap + j2_slot(m, RGN);
                        mem[j * mcap + j2_mem(m, RGN)] = (int32_t)u;
                        thr[sl] = Gold[(int64_t)u * k + k - 1];
                        if (lids) slid[sl] = __ldg(reinterpret_cast<const int4*>(leafid) + u);
                    }
                    M += __popc(bal);
                };
                // at most 64 entries, a mutual neighbour once
                uint64_t key0, key1;
                bool new0, new1;
                member_keys(Gold, R, i, k, rev != 0, fbits, rbits, key0, key1, new0, new1);
                // more members than the slot holds (slots smaller than 2k):
                // the node goes to the overflow list, for the full-slot launch
                const int all = __popc(__ballot_sync(0xffffffffu, key0 != kEmptyKey)) +
                                __popc(__ballot_sync(0xffffffffu, key1 != kEmptyKey));
                if (all > mcap) {
                    if (lane == 0) ovf_list[atomicAdd(ovf_count, 1)] = (int32_t)i;
                    key0 = key1 = kEmptyKey;
                }
                if (by_leaf) {
                    const int4* lp = reinterpret_cast<const int4*>(leafid);
                    const int4 li = __ldg(lp + i);
                    const int q0 = key0 == kEmptyKey ? -1 : leaf_shared(li, __ldg(lp + key_id(key0)), npass);
                    const int q1 = key1 == kEmptyKey ? -1 : leaf_shared(li, __ldg(lp + key_id(key1)), npass);
                    for (int q = 0; q <= npass; ++q) {
                        take_member(key0, q0 == q);
                        take_member(key1, q1 == q);
                    }
                    nn = M;
                } else {
                    for (int want = 1; want >= 0; --want) {
                        take_member(key0, key0 != kEmptyKey && new0 == (want == 1));
                        take_member(key1, key1 != kEmptyKey && new1 == (want == 1));
                        if (want == 1) nn = M;
                    }
                }
            }
            for (int m = M + lane; m < mcap; m += 32) mem[j * mcap + j2_mem(m, RGN)] = -1;
            if (lane == 0) {
                cnt[j] = M;
                cnt[G + j] = nn;
            }
        }
        __syncthreads();
        // list the blocks that can make an offer: both groups hold members, one
        // holds a new one, and not every pair of theirs shared a leaf
        {
            bool on = false;
            if (tid < G * NB) {
                const int j = own & 255, rg = own >> 8 & 255, cg = own >> 16, M = cnt[j], nn = cnt[G + j];
                on = 4 * cg < M && (4 * rg < nn || 4 * cg < nn);
                if (on && by_leaf) {
                    on = false;
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const int4 lb = slid[j * mcap + b * RGN + cg];
#pragma unroll
                        for (int a = 0; a < 4; ++a)
                            on |= 4 * rg + a < M && 4 * cg + b < M && (rg < cg || a < b) &&
                                  !leaf_mates(slid[j * mcap + a * RGN + rg], lb, npass);
                    }
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            int at = 0;
            if (lane == 0 && bal) at = atomicAdd(nlive, __popc(bal));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (on) items[at + __popc(bal & ((1u << lane) - 1u))] = own;
        }
        bool live = false;
        int jn = 0, rg = 0, cg = 0, Mj = 0, nnj = 0;
        // sums of (2 h, 2 w), (2 h + 1, 2 w + 1) and of (2 h, 2 w + 1), (2 h + 1, 2 w)
        uint64_t same[2][2], cross[2][2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int w = 0; w < 2; ++w) same[h][w] = cross[h][w] = 0ull;
        for (int d0 = 0; d0 < D; d0 += dch) {
            const int dl = min(dch, D - d0);
            // gather dims [d0, d0 + dch) of every member, two members
            // interleaved (zeros past D and for a pair row's missing second
            // member; a pair row without members is not written, and nothing
            // reads the sums it enters)
            if (vec) {
                int pr = pr0, c4 = c40;
                while (pr < G * half) {
                    int2 id[kJ2Ahead];
                    float4 u[kJ2Ahead], v[kJ2Ahead];
                    int at[kJ2Ahead], c[kJ2Ahead];
#pragma unroll
                    for (int q = 0; q < kJ2Ahead; ++q) {
                        id[q] = pr < G * half ? *reinterpret_cast<const int2*>(mem + 2 * pr) : make_int2(-1, -1);
                        at[q] = pr * stride;
                        c[q] = c4;
                        const bool in = c4 * 4 < dl;
                        u[q] = v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (in && id[q].x >= 0) u[q] = __ldg(reinterpret_cast<const float4*>(X + (int64_t)id[q].x * D + d0) + c4);
                        if (in && id[q].y >= 0) v[q] = __ldg(reinterpret_cast<const float4*>(X + (int64_t)id[q].y * D + d0) + c4);
                        pr += dpr;
                        c4 += dc;
                        if (c4 >= q4) {
                            c4 -= q4;
                            ++pr;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < kJ2Ahead; ++q)
                        if (id[q].x >= 0) store_pairs(rows + at[q] + c[q] * 8, u[q], v[q], (c[q] >> 2) & 1);
                }
            } else {
                for (int e = tid; e < G * half * dch; e += kJ2Threads) {
                    const int pr = e / dch, c = e - pr * dch;
                    const int2 id = *reinterpret_cast<const int2*>(mem + 2 * pr);
                    const bool in = c < dl;
                    *reinterpret_cast<float2*>(rows + (size_t)pr * stride + 2 * c) =
                        make_float2(in && id.x >= 0 ? __ldg(X + (int64_t)id.x * D + d0 + c) : 0.f,
                                    in && id.y >= 0 ? __ldg(X + (int64_t)id.y * D + d0 + c) : 0.f);
                }
            }
            __syncthreads();
            if (d0 == 0) {  // the blocks go densely to the warps, from another one for each CTA of an SM
                const int it = (tid + 32 * (int)(grp / 152)) & (kJ2Threads - 1);
                live = it < *nlive;
                if (live) {
                    const uint32_t e = items[it];
                    jn = e & 255, rg = e >> 8 & 255, cg = e >> 16;
                    Mj = cnt[jn], nnj = cnt[G + jn];
                }
            }
            if (live) {
                const float* rp = rows + (size_t)(jn * half + rg) * stride;
                const float* cp = rows + (size_t)(jn * half + cg) * stride;
                const int step = RGN * stride;  // members 4 g + 2, 4 g + 3 sit RGN rows below 4 g, 4 g + 1
                for (int dq = 0; dq < 2 * dch; dq += 8) {  // 4 dims
                    ulonglong2 r[2][2], c[2][2];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            r[h][p] = *reinterpret_cast<const ulonglong2*>(rp + h * step + dq + 4 * p);
                            c[h][p] = *reinterpret_cast<const ulonglong2*>(cp + h * step + dq + 4 * p);
                        }
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int w = 0; w < 2; ++w) {
                            const uint64_t c0 = c[w][p].x, c1 = c[w][p].y, x0 = swap_pair(c0), x1 = swap_pair(c1);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                same[h][w] = add_square(r[h][p].x, c0, same[h][w]);
                                cross[h][w] = add_square(r[h][p].x, x0, cross[h][w]);
                                same[h][w] = add_square(r[h][p].y, c1, same[h][w]);
                                cross[h][w] = add_square(r[h][p].y, x1, cross[h][w]);
                            }
                        }
                }
            }
            __syncthreads();  // the next chunk overwrites the rows
        }
        // offers: a bit per direction of the block's 16 pairs (2 (4 a + b): b
        // offered to a; plus 1: a to b), their distances in shared memory (the
        // rows are done with), then one slot range per warp
        uint32_t hits = 0;
        float* dist = rows + tid * kJ2Dist;
        const int2* id2 = reinterpret_cast<const int2*>(mem) + jn * half;  // the node's ids by pair row
        if (live) {
            const int2 u0 = id2[rg], u1 = id2[RGN + rg], v0 = id2[cg], v1 = id2[RGN + cg];
            const uint32_t u[4] = {(uint32_t)u0.x, (uint32_t)u0.y, (uint32_t)u1.x, (uint32_t)u1.y};
            const uint32_t v[4] = {(uint32_t)v0.x, (uint32_t)v0.y, (uint32_t)v1.x, (uint32_t)v1.y};
            uint64_t tv[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) tv[b] = thr[jn * mcap + b * RGN + cg];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const uint64_t tu = thr[jn * mcap + a * RGN + rg];
                float d[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const uint64_t sum = (a ^ b) & 1 ? cross[a >> 1][b >> 1] : same[a >> 1][b >> 1];
                    d[b] = __uint_as_float((uint32_t)(a & 1 ? sum >> 32 : sum));
                    const int ia = 4 * rg + a, ib = 4 * cg + b;
                    const bool pair = ia < Mj && ib < Mj && (ia < nnj || ib < nnj) && (rg < cg || a < b) && u[a] != v[b];
                    hits |= (uint32_t)(pair && make_key(d[b], v[b]) < tu) << (2 * (4 * a + b));
                    hits |= (uint32_t)(pair && make_key(d[b], u[a]) < tv[b]) << (2 * (4 * a + b) + 1);
                }
                *reinterpret_cast<float4*>(dist + 4 * a) = make_float4(d[0], d[1], d[2], d[3]);
            }
        }
        if (lids) {
            for (uint32_t rest = (hits | hits >> 1) & 0x55555555u; rest; rest &= rest - 1) {
                const int bit = __ffs(rest) - 1, a = bit >> 3, b = bit >> 1 & 3;
                if (leaf_mates(slid[jn * mcap + a * RGN + rg], slid[jn * mcap + b * RGN + cg], npass))
                    hits &= ~(3u << bit);
            }
        }
        const int c = __popc(hits), incl = warp_incl_scan(c);
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (total > 0) {
            uint32_t at = 0;
            if (lane == 31) at = atomicAdd(counter, (uint32_t)total);
            at = __shfl_sync(0xffffffffu, at, 31);
            if ((int64_t)at + total > cap) {
                if (lane == 0) atomicOr(status, kStatusOverflow);
            } else {
                uint32_t w = at + incl - c;
                const int* ids = mem + jn * mcap;
                for (; hits; hits &= hits - 1) {
                    const int bit = __ffs(hits) - 1, a = bit >> 3, b = bit >> 1 & 3;
                    const uint32_t u = (uint32_t)ids[2 * ((a >> 1) * RGN + rg) + (a & 1)],
                                   v = (uint32_t)ids[2 * ((b >> 1) * RGN + cg) + (b & 1)];
                    const uint32_t to = bit & 1 ? v : u;
                    ptgt[w] = to;
                    pkey[w] = make_key(dist[bit >> 1], bit & 1 ? u : v);
                    ++w;
                    atomicAdd(&pcnt[to], 1);
                }
            }
        }
        __syncthreads();  // the next group overwrites members, thresholds and counts
    }
}

__global__ void k5_scatter(const uint32_t* __restrict__ ptgt, const uint64_t* __restrict__ pkey,
                           const uint32_t* __restrict__ counter, int64_t cap, const int32_t* __restrict__ poff,
                           int32_t* __restrict__ pcur, uint64_t* __restrict__ grouped,
                           const int* __restrict__ status, unsigned long long* __restrict__ offers_total) {
    // after an overflow some reserved slots were never written: group nothing
    if (*status & kStatusStop) return;
    const int64_t total = min((int64_t)*counter, cap);
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(offers_total, (unsigned long long)total);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = ptgt[q];
        const int pos = poff[t] + atomicAdd(&pcur[t], 1);
        grouped[pos] = pkey[q];
    }
}

// An offer of `key` to a node whose sorted list is row[0..k) can change the
// list only if it beats the k-th entry and is not one of the entries already
// (an id always comes with the same canonical distance, hence the same key).
__device__ __forceinline__ bool offer_useful(uint64_t key, const uint64_t* row, int k) {
    if (!(key < row[k - 1])) return false;
    int lo = 0, len = k;
    while (len > 0) {
        const int half = len >> 1;
        if (row[lo + half] < key) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return row[lo] != key;
}

// Merges up to kFewOffers offers into a list of k <= 32 distinct keys held one
// per lane (`run`, ascending; lanes past k hold empty keys), 32 at a time.  An
// offer enters when it is below the k-th key and its id is neither in the list
// nor in a lower lane (a pair always has the same canonical distance, and a
// repeat of an offer that did not make the list cannot make it later: the k-th
// key only falls).  Every list entry and every offer that enters then counts
// what lies below it: that is its place.  `key`: the lane's first offer.
// Returns whether the list changed.
constexpr int kFewOffers = 160;
__device__ __forceinline__ bool merge_few_offers(const uint64_t* __restrict__ grouped, int beg, int end, int k,
                                                 uint64_t key, uint64_t& run, uint64_t* scratch) {
    const int lane = threadIdx.x & 31;
    bool changed = false;
    for (int c = beg; c < end; c += 32) {
        if (c > beg) key = c + lane < end ? grouped[c + lane] : kEmptyKey;
        bool in = key < shfl64(run, k - 1);
        if (!__any_sync(0xffffffffu, in)) continue;
        // lanes without an offer match themselves only: ids are below 2^31
        const uint32_t id = in ? key_id(key) : 0x80000000u | (uint32_t)lane;
        const unsigned same = __match_any_sync(0xffffffffu, id);
        in &= (same & ((1u << lane) - 1u)) == 0;
        const uint32_t have = run == kEmptyKey ? 0xFFFFFFFFu : key_id(run);
        for (int e = 0; e < k; ++e) {
            const uint32_t other = __shfl_sync(0xffffffffu, have, e);
            in &= other != id;
        }
        const unsigned ins = __ballot_sync(0xffffffffu, in);
        if (!ins) continue;
        int at = 0, to = lane;  // places of the lane's offer and of its list entry
        for (unsigned m = ins; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const uint64_t o = shfl64(key, src);
            const int below = __popc(__ballot_sync(0xffffffffu, run < o));
            at += lane == src ? below : (o < key ? 1 : 0);
            to += o < run ? 1 : 0;
        }
        if (to < k) scratch[to] = run;
        __syncwarp();
        if (in && at < k) scratch[at] = key;
        __syncwarp();
        run = lane < k ? scratch[lane] : kEmptyKey;
        __syncwarp();
        changed = true;
    }
    return changed;
}

// A node's list and its first 32 offers, one per lane, as loaded.
template <int NO>
struct MergeLoad {
    int64_t u;
    int beg, end;
    uint64_t run[NO], key;
    __device__ __forceinline__ void load(const uint64_t* Gnew, const uint64_t* __restrict__ grouped, int64_t u_,
                                         int beg_, int end_, int k) {
        const int lane = threadIdx.x & 31;
        u = u_;
        beg = beg_;
        end = end_;
#pragma unroll
        for (int o = 0; o < NO; ++o) run[o] = lane + 32 * o < k ? Gnew[u * k + lane + 32 * o] : kEmptyKey;
        key = beg + lane < end ? grouped[beg + lane] : kEmptyKey;
    }
};

// Merges one node's offers into its list.  Usually by merge_few_offers; else
// (k > 32, more offers, or a given list that holds a key twice) the list sits
// in shared memory, every lane drops the offers that cannot change it, and
// the rest go through the warp selection.  Bound by instructions and the latency
// of its loads: four rounds on 10M x 96, k = 16 took 48.7 ms when the ids went
// through a hash set in shared memory and the survivors through a bitonic sort
// and merge, 35.1 by counting places and with the next node's loads in flight;
// 1M x 128, k = 20 1.55 -> 1.23.
template <int NO>
__device__ __forceinline__ void merge_node(uint64_t* __restrict__ Gnew, const uint64_t* __restrict__ grouped,
                                           const MergeLoad<NO>& in, int k, uint64_t* srow, uint64_t* scratch) {
    const int lane = threadIdx.x & 31, beg = in.beg, end = in.end;
    uint64_t* row = Gnew + in.u * k;
    uint64_t run[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) run[o] = in.run[o];
    if (NO == 1 && end - beg <= kFewOffers) {
        const uint64_t next = shfl64(run[0], (lane + 1) & 31);
        if (!__any_sync(0xffffffffu, lane < 31 && run[0] != kEmptyKey && run[0] == next)) {
            if (merge_few_offers(grouped, beg, end, k, in.key, run[0], scratch) && lane < k) row[lane] = run[0];
            return;
        }
    }
#pragma unroll
    for (int o = 0; o < NO; ++o) srow[lane + 32 * o] = run[o];
    __syncwarp();
    constexpr int NC = 4;
    bool changed = false;
    for (int c = beg; c < end; c += 32 * NC) {
        uint64_t a[NC + NO];
        bool any = false;
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            const int e = c + lane + 32 * s;
            a[s] = (e < end) ? grouped[e] : kEmptyKey;
            if (a[s] != kEmptyKey && !offer_useful(a[s], srow, k)) a[s] = kEmptyKey;
            any |= a[s] != kEmptyKey;
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int o = 0; o < NO; ++o) a[NC + o] = run[o];
        sort_regs<NC + NO>(a);
        warp_select_unique<NC + NO, NO>(a, k, run);
        __syncwarp();
#pragma unroll
        for (int o = 0; o < NO; ++o) srow[lane + 32 * o] = run[o];
        __syncwarp();
        changed = true;
    }
    if (changed) {
#pragma unroll
        for (int o = 0; o < NO; ++o)
            if (lane + 32 * o < k) row[lane + 32 * o] = run[o];
    }
    __syncwarp();  // srow is reused by the warp's next node
}

// Warps stride over groups of 32 targets; the targets of a group that
// received offers are merged one after the other.
template <int NO>
__global__ void __launch_bounds__(256) k4_merge(uint64_t* __restrict__ Gnew, const uint64_t* __restrict__ grouped,
                                                const int32_t* __restrict__ poff, int64_t n, int k,
                                                const int* __restrict__ status) {
    __shared__ uint64_t rows[8][32 * NO];
    __shared__ uint64_t scratch[8][32];
    if (*status & kStatusStop) return;
    const int lane = threadIdx.x & 31;
    uint64_t* srow = rows[threadIdx.x >> 5];
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t g0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32; g0 < n; g0 += warps * 32) {
        const int64_t u = g0 + lane;
        const int beg = u < n ? poff[u] : 0, end = u < n ? poff[u + 1] : 0;
        unsigned todo = __ballot_sync(0xffffffffu, end > beg);
        // the next node's loads are in flight while one is merged
        MergeLoad<NO> now, next;
        auto load = [&](MergeLoad<NO>& to) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            to.load(Gnew, grouped, g0 + src, __shfl_sync(0xffffffffu, beg, src), __shfl_sync(0xffffffffu, end, src), k);
        };
        if (todo) load(next);
        else continue;
        for (bool more = true; more;) {
            now = next;
            more = todo != 0;
            if (more) load(next);
            merge_node<NO>(Gnew, grouped, now, k, srow, scratch[threadIdx.x >> 5]);
        }
    }
}

// One warp per leaf: slot `slot` of point perm[p]'s leaf ids = leaf, for the
// leaf's positions p.
__global__ void __launch_bounds__(256) k_leaf_ids(const int32_t* __restrict__ perm,
                                                  const int32_t* __restrict__ leaf_off, int nleaf, int slot,
                                                  int32_t* __restrict__ lid) {
    const int lane = threadIdx.x & 31;
    for (int l = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5); l < nleaf;
         l += (int)((gridDim.x * (int64_t)blockDim.x) >> 5))
        for (int p = leaf_off[l] + lane; p < leaf_off[l + 1]; p += 32)
            lid[(int64_t)perm[p] * kMaxLeafPasses + slot] = l;
}

inline int grid_for(int64_t count, int block) {
    int64_t g = (count + block - 1) / block;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

size_t scan_tmp_ints(int64_t n) { return (size_t)((n + kScanTile - 1) / kScanTile) + 1; }

void launch_scan(const int32_t* cnt, int32_t* off, int64_t n, int32_t* tmp, cudaStream_t s) {
    const int nb = (int)((n + kScanTile - 1) / kScanTile);
    LaunchScope ls("k_scan", s, n * 8.0, 0, nb == 0 ? 0 : 3);
    if (nb == 0) {
        cudaMemsetAsync(off, 0, sizeof(int32_t), s);
        return;
    }
    k_scan_partial<<<nb, kScanBlock, 0, s>>>(cnt, n, tmp);
    k_scan_blocks<<<1, kScanBlock, 0, s>>>(tmp, nb);
    k_scan_final<<<nb, kScanBlock, 0, s>>>(cnt, n, tmp, off);
}

void launch_leaf_ids(const int32_t* perm, const int32_t* leaf_off, int nleaf, int64_t n, int slot, int32_t* lid,
                     cudaStream_t s) {
    if (nleaf <= 0) return;
    LaunchScope ls("k_leaf_ids", s, n * 8.0 + nleaf * 4.0, 0);
    k_leaf_ids<<<grid_for((int64_t)nleaf * 32, 256), 256, 0, s>>>(perm, leaf_off, nleaf, slot, lid);
}

void launch_fill_empty(uint64_t* G, int64_t count, cudaStream_t s) {
    LaunchScope ls("k_fill_empty", s, count * 8.0, 0);
    k_fill_empty<<<grid_for(count, 256), 256, 0, s>>>(G, count);
}

void launch_pack(const int32_t* ids, const float* d, uint64_t* G, int64_t count, int64_t n, int* status,
                 cudaStream_t s) {
    LaunchScope ls("k_pack", s, count * 16.0, 0);
    k_pack<<<grid_for(count, 256), 256, 0, s>>>(ids, d, G, count, n, status);
}

void launch_check_ids(const int32_t* ids, int64_t count, int64_t lo, int64_t hi, int* status, cudaStream_t s) {
    if (count <= 0) return;
    LaunchScope ls("k_check_ids", s, count * 4.0, 0);
    k_check_ids<<<grid_for(count, 256), 256, 0, s>>>(ids, count, lo, hi, status);
}

void launch_unpack(const uint64_t* G, int32_t* ids, float* d, int64_t count, cudaStream_t s, int64_t id_offset) {
    LaunchScope ls("k_unpack", s, count * 16.0, 0);
    k_unpack<<<grid_for(count, 256), 256, 0, s>>>(G, ids, d, count, id_offset);
}

void launch_reverse_lists(const uint64_t* G, int64_t n, int k, const JoinBuffers& b, cudaStream_t s) {
    const int64_t nk = n * k;
    cudaMemsetAsync(b.deg, 0, sizeof(int32_t) * (n + 1), s);
    {
        LaunchScope ls("k6_count", s, nk * 8.0 + nk * 4.0, 0);
        k6_count<<<grid_for(nk, 256), 256, 0, s>>>(G, nk, b.deg);
    }
    launch_scan(b.deg, b.roff, n, b.scan_tmp, s);
    cudaMemcpyAsync(b.cur, b.roff, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
    {
        LaunchScope ls("k6_fill", s, nk * (8.0 + 8.0 + 8.0), 0);
        k6_fill<<<grid_for(nk, 256), 256, 0, s>>>(G, (uint32_t)nk, (uint32_t)k, n, b.order, b.cur, b.rbuf);
    }
    LaunchScope ls("k6_select", s, nk * 16.0 + n * 8.0, 0);
    const int grid = (int)((n * 32 + 255) / 256);
    if (k > 32)
        k6_select<2><<<grid, 256, 0, s>>>(b.rbuf, b.roff, n, k, b.R);
    else
        k6_select<1><<<grid, 256, 0, s>>>(b.rbuf, b.roff, n, k, b.R);
}

namespace {

// One refinement round over the nodes at positions [0, count) of b.list
// (all nodes when b.list is NULL): reads Gold (and b.R), writes Gnew.
const char* launch_join_chunk(const float* X, int64_t n, int D, int k, bool rev, const uint64_t* Gold,
                              const JoinBuffers& b, bool tc, int64_t c0, int64_t c1, int mcap,
                              int* status, cudaStream_t s);
void finish_chunk(int64_t n, int k, uint64_t* Gnew, const JoinBuffers& b, double offers, int* status,
                  cudaStream_t s);

// KNNG_JOIN_SCREEN=1: with a 16-bit copy that is not exact, the join screens
// pairs on the tensor cores and computes canonical distances only for those
// the screen cannot exclude (k5_join_tc_cert) instead of running the FP32 join.
// The screen runs on request (KNNG_JOIN_SCREEN=1): on every measured float
// workload the FP32 join was faster (unit-sphere D = 96: 934 against 730 ms;
// GIST-like D = 960: 434 against 285 ms), its canonical distances of the
// surviving pairs (a thread per pair over two FP32 rows) costing more than the
// pairs it saves.
bool join_screen(int D) {
    (void)D;
    const char* e = getenv("KNNG_JOIN_SCREEN");
    return e && e[0] == '1';
}

// Chunks are sized from `est` (offers per node, measured on the previous
// chunk), but never below nodes_per_chunk, which fits the offer buffer even
// when every member pair offers both ways.  After each join the offer
// counter is read back; on an overflow the flag is cleared and the join
// re-runs on a smaller chunk (no target list has been touched yet).  `tc`:
// the tensor-core join does the work.
// `Gbase`, when given, is the list Gnew starts from and Gold only the
// members' view (the sampled round); thresholds come from Gold either way.
void join_round(const float* X, int64_t n, int D, int k, bool rev, const uint64_t* Gold, uint64_t* Gnew,
                const JoinBuffers& b, bool tc, int64_t count, int64_t nodes_per_chunk, double& est, int* status,
                cudaStream_t s, const uint64_t* Gbase = nullptr) {
    cudaMemcpyAsync(Gnew, Gbase ? Gbase : Gold, sizeof(uint64_t) * n * k, cudaMemcpyDeviceToDevice, s);
    const int mcap = ((rev ? 2 * k : k) + 3) & ~3;
    const double m_max = rev ? 2.0 * k : (double)k;
    // the 32-bit offer counter must not wrap, even in the worst case
    const int64_t wrap_nodes = (int64_t)(4294967295.0 / std::max(1.0, m_max * (m_max - 1)));
    if (b.capture) {  // no host reads: worst-case chunks over every position
        for (int64_t c0 = 0; c0 < count; c0 += nodes_per_chunk) {
            const int64_t c1 = std::min(count, c0 + nodes_per_chunk);
            launch_join_chunk(X, n, D, k, rev, Gold, b, tc, c0, c1, mcap, status, s);
            finish_chunk(n, k, Gnew, b, 0.0, status, s);
        }
        return;
    }
    for (int64_t c0 = 0, c1 = 0; c0 < count; c0 = c1) {
        int64_t want = (int64_t)((double)b.cap / std::max(est, 1.0));
        want = std::max(nodes_per_chunk, std::min(want, wrap_nodes));
        c1 = std::min(count, c0 + want);
        uint32_t offers = 0;
        for (;;) {
            const char* who = launch_join_chunk(X, n, D, k, rev, Gold, b, tc, c0, c1, mcap, status, s);
            int st = 0;
            cudaMemcpyAsync(&offers, b.counter, sizeof offers, cudaMemcpyDeviceToHost, s);
            cudaMemcpyAsync(&st, status, sizeof st, cudaMemcpyDeviceToHost, s);
            cudaStreamSynchronize(s);
            est = std::max((double)offers / (double)(c1 - c0), 1.0);
            // a chunk of nodes_per_chunk nodes cannot overflow; should it all
            // the same, the flag stays and the call reports it
            if ((int64_t)offers <= b.cap || c1 - c0 <= nodes_per_chunk) {
                record_bytes(who, std::min<double>(offers, (double)b.cap) * 12.0);  // offers written (id + key)
                break;
            }
            st &= ~kStatusOverflow;
            cudaMemcpyAsync(status, &st, sizeof st, cudaMemcpyHostToDevice, s);
            cudaStreamSynchronize(s);
            c1 = c0 + std::max(nodes_per_chunk, (int64_t)((double)(c1 - c0) * (double)b.cap / offers * 0.9));
            record_items("k5_join_retry", 1.0);
        }
        finish_chunk(n, k, Gnew, b, (double)offers, status, s);
    }
}

// The join of the chunk [c0, c1); returns the name of the kernel that ran.
const char* launch_join_chunk(const float* X, int64_t n, int D, int k, bool rev, const uint64_t* Gold,
                              const JoinBuffers& b, bool tc, int64_t c0, int64_t c1, int mcap,
                              int* status, cudaStream_t s) {
    {
        cudaMemsetAsync(b.pcnt, 0, sizeof(int32_t) * (n + 1), s);
        cudaMemsetAsync(b.pcur, 0, sizeof(int32_t) * n, s);
        cudaMemsetAsync(b.counter, 0, sizeof(uint32_t), s);
        if (tc && launch_join_tc(b.Xq, D, b.qnrm, k, rev, Gold, b.R, c0, c1, b, status, b.notexact, b.bf16, s))
            return "k5_join_tc";
        // capture: the tensor-core join returns at once on the device unless
        // the copy is exact, and the FP32 join below returns at once if it is
        const bool tc_dev = b.capture && b.lp &&
                            launch_join_tc(b.Xq, D, b.qnrm, k, rev, Gold, b.R, c0, c1, b, status, b.notexact,
                                           b.bf16, s);
        // not exact: the tensor cores screen the pairs and canonical distances
        // decide (on request).  In a capture the screening join returns at
        // once on the device when the copy is exact (the exact join above has
        // run), so no FP32 join is needed
        if ((!tc || b.capture) && b.lp && join_screen(D) &&
            launch_join_tc(b.Xq, D, b.qnrm, k, rev, Gold, b.R, c0, c1, b, status, b.notexact, b.bf16, s, true, X))
            return "k5_join_tc_cert";
        {
            const double m = rev ? 2.0 * k : (double)k;
            const bool lids = b.leafid != nullptr && b.npass > 0;
            const J2Layout L2 = j2_layout(D, mcap, lids);
            // With reverse lists a mutual neighbour is one member: slots of
            // three quarters of 2k when that packs more nodes into a CTA, the
            // nodes that overflow joined after them with full slots (their
            // count read on the device)
            const int small = (mcap * 3 / 4 + 3) & ~3;
            const bool packed = rev && b.ovf_list && b.ovf_count && small >= 4 &&
                                j2_layout(D, small, lids).G > L2.G;
            LaunchScope ls("k5_join", s, (double)(c1 - c0) * (m * D * 4.0 + 2 * k * 8.0 + m * 8.0),
                           (double)(c1 - c0) * m * (m - 1) / 2 * 3.0 * D, packed ? 2 : 1);
            auto cta_launch = [&](int mc, const int32_t* lst, const int32_t* cnt_dev, int64_t n0, int64_t n1,
                                  bool ovf) {
                const J2Layout Lc = j2_layout(D, mc, lids);
                allow_smem(k5_join_cta);
                const int per_sm = (int)std::min<size_t>(1024 / kJ2Threads, (227 * 1024) / (Lc.total + 1024));
                const int64_t groups = (n1 - n0 + Lc.G - 1) / Lc.G;
                const int grid2 = (int)std::max<int64_t>(1, std::min<int64_t>(groups, (int64_t)152 * per_sm));
                k5_join_cta<<<grid2, kJ2Threads, Lc.total, s>>>(
                    X, D, k, rev ? 1 : 0, mc, Gold, b.R, lst, b.fnew, b.rnew, n0, n1, b.counter, b.cap, b.ptgt,
                    b.pkey, b.pcnt, status, tc_dev ? b.notexact : nullptr, cnt_dev, lids ? b.leafid : nullptr,
                    b.npass, ovf ? b.ovf_list : nullptr, ovf ? b.ovf_count : nullptr);
            };
            if (packed) {
                cudaMemsetAsync(b.ovf_count, 0, sizeof(int32_t), s);
                cta_launch(small, b.list, b.count_dev, c0, c1, true);
                cta_launch(mcap, b.ovf_list, b.ovf_count, 0, c1 - c0, false);
            } else {
                cta_launch(mcap, b.list, b.count_dev, c0, c1, false);
            }
        }
    }
    return "k5_join";
}

// Groups the chunk's offers by target and merges them into Gnew.
void finish_chunk(int64_t n, int k, uint64_t* Gnew, const JoinBuffers& b, double offers, int* status,
                  cudaStream_t s) {
    {
        launch_scan(b.pcnt, b.poff, n, b.scan_tmp, s);
        {
            // per offer: target and key read, its target's offset, the key written
            LaunchScope ls("k5_scatter", s, offers * 24.0, 0);
            k5_scatter<<<152 * 16, 256, 0, s>>>(b.ptgt, b.pkey, b.counter, b.cap, b.poff, b.pcur, b.grouped,
                                                status, b.offers_total);
        }
        {
            // offsets, every grouped offer, and the list of each target reached
            // (at most min(n, offers) of them) read and written
            LaunchScope ls("k4_merge", s, n * 4.0 + offers * 8.0 + std::min((double)n, offers) * 16.0 * k, 0);
            const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
            if (k > 32)
                k4_merge<2><<<grid, 256, 0, s>>>(Gnew, b.grouped, b.poff, n, k, status);
            else
                k4_merge<1><<<grid, 256, 0, s>>>(Gnew, b.grouped, b.poff, n, k, status);
        }
    }
}

}  // namespace

void run_refine(const float* X, int64_t n, int D, int k, bool rev, uint64_t*& G, uint64_t*& G2,
                const JoinBuffers& jb, int64_t nodes_per_chunk, int rounds, int* status, cudaStream_t s) {
    JoinBuffers b = jb;
    // offers per node of the first round's chunks: a guess (a quarter of the
    // worst case); then what the previous chunk measured
    const double m_max = rev ? 2.0 * k : (double)k;
    double est = m_max * (m_max - 1) / 4;
    // the tensor-core join runs when the 16-bit copy is exact for this input
    bool tc = false;
    if (b.lp && !b.capture) {
        int f = 0;
        cudaMemcpyAsync(&f, b.notexact, sizeof f, cudaMemcpyDeviceToHost, s);
        cudaStreamSynchronize(s);
        tc = (f & 1) == 0 && !((f & 2) && (f & 4));
    }
    for (int r = 0; r < rounds; ++r) {
        if (rev) launch_reverse_lists(G, n, k, b, s);  // into b.R; b.R2 keeps the previous round's
        b.list = b.order;  // every node (in the last tree pass's leaf order when it is known)
        b.fnew = b.rnew = nullptr;
        b.count_dev = nullptr;
        int64_t count = n;
        if (r > 0) {
            // G2 still holds the previous round's G_old
            cudaMemsetAsync(b.nactive, 0, sizeof(int32_t), s);
            {
                LaunchScope ls("k6_flags", s, n * k * 8.0 * (rev ? 4.0 : 2.0) + n * 20.0, 0);
                const int grid = (int)((n + kFlagWarps - 1) / kFlagWarps);
                // with an order, k6_active lists the nodes after the flags
                int32_t* act = b.order ? nullptr : b.active;
                if (k > 32)
                    k6_flags<2><<<grid, 32 * kFlagWarps, 0, s>>>(G, rev ? b.R : nullptr, G2, rev ? b.R2 : nullptr,
                                                                 n, k, b.fnew_buf, b.rnew_buf, act, b.nactive);
                else
                    k6_flags<1><<<grid, 32 * kFlagWarps, 0, s>>>(G, rev ? b.R : nullptr, G2, rev ? b.R2 : nullptr,
                                                                 n, k, b.fnew_buf, b.rnew_buf, act, b.nactive);
            }
            if (b.order) {
                // the order (4 B), the flags of each node (8 or 16 B), the list written (4 B)
                LaunchScope ls("k6_active", s, n * (rev ? 24.0 : 16.0), 0);
                k6_active<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(b.order, b.fnew_buf, rev ? b.rnew_buf : nullptr,
                                                                     n, b.active, b.nactive);
            }
            if (b.capture) {
                b.count_dev = b.nactive;  // the kernels read how many nodes are listed
            } else {
                int32_t h = 0;
                cudaMemcpyAsync(&h, b.nactive, sizeof h, cudaMemcpyDeviceToHost, s);
                cudaStreamSynchronize(s);
                count = h;
                record_items("k6_flags", (double)count);
            }
            b.list = b.active;
            b.fnew = b.fnew_buf;
            b.rnew = rev ? b.rnew_buf : nullptr;
        }
        join_round(X, n, D, k, rev, G, G2, b, tc, count, nodes_per_chunk, est, status, s);
        std::swap(G, G2);
        if (rev) std::swap(b.R, b.R2);
    }
}

void run_refine_sampled(const float* X, int64_t n, int D, int k, uint64_t*& G, uint64_t*& G2, const JoinBuffers& jb,
                        int64_t nodes_per_chunk, int rounds, int ms, uint64_t seed, int* status, cudaStream_t s) {
    JoinBuffers b = jb;
    double est = 2.0 * k * (2.0 * k - 1) / 4;
    bool tc = false;
    if (b.lp) {
        int f = 0;
        cudaMemcpyAsync(&f, b.notexact, sizeof f, cudaMemcpyDeviceToHost, s);
        cudaStreamSynchronize(s);
        tc = (f & 1) == 0 && !((f & 2) && (f & 4));
    }
    cudaMemsetAsync(b.flags, 0xFF, sizeof(uint64_t) * n, s);  // every entry new before the first round
    for (int r = 0; r < rounds; ++r) {
        const uint64_t h0 = splitmix64(seed ^ (uint64_t)(uint32_t)r);
        // member view in R2, sampled-new mask in fnew_buf, reverse samples in R
        launch_sampled_prepare(G, b.flags, n, k, ms, h0, b.R2, b.fnew_buf, b.flags_post, b.deg, b.roff, b.cur,
                               b.scan_tmp, b.rbuf, b.R, b.rnew_buf, s);
        b.list = b.order;  // every node (in the last tree pass's leaf order when it is known)
        b.count_dev = nullptr;
        b.fnew = b.fnew_buf;
        b.rnew = b.rnew_buf;
        join_round(X, n, D, k, true, b.R2, G2, b, tc, n, nodes_per_chunk, est, status, s, G);
        launch_sampled_flags(G2, G, b.flags_post, n, k, b.flags, nullptr, s);
        std::swap(G, G2);
    }
}

}  // namespace knng
