// select.cu -- K1: the cut of segments too large for a warp group's sort and
// small enough for one cluster: select the key of rank floor(m/2) and, on a
// level's last cut, partition, in one launch.
//
// A cluster of 1, 2, 4 or 8 CTAs takes one segment.  Every thread keeps up to
// kSelPer projections in registers, so S is read once; the histograms of the
// 8-bit digits are added up through distributed shared memory, and as soon as
// at most 32 keys match they are ranked by counting.  (The passes of split.cu
// read S again for every digit and meet in global memory between launches:
// three digit launches and one for ties, about 10 us each however small the
// segment, and two more for the partition.)
//
// Bound by latency: a cluster synchronisation and a block's two for each of
// two to four digits.  1,024 threads with 16 values each: a recorded build of
// 100,000 x 128 4.06 -> 3.69 ms, 10,000 x 32 0.92 -> 0.83, 1M x 128 33.9 -> 33.1;
// 512 threads with 32 values 3.82, 0.84 and 33.2.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace knng {

namespace {

constexpr int kSelThreads = 1024, kSelPer = 16, kSelShare = kSelThreads * kSelPer;

// Exclusive scan of one int per thread over the CTA; *total gets the sum.
__device__ __forceinline__ int sel_excl_scan(int v, int* warp_tot, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_tot[lane] = w;
    }
    __syncthreads();
    const int before = warp ? warp_tot[warp - 1] : 0;
    *total = warp_tot[31];
    __syncthreads();
    return before + x - v;
}

template <int C>
__global__ void __launch_bounds__(kSelThreads, 1) k1_select_cluster(const float* __restrict__ S,
                                                                   const int32_t* __restrict__ seg_off,
                                                                   const int32_t* __restrict__ seg_tile0,
                                                                   int pos_bits, uint64_t* __restrict__ thr,
                                                                   const int32_t* __restrict__ perm_in,
                                                                   int32_t* __restrict__ perm_out,
                                                                   int* __restrict__ status) {
    __shared__ int hist[2][256], warp_tot[32], sh[4], nfew, ccount[8], tie_pos;
    __shared__ __align__(16) int all[256];
    __shared__ uint64_t few[32];
    const int seg = (int)(blockIdx.x / C), rank = (int)(blockIdx.x % C);
    if (seg_tile0[seg + 1] == seg_tile0[seg]) return;  // a finished tree's leaf (the whole cluster)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int a = seg_off[seg], m = seg_off[seg + 1] - a, K = m / 2;
    const int q = (m + C - 1) / C, p0 = min(m, rank * q), ql = min(m, p0 + q) - p0;
    if (q > kSelShare) {  // the plan sized the cluster from the level's largest segment
        if (tid == 0) atomicOr(status, kStatusInternal);
        return;
    }
    auto sync = [&] {
        if (C > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    auto peer = [&](auto* p, int r) {
        if (C > 1) return cg::this_cluster().map_shared_rank(p, r);
        return p;
    };
    uint32_t u[kSelPer];  // position p0 + tid + kSelThreads i; past the share: not used
#pragma unroll
    for (int i = 0; i < kSelPer; ++i) {
        const int e = tid + kSelThreads * i;
        u[i] = e < ql ? ord32(S[a + p0 + e]) : 0u;
    }
    if (tid == 0) nfew = 0;
    sync();  // every CTA of the cluster runs, and rank 0's counter is set
    uint32_t v = 0;
    int krem = K, match = m, sft = 32, turn = 0;
    while (sft > 0 && match > 32) {
        sft -= 8;
        int* h = hist[turn & 1];  // a peer may still read the other one
        ++turn;
        if (tid < 256) h[tid] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kSelPer; ++i)
            if (tid + kSelThreads * i < ql && (sft == 24 || (u[i] >> (sft + 8)) == (v >> (sft + 8))))
                atomicAdd(h + ((u[i] >> sft) & 255), 1);
        sync();
        if (tid < 256) {
            int c = 0;
#pragma unroll
            for (int r = 0; r < C; ++r) c += peer(h, r)[tid];
            all[tid] = c;
        }
        __syncthreads();
        if (warp == 0) {  // lane l: bins 8 l .. 8 l + 7
            const int4 h0 = reinterpret_cast<const int4*>(all)[2 * lane];
            const int4 h1 = reinterpret_cast<const int4*>(all)[2 * lane + 1];
            const int c[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
            int sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) sum += c[j];
            int x = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            int run = x - sum;
            if (run <= krem && krem < x) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (run <= krem && krem < run + c[j]) {
                        sh[0] = 8 * lane + j;
                        sh[1] = run;
                        sh[2] = c[j];
                    }
                    run += c[j];
                }
            }
        }
        __syncthreads();
        v |= (uint32_t)sh[0] << sft;
        krem -= sh[1];
        match = sh[2];
    }
    int tpos = 0;  // left: value < v, or value v before this position
    if (match <= 32) {
        int* n0 = peer(&nfew, 0);
        uint64_t* f0 = peer(few, 0);
#pragma unroll
        for (int i = 0; i < kSelPer; ++i) {
            const int e = tid + kSelThreads * i;
            if (e < ql && (sft == 32 || (u[i] >> sft) == (v >> sft)))
                f0[atomicAdd(n0, 1)] = ((uint64_t)u[i] << 32) | (uint32_t)(p0 + e);
        }
        sync();
        const uint64_t mine = lane < match ? f0[lane] : ~0ull;
        int below = 0;
        for (int j = 0; j < match; ++j) below += shfl64(mine, j) < mine;
        const int src = __ffs(__ballot_sync(0xffffffffu, lane < match && below == krem)) - 1;
        const uint64_t key = shfl64(mine, src);
        v = (uint32_t)(key >> 32);
        tpos = (int)(uint32_t)key;
    } else if (krem > 0) {  // more than 32 equal values: the krem-th of them by position
        int c = 0, total;
#pragma unroll
        for (int i = 0; i < kSelPer; ++i) c += tid + kSelThreads * i < ql && u[i] == v;
        sel_excl_scan(c, warp_tot, &total);
        if (tid < C) peer(ccount, tid)[rank] = total;
        sync();
        int before = 0;
        for (int r = 0; r < rank; ++r) before += ccount[r];
        if (before <= krem && krem < before + total) {  // this CTA holds it (uniform)
            for (int i = 0; i < kSelPer; ++i) {
                const int e = tid + kSelThreads * i;
                uint32_t ui = 0;
#pragma unroll
                for (int z = 0; z < kSelPer; ++z) ui = z == i ? u[z] : ui;
                const int tied = e < ql && ui == v;
                int t;
                const int at = before + sel_excl_scan(tied, warp_tot, &t);
                if (tied && at == krem)
                    for (int r = 0; r < C; ++r) *peer(&tie_pos, r) = p0 + e;
                before += t;
            }
        }
        sync();
        tpos = tie_pos;
    }
    if (perm_out == nullptr) {
        if (rank == 0 && tid == 0) thr[seg] = ((uint64_t)v << pos_bits) | (uint32_t)tpos;
        sync();  // no CTA leaves while a peer may read its shared memory
        return;
    }
    // the cut: left positions first, each side in position order
    unsigned left = 0;
#pragma unroll
    for (int i = 0; i < kSelPer; ++i) {
        const int e = tid + kSelThreads * i;
        left |= (e < ql && (u[i] < v || (u[i] == v && p0 + e < tpos))) ? 1u << i : 0u;
    }
    int total;
    sel_excl_scan(__popc(left), warp_tot, &total);
    sync();  // the counts of the ties are read
    if (tid < C) peer(ccount, tid)[rank] = total;
    sync();
    int before = 0;
    for (int r = 0; r < rank; ++r) before += ccount[r];
    for (int i = 0; kSelThreads * i < ql; ++i) {
        const int e = tid + kSelThreads * i;
        const int isl = (left >> i) & 1u;
        int t;
        const int lb = before + sel_excl_scan(isl, warp_tot, &t);
        if (e < ql) {
            const int np = isl ? lb : K + (p0 + e - lb);
            if ((isl ? np < K : np < m) && np >= 0)
                perm_out[a + np] = perm_in[a + p0 + e];
            else
                atomicOr(status, kStatusInternal);
        }
        before += t;
    }
}

template <int C>
bool launch_c(const LevelPlan& lp, const float* S, uint64_t* thr, const int32_t* perm_in, int32_t* perm_out,
              int* status, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)lp.nseg * C);
    cfg.blockDim = dim3(kSelThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k1_select_cluster<C>, S, lp.seg_off, lp.seg_tile0, lp.pos_bits, thr, perm_in,
                              perm_out, status) == cudaSuccess;
}

}  // namespace

static_assert(8 * kSelShare == kClusterSelectMax, "the largest cluster's segment");

bool launch_select_cluster(const LevelPlan& lp, const float* S, uint64_t* thr, const int32_t* perm_in,
                           int32_t* perm_out, int* status, cudaStream_t s) {
    LaunchScope ls("k1_select", s, lp.n * 4.0 + (perm_out ? lp.n * 8.0 : 0.0), 0);
    if (lp.max_m <= kSelShare) return launch_c<1>(lp, S, thr, perm_in, perm_out, status, s);
    if (lp.max_m <= 2 * kSelShare) return launch_c<2>(lp, S, thr, perm_in, perm_out, status, s);
    if (lp.max_m <= 4 * kSelShare) return launch_c<4>(lp, S, thr, perm_in, perm_out, status, s);
    return launch_c<8>(lp, S, thr, perm_in, perm_out, status, s);
}

}  // namespace knng
