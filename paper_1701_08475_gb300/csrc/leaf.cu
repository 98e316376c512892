// leaf.cu -- K2f: exhaustive comparison inside each cluster (Alg. 1: for
// every pair <i, j>, i != j, of a cluster, update G[i] and G[j] with
// d(x_i, x_j)), in canonical FP32, fused with the merge into the graph.
//
// One CTA per leaf (m <= MC points).  The leaf's rows sit in shared memory
// (DCH dims at a time); each thread accumulates a 4 x 8 block of pairs, dims
// ascending with fmaf, so every distance has the canonical bits.  A row
// block of distances goes to shared memory, and one warp per row selects the
// row's k best of (its G row) + (the leaf) with duplicates merged.  No
// distance matrix reaches HBM; G is updated in place (a point lives in one
// leaf per pass).
//
// Bound by its FP32 instructions and the selection's.  The rows come by
// cp.async; with more dims than fit at once, equal chunks alternate between
// two buffers.  Before that (a division and a 4-byte load per value, one
// buffer, the last chunk padded to the first one's size) three passes over
// 104,000 x 960 took 23.3 ms at leaves of up to 256 and 7.6 at 128, now 8.0 and
// 3.9; 400,000 x 96 at 256 9.0, now 4.2, and at 128 3.7, now 3.5.
#include "common.cuh"
#include "kernels.h"

namespace knng {

namespace {

template <int MC>
struct LeafCfg {
    static constexpr int RB = (MC < 8192 / MC) ? MC : 8192 / MC;  // rows per block
    static constexpr int NT = RB * MC / 32;                        // threads
    static constexpr int RG = RB / 4;                              // row groups
    static constexpr int CG = MC / 8;                              // col groups
};

// Dims per chunk, chunks (of equal size: the last one computes no more zeros
// than it must) and padded stride (stride / 4 odd: conflict-free float4 rows).
// Several chunks alternate between two buffers: the next one's copies are in
// flight while one is used.
__host__ __device__ inline void leaf_chunk(int D, int MC, int* dch, int* nch, int* stride) {
    const int d4 = (D + 3) & ~3;
    const int cap = (72 * 1024 / (MC * 4) - 4) & ~3, half = (36 * 1024 / (MC * 4) - 4) & ~3;
    *nch = d4 <= cap ? 1 : (d4 + half - 1) / half;
    const int c = ((d4 + *nch - 1) / *nch + 3) & ~3;
    *dch = c;
    *stride = ((c / 4) & 1) ? c : c + 4;
}

// NB: CTAs per SM the registers must allow.
template <int MC, int NSG, int NB>
__global__ void __launch_bounds__(LeafCfg<MC>::NT, NB) k2_leaf_fp32(const float* __restrict__ X, int D,
                                                                 const int32_t* __restrict__ perm,
                                                                 const int32_t* __restrict__ leaf_off, int k,
                                                                 uint64_t* __restrict__ G,
                                                                 const int* __restrict__ status,
                                                                 const int* __restrict__ skip_if_exact) {
    using C = LeafCfg<MC>;
    if (*status & kStatusStop) return;  // ids or offsets failed their check
    if (skip_if_exact) {  // the tensor-core leaf did this pass
        const int f = *skip_if_exact;
        if ((f & 1) == 0 && !((f & 2) && (f & 4))) return;
    }
    constexpr int NS = MC / 32 + NSG;
    extern __shared__ float4 smem4[];
    int dch, nch, stride;
    leaf_chunk(D, MC, &dch, &nch, &stride);
    float* xs = reinterpret_cast<float*>(smem4);          // [1 or 2][MC][stride]
    float* dt = xs + (nch > 1 ? 2 : 1) * MC * stride;      // [RB][MC + 1]
    int32_t* ids = reinterpret_cast<int32_t*>(dt + C::RB * (MC + 1));  // [MC]
    uint64_t* wscratch = reinterpret_cast<uint64_t*>(ids + MC) + (threadIdx.x >> 5) * 32;  // 32 keys per warp

    const int leaf = blockIdx.x;
    const int a = leaf_off[leaf];
    const int m = leaf_off[leaf + 1] - a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = tid % C::RG, cg = tid / C::RG;
    for (int r = tid; r < MC; r += C::NT) ids[r] = r < m ? perm[a + r] : 0;
    __syncthreads();

    // copies of chunk c's dims of every row into buffer c & 1 (zeros past the
    // leaf and past D)
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    auto load_chunk = [&](int c) {
        const int d0 = c * dch, dl = min(dch, D - d0);
        float* buf = xs + (c & 1) * MC * stride;
        if (vec) {
            const int q4 = dch / 4;
            // consecutive threads take a row's 16-byte pieces; the row moves on
            // by C::NT / q4 rows and a remainder, without a division per piece
            int r = tid / q4, p = tid - r * q4;
            const int dr = C::NT / q4, dp = C::NT - dr * q4;
            while (r < MC) {
                float* dst = buf + r * stride + 4 * p;
                if (r < m && 4 * p < dl)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(dst)),
                                 "l"(X + (int64_t)ids[r] * D + d0 + 4 * p)
                                 : "memory");
                else
                    *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
                r += dr;
                p += dp;
                if (p >= q4) {
                    p -= q4;
                    ++r;
                }
            }
        } else {
            for (int e = tid; e < MC * dch; e += C::NT) {
                const int r = e / dch, dd = e - r * dch;
                float v = 0.f;
                if (r < m && dd < dl) v = __ldg(X + (int64_t)ids[r] * D + d0 + dd);
                buf[r * stride + dd] = v;
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (nch == 1) {
        load_chunk(0);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
    }

    for (int rb = 0; rb * C::RB < m; ++rb) {
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        if (nch > 1) load_chunk(0);
        for (int c = 0; c < nch; ++c) {
            if (nch > 1) {
                if (c + 1 < nch) {
                    load_chunk(c + 1);
                    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                } else {
                    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                }
                __syncthreads();
            }
            const float* rp = xs + (c & 1) * MC * stride + (rb * C::RB + rg) * stride;
            const float* cp = xs + (c & 1) * MC * stride + cg * stride;
            for (int dq = 0; dq < dch; dq += 4) {
                float4 rv[4], cv[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) rv[i] = *reinterpret_cast<const float4*>(rp + i * C::RG * stride + dq);
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = *reinterpret_cast<const float4*>(cp + j * C::CG * stride + dq);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float t = __fsub_rn(rv[i].x, cv[j].x);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(rv[i].y, cv[j].y);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(rv[i].z, cv[j].z);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(rv[i].w, cv[j].w);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                    }
            }
            if (nch > 1) __syncthreads();  // the buffer is refilled
        }
        __syncthreads();  // previous selection done with dt
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) dt[(rg + i * C::RG) * (MC + 1) + cg + j * C::CG] = acc[i][j];
        __syncthreads();
        // one warp per row: k best of G[i] + leaf candidates
        for (int r = warp; r < C::RB; r += C::NT / 32) {
            const int row = rb * C::RB + r;
            if (row >= m) break;
            const int gi = ids[row];
            uint64_t* grow = G + (int64_t)gi * k;
            uint64_t cand[NS];
#pragma unroll
            for (int s = 0; s < MC / 32; ++s) {
                const int c = lane + 32 * s;
                cand[s] = (c < m && c != row) ? make_key(dt[r * (MC + 1) + c], (uint32_t)ids[c]) : kEmptyKey;
            }
            if (NSG == 1) {
                // few candidates beat the row's k-th entry after the first pass
                uint64_t few[MC / 32], out;
                bool changed;
#pragma unroll
                for (int s = 0; s < MC / 32; ++s) few[s] = cand[s];
                const uint64_t cur = lane < k ? grow[lane] : kEmptyKey;
                if (warp_merge_few<MC / 32>(few, cur, k, wscratch, out, changed)) {
                    if (changed && lane < k) grow[lane] = out;
                    continue;
                }
                // many survive (the first pass): the lanes' smallest first
#pragma unroll
                for (int s = 0; s < MC / 32; ++s) few[s] = cand[s];
                if (warp_merge_many<MC / 32>(few, cur, k, wscratch, out, changed)) {  // MC >= 64
                    if (changed && lane < k) grow[lane] = out;
                    continue;
                }
            }
#pragma unroll
            for (int s = 0; s < NSG; ++s) {
                const int e = lane + 32 * s;
                cand[MC / 32 + s] = e < k ? grow[e] : kEmptyKey;
            }
            sort_regs<NS>(cand);
            uint64_t out[NSG];
            warp_select_unique<NS, NSG>(cand, k, out);
#pragma unroll
            for (int s = 0; s < NSG; ++s) {
                const int e = lane + 32 * s;
                if (e < k) grow[e] = out[s];
            }
        }
    }
}

template <int MC, int NSG, int NB>
void launch_leaf_t(const float* X, int D, const int32_t* perm, const int32_t* leaf_off, int nleaf, int k,
                   uint64_t* G, const int* status, cudaStream_t s, const int* skip) {
    using C = LeafCfg<MC>;
    int dch, nch, stride;
    leaf_chunk(D, MC, &dch, &nch, &stride);
    const size_t smem = (size_t)(nch > 1 ? 2 : 1) * MC * stride * 4 + (size_t)C::RB * (MC + 1) * 4 + MC * 4 + (C::NT / 32) * 32 * 8;
    cudaFuncSetAttribute(k2_leaf_fp32<MC, NSG, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k2_leaf_fp32<MC, NSG, NB><<<nleaf, C::NT, smem, s>>>(X, D, perm, leaf_off, k, G, status, skip);
}

}  // namespace

void launch_leaf_fp32(const float* X, int D, const int32_t* perm, const int32_t* leaf_off, int nleaf,
                      int max_leaf, int k, uint64_t* G, const int* status, cudaStream_t s, const int* skip_if_exact) {
    // algorithmic work: every leaf row once, every ordered pair once
    const double mm = (double)max_leaf;
    LaunchScope ls("k2_leaf_fp32", s, (double)nleaf * mm * (D * 4.0 + 2 * 8.0 * k),
                   (double)nleaf * mm * (mm - 1) * 3.0 * D);
    const bool two = k > 32;
    if (max_leaf <= 64 && D <= 96) {
        // six CTAs of short leaves fit an SM when registers allow it (80 instead
        // of 122): 400,000 x 64 1.35 -> 1.20 ms for three passes; from 128 dims
        // on shared memory allows fewer and the registers are worth more (1.73
        // against 1.83 ms)
        if (two) launch_leaf_t<64, 2, 6>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
        else launch_leaf_t<64, 1, 6>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
    } else if (max_leaf <= 64) {
        if (two) launch_leaf_t<64, 2, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
        else launch_leaf_t<64, 1, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
    } else if (max_leaf <= 128) {
        if (two) launch_leaf_t<128, 2, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
        else launch_leaf_t<128, 1, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
    } else {
        if (two) launch_leaf_t<256, 2, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
        else launch_leaf_t<256, 1, 1>(X, D, perm, leaf_off, nleaf, k, G, status, s, skip_if_exact);
    }
}

}  // namespace knng
