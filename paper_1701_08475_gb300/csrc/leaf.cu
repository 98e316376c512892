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
// Bound by its FP32 instructions and the selection's.  Leaves whose dims fit
// at once are held as interleaved pairs of points and computed with paired
// instructions (400,000 points in three passes: 64 dims at leaves of up to 64
// 1.38 -> 1.09 ms, 96 at 64 1.58 -> 1.33, 128 at 128 3.63 -> 3.30, 64 at 256
// 3.04 -> 2.92).  With more dims, equal chunks come by cp.async and alternate
// between two buffers.  Before that (a division and a 4-byte load per value,
// one buffer, the last chunk padded to the first one's size) three passes over
// 104,000 x 960 took 23.3 ms at leaves of up to 256 and 7.6 at 128, now 7.8 and
// 3.9; 400,000 x 96 at 256 9.0, now 4.1, and at 128 3.7, now 3.3.
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
// than it must) and padded stride.  One chunk: pair rows, which hold points 2 p
// and 2 p + 1 of the leaf interleaved dim by dim for paired FP32 instructions.
// Several chunks alternate between two buffers of plain rows: the next one's
// 16-byte copies are in flight while one is used (copies that interleave move 4
// bytes each, and cost more than the pairing saves: 104,000 x 960 at leaves of
// 256 points 8.0 against 10.0 ms for three passes).  stride / 4 is odd: 16-byte
// reads of consecutive rows are free of conflicts.
__host__ __device__ inline void leaf_chunk(int D, int MC, int* dch, int* nch, int* stride) {
    const int d4 = (D + 3) & ~3;
    const int cap = (72 * 1024 / (MC * 4) - 4) & ~3, half = (36 * 1024 / (MC * 4) - 4) & ~3;
    *nch = d4 <= cap ? 1 : (d4 + half - 1) / half;
    const int c = ((d4 + *nch - 1) / *nch + 3) & ~3;
    *dch = c;
    *stride = *nch == 1 ? 2 * c + 4 : ((c / 4) & 1) ? c : c + 4;
}

// NB: CTAs per SM the registers must allow.  PAIR: one chunk.
template <int MC, int NSG, int NB, bool PAIR>
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
    float* xs = reinterpret_cast<float*>(smem4);           // [MC / 2][stride], or [2][MC][stride]
    float* dt = xs + (PAIR ? MC / 2 : 2 * MC) * stride;     // [RB][MC + 1]
    int32_t* ids = reinterpret_cast<int32_t*>(dt + C::RB * (MC + 1));  // [MC]
    uint64_t* wscratch = reinterpret_cast<uint64_t*>(ids + MC) + (threadIdx.x >> 5) * 32;  // 32 keys per warp

    const int leaf = blockIdx.x;
    const int a = leaf_off[leaf];
    const int m = leaf_off[leaf + 1] - a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = tid % C::RG, cg = tid / C::RG;
    for (int r = tid; r < MC; r += C::NT) ids[r] = r < m ? perm[a + r] : 0;
    __syncthreads();

    // chunk c's dims of every row (zeros past the leaf and past D)
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    auto load_chunk = [&](int c) {
        const int d0 = c * dch, dl = min(dch, D - d0);
        float* buf = xs + (c & 1) * MC * stride;  // one chunk: xs
        if (PAIR && vec) {
            const int q4 = dch / 4;
            for (int e = tid; e < (MC / 2) * q4; e += C::NT) {
                const int p = e / q4, c4 = e - p * q4;
                float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
                if (4 * c4 < dl) {
                    if (2 * p < m) u = __ldg(reinterpret_cast<const float4*>(X + (int64_t)ids[2 * p] * D) + c4);
                    if (2 * p + 1 < m) v = __ldg(reinterpret_cast<const float4*>(X + (int64_t)ids[2 * p + 1] * D) + c4);
                }
                store_pairs(buf + p * stride + 8 * c4, u, v, (c4 >> 2) & 1);
            }
        } else if (vec) {
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
                buf[PAIR ? (r >> 1) * stride + 2 * dd + (r & 1) : r * stride + dd] = v;
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (PAIR) {
        load_chunk(0);
        __syncthreads();
    }

    for (int rb = 0; rb * C::RB < m; ++rb) {
        // the thread's 4 x 8 distances.  PAIR: rows 2 (rg + h RG) + {0, 1} and
        // columns 2 (cg + w CG) + {0, 1}, as the sums of (0, 0), (1, 1) and of
        // (1, 0), (0, 1).  Else rows rg + i RG and columns cg + j CG.
        uint64_t same[2][4], cross[2][4];
        float acc[4][8];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int w = 0; w < 4; ++w) same[h][w] = cross[h][w] = 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        if (!PAIR) load_chunk(0);
        for (int c = 0; c < (PAIR ? 1 : nch); ++c) {
            if (!PAIR) {
                if (c + 1 < nch) {
                    load_chunk(c + 1);
                    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                } else {
                    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                }
                __syncthreads();
            }
            if constexpr (PAIR) {
                const float* rp = xs + (rb * (C::RB / 2) + rg) * stride;
                const float* cp = xs + cg * stride;
                for (int dq = 0; dq < 2 * dch; dq += 8) {  // 4 dims
                    ulonglong2 r[2][2], x[2][2];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            r[h][p] = *reinterpret_cast<const ulonglong2*>(rp + h * C::RG * stride + dq + 4 * p);
                            x[h][p].x = swap_pair(r[h][p].x);
                            x[h][p].y = swap_pair(r[h][p].y);
                        }
#pragma unroll
                    for (int w = 0; w < 4; ++w)
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(cp + w * C::CG * stride + dq + 4 * p);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                same[h][w] = add_square(r[h][p].x, v.x, same[h][w]);
                                cross[h][w] = add_square(x[h][p].x, v.x, cross[h][w]);
                                same[h][w] = add_square(r[h][p].y, v.y, same[h][w]);
                                cross[h][w] = add_square(x[h][p].y, v.y, cross[h][w]);
                            }
                        }
                }
            } else {
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
            }
            if (!PAIR) __syncthreads();  // the buffer is refilled
        }
        __syncthreads();  // previous selection done with dt
        if constexpr (PAIR) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    float* at = dt + 2 * (rg + h * C::RG) * (MC + 1) + 2 * (cg + w * C::CG);
                    at[0] = __uint_as_float((uint32_t)same[h][w]);
                    at[MC + 2] = __uint_as_float((uint32_t)(same[h][w] >> 32));
                    at[MC + 1] = __uint_as_float((uint32_t)cross[h][w]);
                    at[1] = __uint_as_float((uint32_t)(cross[h][w] >> 32));
                }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) dt[(rg + i * C::RG) * (MC + 1) + cg + j * C::CG] = acc[i][j];
        }
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
    const size_t smem = (size_t)(nch > 1 ? 2 * MC : MC / 2) * stride * 4 + (size_t)C::RB * (MC + 1) * 4 + MC * 4 + (C::NT / 32) * 32 * 8;
    auto kernel = nch == 1 ? k2_leaf_fp32<MC, NSG, NB, true> : k2_leaf_fp32<MC, NSG, NB, false>;
    allow_smem(kernel);
    kernel<<<nleaf, C::NT, smem, s>>>(X, D, perm, leaf_off, k, G, status, skip);
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
