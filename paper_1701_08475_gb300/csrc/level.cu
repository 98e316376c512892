// level.cu -- K1 for segments that fit the shared memory of one cluster: a
// whole level of the two-means tree in one launch.
//
// The sweep kernels of split.cu read every row of the level once per
// projection and again for the sums, about 2 (T + 1) launches and as many
// passes over the rows for T Lloyd iterations.  Here a cluster of 1, 2, 4 or 8
// CTAs takes one segment: its rows are read once and stay in shared memory
// (spread over the CTAs by position) for all iterations and the final cut.
// What crosses CTAs goes through distributed shared memory: every projection
// is stored to all CTAs (each then selects the cut for itself), each CTA's
// centroid sums go to the CTA that owns the dim, and its new w component goes
// to all.
//
// The projection is the canonical one (one thread per row, dims ascending,
// fmaf), the cut is by the (projection, position) key, and the sums are
// compensated FP32 (TwoSum) per warp, FP64 across warps, CTAs and iterations
// (integers: exact int64): split.cu's definitions, with the rows of a sum in
// another fixed order.  A warp adds up to a sixteenth of the CTA's rows before
// FP64 (68 of 32 dims, about 150 of 8; the sweeps 32): r rows leave the low part
// within r^2 2^-48 of their magnitudes' sum, 8e-11 at 150, against the 6e-8 of
// the mean's own rounding to FP32.
//
// Its own bound is latency: 3 synchronisations and about four short dependent
// phases per iteration, 8-15 us an iteration.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace knng {

namespace {

constexpr int kLvDims = 128;  // dims of one sums chunk: 4 per lane
constexpr int kLvSms = 152;
// Dynamic shared memory of a CTA: the block limit (227 KB), and what two CTAs
// may take of an SM's 228 KB, of which each CTA also costs 1 KB.  The kernel
// declares no static shared memory, so these are all of it.
constexpr size_t kLvOne = 227 * 1024, kLvTwo = 113 * 1024;

struct LvLayout {
    int C, q, nt;      // CTAs, rows per CTA, threads
    int stride;        // bytes per staged row
    int dcap;          // dims owned per CTA
    size_t S, ids, side, W, red, part, tot, misc, total;
};

// What a segment's cut needs besides: keys to rank by counting, the means'
// reciprocals, warps' scan totals, and values one thread gives to all.
struct LvMisc {
    uint64_t few[32];
    double inv[2];
    int warp_tot[16], sh[4];
};

// Bytes of a staged row: whole 16-byte pieces, an odd number of them (the
// 16-byte reads of 8 consecutive rows then cover all banks).
__host__ __device__ inline int lv_stride(int row_bytes) {
    const int p = (row_bytes + 15) / 16;
    return 16 * (p | 1);
}

__host__ __device__ inline LvLayout lv_layout(int D, int m, int row_bytes, int C) {
    LvLayout L;
    L.C = C;
    L.q = (m + C - 1) / C;
    const int nt = (L.q + 31) & ~31;
    L.nt = nt < 128 ? 128 : nt > 512 ? 512 : nt;
    L.stride = lv_stride(row_bytes);
    L.dcap = (D + C - 1) / C;
    auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
    L.S = up((size_t)L.q * L.stride);                     // rows first
    L.ids = L.S + up((size_t)m * 4);                      // [m] projections (ord32)
    L.side = L.ids + up((size_t)L.q * 4);
    L.W = L.side + up((size_t)L.q);
    L.red = L.W + up((size_t)((D + 15) & ~15) * 4);
    L.part = L.red + (size_t)(L.nt / 32) * 2 * kLvDims * 8;  // also the selection's histogram
    L.tot = L.part + (size_t)C * 2 * L.dcap * 8;
    L.misc = L.tot + (size_t)2 * L.dcap * 8;
    L.total = L.misc + sizeof(LvMisc);
    return L;
}

__device__ __forceinline__ void lv_cp16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

template <int Q>  // 1 = BF16, 2 = FP16
__device__ __forceinline__ float lv_q16(uint32_t h) {
    if (Q == 1) return __uint_as_float(h << 16);
    return __half2float(__ushort_as_half((unsigned short)h));
}
// byte i of a word as a float, exactly
__device__ __forceinline__ float lv_u8(uint32_t word, int i) {
    return __fsub_rn(__uint_as_float(__byte_perm(word, 0x4B000000u, 0x7540u + (uint32_t)i)), 8388608.f);
}

// Four dims (quad `qd`) of a staged row.
template <int Q>
__device__ __forceinline__ void lv_quad(const uint8_t* row, int qd, float (&v)[4]) {
    if (Q == 3) {
        const uint32_t b = *reinterpret_cast<const uint32_t*>(row + 4 * qd);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = lv_u8(b, j);
    } else if (Q != 0) {
        const uint2 b = *reinterpret_cast<const uint2*>(row + 8 * qd);
        v[0] = lv_q16<Q>(b.x & 0xFFFFu);
        v[1] = lv_q16<Q>(b.x >> 16);
        v[2] = lv_q16<Q>(b.y & 0xFFFFu);
        v[3] = lv_q16<Q>(b.y >> 16);
    } else {
        const float4 f = *reinterpret_cast<const float4*>(row + 16 * qd);
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
    }
}

struct LvArgs {
    const float* X;
    int64_t n;  // rows of X
    int D;
    bool vec;   // rows of X are 16-byte aligned multiples of 16 bytes
    const uint16_t* Xq;
    int Dq, qtype;
    const int* qflag;
    const uint8_t* Xb;
    int Db;
    const int* bflag;
    const int32_t* seg_off;
    const int32_t* seg_tile0;
    const int32_t* seg_local;
    int level, iters;
    uint64_t pass_seed;
    const int32_t* perm_in;
    int32_t* perm_out;
    int* status;
    int max_m, row_bytes;
};

__device__ __forceinline__ int lv_excl_scan(int v, int* warp_tot, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w < nw; ++w) {
        const int t = warp_tot[w];
        before += w < warp ? t : 0;
        all += t;
    }
    *total = all;
    __syncthreads();
    return before + x - v;
}

template <int Q, int C>
__device__ __forceinline__ void level_segment(const LvArgs& P, const LvLayout& L, uint8_t* smem, int seg, int rank) {
    LvMisc& misc = *reinterpret_cast<LvMisc*>(smem + L.misc);
    uint64_t* few = misc.few;
    double* inv = misc.inv;
    int *warp_tot = misc.warp_tot, *sh = misc.sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (int)blockDim.x >> 5;
    const int a = P.seg_off[seg], m = P.seg_off[seg + 1] - a, K = m / 2, D = P.D;
    const int p0 = min(m, rank * L.q), ql = min(m, p0 + L.q) - p0;  // this CTA's positions p0 .. p0 + ql - 1
    uint32_t* S = reinterpret_cast<uint32_t*>(smem + L.S);
    int32_t* ids = reinterpret_cast<int32_t*>(smem + L.ids);
    uint8_t* side = smem + L.side;  // bit 0: left now, bit 1: left at the previous cut
    float* W = reinterpret_cast<float*>(smem + L.W);
    int* hist = reinterpret_cast<int*>(smem + L.red);
    double* red = reinterpret_cast<double*>(smem + L.red);      // [nw][2][kLvDims], or int64
    double* part = reinterpret_cast<double*>(smem + L.part);    // [C][2][dcap], or int64
    double* tot = reinterpret_cast<double*>(smem + L.tot);      // [dcap], then the left sums
    constexpr int kPer = Q == 3 ? 16 : Q != 0 ? 8 : 4;          // dims per 16-byte piece
    const int pieces = (D + kPer - 1) / kPer, stride = lv_stride(pieces * 16);
    auto sync = [&] {
        if (C > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    auto peer = [&](auto* p, int r) {
        if (C > 1) return cg::this_cluster().map_shared_rank(p, r);
        return p;
    };
    // the rows, once
    for (int r = tid; r < ql; r += blockDim.x) {
        int32_t id = P.perm_in[a + p0 + r];
        if (id < 0 || id >= P.n) {  // a failed partition above (reported): stay in bounds
            atomicOr(P.status, kStatusInternal);
            id = 0;
        }
        ids[r] = id;
        side[r] = 0;
    }
    for (int d = D + tid; d < ((D + 15) & ~15); d += blockDim.x) W[d] = 0.f;
    // initial centroids: the points at positions h, h2 of the segment, as
    // k1_init; and the means' reciprocals
    if (tid == 0) {
        const uint64_t sl = P.seg_local ? (uint64_t)P.seg_local[seg] : (uint64_t)seg;
        const uint64_t r1 = splitmix64(splitmix64(splitmix64(P.pass_seed) ^ (uint64_t)P.level) ^ sl);
        const uint64_t r2 = splitmix64(r1);
        const int64_t h = (int64_t)(r1 % (uint64_t)m);
        const int64_t h2 = (h + 1 + (int64_t)(r2 % (uint64_t)(m - 1))) % m;
        const int32_t i0 = P.perm_in[a + h], i1 = P.perm_in[a + h2];
        sh[0] = i0 < 0 || i0 >= P.n ? 0 : i0;
        sh[1] = i1 < 0 || i1 >= P.n ? 0 : i1;
    }
    if (Q == 0 && tid == 32) {
        inv[0] = 1.0 / (double)K;
        inv[1] = 1.0 / (double)(m - K);
    }
    __syncthreads();
    for (int d = tid; d < D; d += blockDim.x)
        W[d] = __fsub_rn(__ldg(P.X + (int64_t)sh[1] * D + d), __ldg(P.X + (int64_t)sh[0] * D + d));
    {
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
        if (Q != 0 || P.vec) {
            const uint8_t* src = Q == 3   ? P.Xb
                                 : Q != 0 ? reinterpret_cast<const uint8_t*>(P.Xq)
                                          : reinterpret_cast<const uint8_t*>(P.X);
            const int64_t pitch = Q == 3 ? P.Db : Q != 0 ? 2 * (int64_t)P.Dq : 4 * (int64_t)D;
            for (int e = tid; e < ql * pieces; e += blockDim.x) {
                const int r = e / pieces, c = e - r * pieces;
                lv_cp16(base + r * stride + c * 16, src + ids[r] * pitch + c * 16);
            }
            asm volatile("cp.async.wait_all;\n" ::: "memory");
        } else {
            const int D4 = pieces * 4;
            for (int e = tid; e < ql * D4; e += blockDim.x) {
                const int r = e / D4, d = e - r * D4;
                *reinterpret_cast<float*>(smem + r * stride + d * 4) =
                    d < D ? __ldg(P.X + (int64_t)ids[r] * D + d) : 0.f;
            }
        }
    }
    __syncthreads();
    // a peer may be stored to only once it runs
    sync();
    for (int it = 0;; ++it) {
        // project
        for (int r = tid; r < ql; r += blockDim.x) {
            const uint8_t* row = smem + r * stride;
            const float4* w4 = reinterpret_cast<const float4*>(W);
            float acc = 0.f;
#pragma unroll 4
            for (int c = 0; c < pieces; ++c) {
                const uint4 h = *reinterpret_cast<const uint4*>(row + c * 16);
                const uint32_t hv[4] = {h.x, h.y, h.z, h.w};
                if (Q == 3) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 w = w4[4 * c + u];
                        acc = __fmaf_rn(lv_u8(hv[u], 0), w.x, acc);
                        acc = __fmaf_rn(lv_u8(hv[u], 1), w.y, acc);
                        acc = __fmaf_rn(lv_u8(hv[u], 2), w.z, acc);
                        acc = __fmaf_rn(lv_u8(hv[u], 3), w.w, acc);
                    }
                } else if (Q != 0) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const float4 w = w4[2 * c + u];
                        acc = __fmaf_rn(lv_q16<Q>(hv[2 * u] & 0xFFFFu), w.x, acc);
                        acc = __fmaf_rn(lv_q16<Q>(hv[2 * u] >> 16), w.y, acc);
                        acc = __fmaf_rn(lv_q16<Q>(hv[2 * u + 1] & 0xFFFFu), w.z, acc);
                        acc = __fmaf_rn(lv_q16<Q>(hv[2 * u + 1] >> 16), w.w, acc);
                    }
                } else {
                    const float4 w = w4[c];
                    acc = __fmaf_rn(__uint_as_float(hv[0]), w.x, acc);
                    acc = __fmaf_rn(__uint_as_float(hv[1]), w.y, acc);
                    acc = __fmaf_rn(__uint_as_float(hv[2]), w.z, acc);
                    acc = __fmaf_rn(__uint_as_float(hv[3]), w.w, acc);
                }
            }
            const uint32_t o = ord32(__fadd_rn(acc, 0.f));  // -0 -> +0
#pragma unroll
            for (int r2 = 0; r2 < C; ++r2) peer(S, r2)[p0 + r] = o;
        }
        sync();
        // select the key (value, position) of rank K: 8-bit digits of the
        // value until at most 32 keys match (or the digits end), then those by
        // counting
        uint32_t v = 0;
        int krem = K, match = m, sft = 32;
        while (sft > 0 && match > 32) {
            sft -= 8;
            for (int b = tid; b < 256; b += blockDim.x) hist[b] = 0;
            __syncthreads();
            for (int p = tid; p < m; p += blockDim.x) {
                const uint32_t u = S[p];
                if (sft == 24 || (u >> (sft + 8)) == (v >> (sft + 8))) atomicAdd(hist + ((u >> sft) & 255), 1);
            }
            __syncthreads();
            if (warp == 0) {  // lane l: bins 8 l .. 8 l + 7
                const int4 h0 = reinterpret_cast<const int4*>(hist)[2 * lane];
                const int4 h1 = reinterpret_cast<const int4*>(hist)[2 * lane + 1];
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
            if (tid == 0) sh[3] = 0;
            __syncthreads();
            for (int p = tid; p < m; p += blockDim.x) {
                const uint32_t u = S[p];
                if (sft == 32 || (u >> sft) == (v >> sft)) few[atomicAdd(&sh[3], 1)] = ((uint64_t)u << 32) | (uint32_t)p;
            }
            __syncthreads();
            const uint64_t mine = lane < match ? few[lane] : ~0ull;
            int below = 0;
            for (int j = 0; j < match; ++j) below += shfl64(mine, j) < mine;
            const int src = __ffs(__ballot_sync(0xffffffffu, lane < match && below == krem)) - 1;
            const uint64_t key = shfl64(mine, src);
            v = (uint32_t)(key >> 32);
            tpos = (int)(uint32_t)key;
        } else if (krem > 0) {  // more than 32 equal values
            const int per = (m + (int)blockDim.x - 1) / (int)blockDim.x, b0 = min(m, tid * per), b1 = min(m, b0 + per);
            int c = 0, all;
            for (int p = b0; p < b1; ++p) c += S[p] == v;
            int before = lv_excl_scan(c, warp_tot, &all);
            if (before <= krem && krem < before + c)
                for (int p = b0; p < b1; ++p)
                    if (S[p] == v && before++ == krem) sh[3] = p;
            __syncthreads();
            tpos = sh[3];
        }
        auto is_left = [&](int p) {
            const uint32_t u = S[p];
            return u < v || (u == v && p < tpos);
        };
        if (it == P.iters) {  // the cut: left positions first, each side in position order
            int c = 0, before;
            for (int p = tid; p < p0; p += blockDim.x) c += is_left(p);
            lv_excl_scan(c, warp_tot, &before);  // left positions before p0
            for (int b = 0; b < ql; b += blockDim.x) {
                const int r = b + tid;
                const int isl = r < ql && is_left(p0 + r);
                int all;
                const int lb = before + lv_excl_scan(isl, warp_tot, &all);
                if (r < ql) {
                    const int np = isl ? lb : K + (p0 + r - lb);
                    if ((isl ? np < K : np < m) && np >= 0)
                        P.perm_out[a + np] = ids[r];
                    else
                        atomicOr(P.status, kStatusInternal);
                }
                before += all;
            }
            return;
        }
        for (int r = tid; r < ql; r += blockDim.x)
            side[r] = (uint8_t)(((side[r] & 1) << 1) | (is_left(p0 + r) ? 1 : 0));
        __syncthreads();
        // sums: both sides at the first cut, then only the rows that moved
        // (into the left sum with +, out of it with -)
        const int per = (ql + nw - 1) / nw, w0 = min(ql, warp * per), w1 = min(ql, w0 + per);
        for (int d0 = 0; d0 < D; d0 += kLvDims) {
            float h[2][4], l[2][4];
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int j = 0; j < 4; ++j) h[s][j] = l[s][j] = 0.f;
            const int qd = d0 / 4 + lane;
            const bool live = 4 * qd < D;
            auto add = [&](int s, const float (&x)[4], float sign) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float y = __fmul_rn(sign, x[j]);
                    if (Q != 0) {  // integers of magnitude <= 2048, at most a few hundred: exact
                        h[s][j] = __fadd_rn(h[s][j], y);
                    } else {  // TwoSum
                        const float sm = __fadd_rn(h[s][j], y), bp = __fsub_rn(sm, h[s][j]);
                        l[s][j] = __fadd_rn(l[s][j],
                                            __fadd_rn(__fsub_rn(h[s][j], __fsub_rn(sm, bp)), __fsub_rn(y, bp)));
                        h[s][j] = sm;
                    }
                }
            };
            for (int b = w0; b < w1; b += 32) {
                const int r = b + lane;
                const int sd = r < w1 ? side[r] : 0;
                const unsigned now = __ballot_sync(0xffffffffu, (sd & 1) != 0);
                const unsigned was = __ballot_sync(0xffffffffu, (sd & 2) != 0);
                if (it == 0) {
                    const int cnt = min(32, w1 - b);
                    for (int j = 0; j < cnt; ++j) {
                        float x[4] = {0.f, 0.f, 0.f, 0.f};
                        if (live) lv_quad<Q>(smem + (b + j) * stride, qd, x);
                        if ((now >> j) & 1u) add(0, x, 1.f);
                        else add(1, x, 1.f);
                    }
                } else {
                    for (unsigned mv = now ^ was; mv; mv &= mv - 1) {
                        const int j = __ffs(mv) - 1;
                        float x[4] = {0.f, 0.f, 0.f, 0.f};
                        if (live) lv_quad<Q>(smem + (b + j) * stride, qd, x);
                        add(0, x, ((now >> j) & 1u) ? 1.f : -1.f);
                    }
                }
            }
            __syncthreads();  // the histogram, or the previous chunk's sums, are read
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int at = (warp * 2 + s) * kLvDims + 4 * lane + j;
                    if (Q != 0)
                        reinterpret_cast<long long*>(red)[at] = (long long)__float2int_rn(h[s][j]);
                    else
                        red[at] = (double)h[s][j] + (double)l[s][j];
                }
            __syncthreads();
            for (int e = tid; e < 2 * kLvDims; e += blockDim.x) {
                const int s = e / kLvDims, dd = e - s * kLvDims, d = d0 + dd;
                if (d >= D || (s == 1 && it > 0)) continue;
                const int own = d / L.dcap, at = (rank * 2 + s) * L.dcap + d - own * L.dcap;
                if (Q != 0) {
                    long long sum = 0;
                    for (int w = 0; w < nw; ++w) sum += reinterpret_cast<long long*>(red)[(w * 2 + s) * kLvDims + dd];
                    peer(reinterpret_cast<long long*>(part), own)[at] = sum;
                } else {
                    double sum = 0.0;
                    for (int w = 0; w < nw; ++w) sum += red[(w * 2 + s) * kLvDims + dd];
                    peer(part, own)[at] = sum;
                }
            }
            __syncthreads();
        }
        sync();
        // the owner of a dim adds the CTAs' sums in order and sends w
        for (int dd = tid; dd < L.dcap; dd += blockDim.x) {
            const int d = rank * L.dcap + dd;
            if (d >= D) continue;
            float w;
            if (Q != 0) {
                const long long* ip = reinterpret_cast<const long long*>(part);
                long long* it_ = reinterpret_cast<long long*>(tot);
                long long s0 = 0, s1 = 0;
                for (int c = 0; c < C; ++c) {
                    s0 += ip[(c * 2 + 0) * L.dcap + dd];
                    if (it == 0) s1 += ip[(c * 2 + 1) * L.dcap + dd];
                }
                const long long sL = it == 0 ? s0 : it_[L.dcap + dd] + s0;
                if (it == 0) it_[dd] = s0 + s1;
                it_[L.dcap + dd] = sL;
                w = __fsub_rn(mean_of_ints(it_[dd] - sL, m - K), mean_of_ints(sL, K));
            } else {
                double s0 = 0.0, s1 = 0.0;
                for (int c = 0; c < C; ++c) {
                    s0 += part[(c * 2 + 0) * L.dcap + dd];
                    if (it == 0) s1 += part[(c * 2 + 1) * L.dcap + dd];
                }
                const double sL = it == 0 ? s0 : tot[L.dcap + dd] + s0;
                if (it == 0) tot[dd] = s0 + s1;
                tot[L.dcap + dd] = sL;
                const double sR = it == 0 ? s1 : tot[dd] - sL;
                w = __fsub_rn((float)div_by(sR, (double)(m - K), inv[1]), (float)div_by(sL, (double)K, inv[0]));
            }
#pragma unroll
            for (int r2 = 0; r2 < C; ++r2) peer(W, r2)[d] = w;
        }
        sync();
    }
}

template <int C>
__global__ void __launch_bounds__(512, 2) k1_level(const LvArgs P) {
    extern __shared__ __align__(16) uint8_t lv_smem[];
    const int seg = (int)(blockIdx.x / C), rank = (int)(blockIdx.x % C);
    if (P.seg_tile0[seg + 1] == P.seg_tile0[seg]) return;  // a finished tree's leaf (the whole cluster)
    const LvLayout L = lv_layout(P.D, P.max_m, P.row_bytes, C);
    // this segment's share of positions, as the plan's largest one would have it
    LvLayout M = L;
    M.q = (P.seg_off[seg + 1] - P.seg_off[seg] + C - 1) / C;
    int q = 0;
    if (P.Xb != nullptr && *P.bflag == 0) q = 3;
    else if (P.Xq != nullptr) {
        const int f = *P.qflag;
        if ((f & 1) == 0 && !((f & 2) && (f & 4))) q = P.qtype;
    }
    if (q == 3) level_segment<3, C>(P, M, lv_smem, seg, rank);
    else if (q == 1) level_segment<1, C>(P, M, lv_smem, seg, rank);
    else if (q == 2) level_segment<2, C>(P, M, lv_smem, seg, rank);
    else level_segment<0, C>(P, M, lv_smem, seg, rank);
}

template <int C>
void launch_level_c(const LvArgs& P, int nseg, int nt, size_t smem, cudaStream_t s) {
    allow_smem(k1_level<C>);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nseg * C);
    cfg.blockDim = dim3((unsigned)nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k1_level<C>, P);  // an error is the call's (LaunchScope)
}

}  // namespace

bool launch_level(const float* X, int64_t n, int D, const LevelPlan& lp, int iters, uint64_t pass_seed,
                  const int32_t* perm_in, int32_t* perm_out, const SplitBuffers& b, cudaStream_t s) {
    // bytes of a staged row; a captured build cannot know which copy is
    // exact, so its rows are sized as FP32
    const int row_bytes = b.u8_host ? (D + 15) / 16 * 16 : b.q16_host ? (D + 7) / 8 * 16 : (D + 3) / 4 * 16;
    // the fewest CTAs whose segments leave room for two per SM, else eight
    // with one per SM; more of them while that still fills no more than the chip
    int C = 1;
    while (C < 8 && lv_layout(D, lp.max_m, row_bytes, C).total > kLvTwo) C *= 2;
    while (C < 8 && lp.max_m / C >= 512 && (int64_t)lp.nseg * 2 * C <= kLvSms) C *= 2;
    const LvLayout L = lv_layout(D, lp.max_m, row_bytes, C);
    if (L.total > kLvOne) return false;
    // A level in one launch costs 40-70 us per wave of CTAs, where the sweeps
    // cost about 20 launches of at least 5 us and then the rows' passes over
    // memory; and other partitions want the chip as well.  Three passes,
    // knng_build_ex, before and after (GB300, this line at 4 waves of one CTA
    // per SM): 1,000 x 96 floats 1.01 -> 0.44 ms, 10,000 x 96 2.37 -> 1.32 ms,
    // 30,000 x 96 integers 2.75 -> 1.57 ms; the 10,000 x 32 mixture with two
    // rounds 1.70 -> 0.92 ms.  At 12 waves 100,000 x 96 gains 10-24 % more but
    // 200,000 x 96 and 100,000 x 256 floats lose 5 %, as do recorded builds.
    if ((int64_t)lp.nseg * C * b.share > 4 * kLvSms) return false;
    LvArgs P{};
    P.X = X;
    P.n = n;
    P.D = D;
    P.vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    P.Xq = b.Xq;
    P.Dq = b.Dq;
    P.qtype = b.qtype;
    P.qflag = b.qflag;
    P.Xb = b.Xb;
    P.Db = b.Db;
    P.bflag = b.bflag;
    P.seg_off = lp.seg_off;
    P.seg_tile0 = lp.seg_tile0;
    P.seg_local = lp.seg_local;
    P.level = lp.level;
    P.iters = iters;
    P.pass_seed = pass_seed;
    P.perm_in = perm_in;
    P.perm_out = perm_out;
    P.status = b.status;
    P.max_m = lp.max_m;
    P.row_bytes = row_bytes;
    // every row read once, with its id; the ids written
    LaunchScope ls("k1_level", s, (double)lp.n * (row_bytes + 8.0), (double)lp.n * D * (2.0 * (iters + 1) + 1.0));
    if (C == 1) launch_level_c<1>(P, lp.nseg, L.nt, L.total, s);
    else if (C == 2) launch_level_c<2>(P, lp.nseg, L.nt, L.total, s);
    else if (C == 4) launch_level_c<4>(P, lp.nseg, L.nt, L.total, s);
    else launch_level_c<8>(P, lp.nseg, L.nt, L.total, s);
    return true;
}

}  // namespace knng
