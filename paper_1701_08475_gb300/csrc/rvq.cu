// rvq.cu -- residue vector quantisation (Sec. 4.1, Eqn. 1) and the inverted
// index whose lists seed the graph search (Sec. 4.2, Eqns. 2 and 3).
//
// Two stages of Lloyd's k-means: stage 1 on the points, stage 2 on the FP32
// residues x - w1[c1(x)].  An iteration assigns every vector to its nearest
// word (canonical FP32 distance, ties to the smaller word index), groups the
// vectors by word with a stable counting sort, and sets each word with members
// to the FP64 mean of its members summed in ascending vector order, rounded to
// FP32 (a word without members keeps its value).  So the words do not depend
// on the launch configuration: each sum has one fixed order.
//
// The index key of a point is c1 * W2 + c2; its lists hold ids ascending (two
// stable 8-bit counting-sort passes, c2 then c1).  A query ranks the stage-1
// words by term 1 of Eqn. 3, keeps the first probe1, ranks their keys by the
// full Eqn. 2 distance built from lookup tables (q.w1, q.w2, |w|^2, w1.w2) and
// takes the ids of the lists in that order as its seeds.  Every decision that
// a float makes (an argmin, a ranking) is taken in FP32 with a fixed operation
// order, the same on every launch.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace knng {

namespace {

// ---------------------------------------------------------------- assignment
constexpr int kAR = 64;    // vectors per CTA
constexpr int kAC = 128;   // words per column tile
constexpr int kAT = 256;   // threads: 16 row groups x 16 column groups, 4 x 8 each

// Dims per shared-memory chunk and the padded row stride (an odd number of
// float4 per row keeps the 16 row groups' float4 reads on distinct banks).
__host__ __device__ inline void assign_chunk(int D, int* dch, int* stride) {
    const int d4 = (D + 3) & ~3;
    const int c = d4 < 64 ? d4 : 64;
    *dch = c;
    *stride = ((c / 4) & 1) ? c : c + 4;
}

size_t assign_smem(int D) {
    int dch, stride;
    assign_chunk(D, &dch, &stride);
    return (size_t)(kAR + kAC) * stride * 4 + (size_t)(8 + 1) * kAR * 8 + kAR * 4;
}

// codes[i * out_stride] = argmin_c |v_i - words_c|^2 for the N vectors
// v_i = X_i (RES false) or X_i - W1[c1[i * c1_stride]] (RES true, FP32).
template <bool RES>
__global__ void __launch_bounds__(kAT) k9_assign(const float* __restrict__ X, int64_t N, int D,
                                                const float* __restrict__ W1, const int32_t* __restrict__ c1,
                                                int c1_stride, const float* __restrict__ words, int W,
                                                int32_t* __restrict__ out, int out_stride) {
    extern __shared__ float4 sm4[];
    int dch, stride;
    assign_chunk(D, &dch, &stride);
    float* rs = reinterpret_cast<float*>(sm4);                      // [kAR][stride]
    float* ws = rs + kAR * stride;                                  // [kAC][stride]
    uint64_t* red = reinterpret_cast<uint64_t*>(ws + kAC * stride);  // [8][kAR]
    uint64_t* best = red + 8 * kAR;                                 // [kAR]
    int32_t* rcode = reinterpret_cast<int32_t*>(best + kAR);        // [kAR]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = tid % 16, cg = tid / 16;
    const int64_t r0 = (int64_t)blockIdx.x * kAR;
    const int nr = (int)min((int64_t)kAR, N - r0);
    if (tid < kAR) {
        best[tid] = kEmptyKey;
        rcode[tid] = (RES && tid < nr) ? c1[(r0 + tid) * c1_stride] : 0;
    }
    for (int c0 = 0; c0 < W; c0 += kAC) {
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        for (int d0 = 0; d0 < D; d0 += dch) {
            const int dl = min(dch, D - d0);
            __syncthreads();
            for (int e = tid; e < kAR * dch; e += kAT) {
                const int r = e / dch, dd = e - r * dch;
                float v = 0.f;
                if (r < nr && dd < dl) {
                    v = __ldg(X + (r0 + r) * D + d0 + dd);
                    if (RES) v = __fsub_rn(v, __ldg(W1 + (int64_t)rcode[r] * D + d0 + dd));
                }
                rs[r * stride + dd] = v;
            }
            for (int e = tid; e < kAC * dch; e += kAT) {
                const int r = e / dch, dd = e - r * dch;
                float v = 0.f;
                if (c0 + r < W && dd < dl) v = __ldg(words + (int64_t)(c0 + r) * D + d0 + dd);
                ws[r * stride + dd] = v;
            }
            __syncthreads();
            const float* rp = rs + rg * stride;
            const float* cp = ws + cg * stride;
            for (int dq = 0; dq < dch; dq += 4) {
                float4 rv[4], cv[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) rv[i] = *reinterpret_cast<const float4*>(rp + i * 16 * stride + dq);
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = *reinterpret_cast<const float4*>(cp + j * 16 * stride + dq);
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
        // the least (d, word) of each row in this tile: the thread's 8 words,
        // its partner of the other column group (lane ^ 16), then the 8 warps
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint64_t b = kEmptyKey;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = c0 + cg + 16 * j;
                if (c < W) b = min(b, make_key(acc[i][j], (uint32_t)c));
            }
            b = min(b, shfl_xor64(b, 16));
            if (lane < 16) red[warp * kAR + rg + 16 * i] = b;
        }
        __syncthreads();
        if (tid < kAR) {
            uint64_t b = best[tid];
#pragma unroll
            for (int w = 0; w < 8; ++w) b = min(b, red[w * kAR + tid]);
            best[tid] = b;
        }
    }
    __syncthreads();
    if (tid < nr) out[(r0 + tid) * out_stride] = (int32_t)key_id(best[tid]);
}

// ---------------------------------------------------------------- stable digit sort
constexpr int kDsThreads = 256;
constexpr int kDsItems = 8;
constexpr int kDsTile = kDsThreads * kDsItems;  // elements per CTA; a warp takes 256 consecutive ones

// Per-CTA histogram of the 8-bit digit key[id * kstride] of its elements
// (id = in[e], or e when in is null), stored digit-major: hist[d * nb + b].
__global__ void __launch_bounds__(kDsThreads) k9_digit_hist(const int32_t* __restrict__ in, int64_t n,
                                                           const int32_t* __restrict__ key, int kstride,
                                                           int32_t* __restrict__ hist, int nb) {
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kDsTile;
#pragma unroll
    for (int t = 0; t < kDsItems; ++t) {
        const int64_t e = base + t * kDsThreads + threadIdx.x;
        if (e < n) {
            const int64_t id = in ? (int64_t)__ldg(in + e) : e;
            atomicAdd(&h[__ldg(key + id * kstride) & 255], 1);
        }
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: element e goes to gofs[d * nb + b] + (elements of digit d
// before it in its CTA).  Warps take consecutive runs of 32 in element order;
// lanes with the same digit rank among themselves by lane (match_any).
__global__ void __launch_bounds__(kDsThreads) k9_digit_scatter(const int32_t* __restrict__ in, int64_t n,
                                                              const int32_t* __restrict__ key, int kstride,
                                                              const int32_t* __restrict__ gofs, int nb,
                                                              int32_t* __restrict__ out) {
    __shared__ int cnt[8][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < 8 * 256; d += kDsThreads) (&cnt[0][0])[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kDsTile + (int64_t)w * (32 * kDsItems);
    const unsigned lt = (1u << lane) - 1u;
    int32_t ids[kDsItems];
    int dig[kDsItems], rk[kDsItems];
#pragma unroll
    for (int t = 0; t < kDsItems; ++t) {
        const int64_t e = base + t * 32 + lane;
        const bool ok = e < n;
        const int32_t id = ok ? (in ? __ldg(in + e) : (int32_t)e) : 0;
        const int d = ok ? (__ldg(key + (int64_t)id * kstride) & 255) : 256;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        int r = __popc(peers & lt);
        if (ok) r += cnt[w][d];
        __syncwarp();
        if (ok && (peers & lt) == 0) cnt[w][d] += __popc(peers);
        __syncwarp();
        ids[t] = id;
        dig[t] = d;
        rk[t] = r;
    }
    __syncthreads();
    {   // exclusive prefix over the warps, one digit per thread
        int run = 0;
#pragma unroll
        for (int ww = 0; ww < 8; ++ww) {
            const int v = cnt[ww][threadIdx.x];
            cnt[ww][threadIdx.x] = run;
            run += v;
        }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kDsItems; ++t)
        if (dig[t] < 256) out[__ldg(gofs + (int64_t)dig[t] * nb + blockIdx.x) + cnt[w][dig[t]] + rk[t]] = ids[t];
}

// ---------------------------------------------------------------- word update
// A word's mean is defined by the FP64 sum of its members in ascending vector
// order.  Taken literally that is one chain of dependent additions per word
// and dim, as long as the largest word.  But FP32 values that are all
// multiples of a quantum q, with sums below 2^53 q, add without any rounding
// in FP64, in any order; nearly every (word, dim) is such a case.  So the
// members are summed in pieces (kUpRows consecutive positions of the sorted
// order per warp, cut where the word changes), then the pieces of a word, with
// the least and greatest magnitude on the way.  Where those do not prove the
// sum exact, an error bound of both orders decides whether the rounded mean
// can differ, and if it could, the word's chain runs as defined.
constexpr int kUpRows = 32;
constexpr int kUpDims = 128;  // dims per warp: 4 per lane

// Piece slots: unit u (positions kUpRows u ..) and word c meet in slot u + c
// (along the sorted order either the unit or the word moves on).  A slot holds
// D sums, then D pairs: the exponent of the lowest last set bit (2^(lo - 150))
// and A = sum |x| (rounded up).
constexpr int kUpNone = 1 << 20;  // no nonzero value
// e with 0 <= x < 2^e
__device__ __forceinline__ int up_exp(float x) { return max((int)(__float_as_uint(x) >> 23), 1) - 126; }
__device__ __forceinline__ double* up_slot(double* part, int64_t slot, int D) { return part + slot * 2 * D; }

template <bool VEC>
__global__ void __launch_bounds__(128) k9_pieces(const float* __restrict__ X, int64_t N, int D,
                                                const int32_t* __restrict__ order, const int32_t* __restrict__ gofs,
                                                int nb, int W, double* __restrict__ part) {
    __shared__ int start[257];  // where each word's positions start
    for (int c = threadIdx.x; c <= W; c += blockDim.x) start[c] = c < W ? gofs[(int64_t)c * nb] : (int)N;
    __syncthreads();
    const int lane = threadIdx.x & 31, d0 = blockIdx.y * kUpDims;
    const int64_t u = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int64_t p0 = u * kUpRows;
    if (p0 >= N) return;
    const int p1 = (int)min(N, p0 + kUpRows);
    const int my_id = p0 + lane < p1 ? order[p0 + lane] : 0;
    int c = 0;  // the last word that starts at or before p0 and is not empty there
    for (int step = 128; step > 0; step >>= 1)
        if (c + step < W && start[c + step] <= (int)p0) c += step;
    for (int p = (int)p0; p < p1;) {
        while (start[c + 1] <= p) ++c;
        const int end = min(p1, start[c + 1]);
        // FP32 sums h with the additions' rounding errors summed in l (Knuth's
        // TwoSum): FP64 issues at a small fraction of the FP32 rate.  With
        // A = sum |x| < 2^ea, each error is at most 2^(ea - 25) and l below
        // 2^(ea - 20), exact up to 2^24 quanta of 2^(lo - 150).
        float h[4], l[4], A[4];
        int lo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            h[j] = l[j] = A[j] = 0.f;
            lo[j] = kUpNone;
        }
        auto load = [&](int id, bool in, float (&v)[4]) {
            const float* x = X + (int64_t)id * D + d0;
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = 0.f;
            if (!in) return;
            if (VEC) {
                if (d0 + 4 * lane < D) {
                    const float4 f = __ldg(reinterpret_cast<const float4*>(x) + lane);
                    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (d0 + 4 * lane + j < D) v[j] = __ldg(x + 4 * lane + j);
            }
        };
        for (int t = p; t < end; t += 8) {  // 8 rows in flight; rows past the end add +0
            float v[8][4];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                load(__shfl_sync(0xffffffffu, my_id, (t + q - (int)p0) & 31), t + q < end, v[q]);
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float x = v[q][j], sm = __fadd_rn(h[j], x), bp = __fsub_rn(sm, h[j]);
                    l[j] = __fadd_rn(l[j], __fadd_rn(__fsub_rn(h[j], __fsub_rn(sm, bp)), __fsub_rn(x, bp)));
                    h[j] = sm;
                    const uint32_t m = __float_as_uint(x) & 0x7fffffffu;
                    const uint32_t man = (m & 0x7fffffu) | (m >= 0x800000u ? 0x800000u : 0u);
                    // exponent field (1 for subnormals) plus the zeros below
                    // the last set bit
                    const int last = max((int)(m >> 23), 1) + 31 - __clz((int)(man & (0u - man)));
                    lo[j] = min(lo[j], m ? last : kUpNone);
                    A[j] = __fadd_ru(A[j], fabsf(x));
                }
        }
        double acc[4];
        bool wide = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc[j] = __dadd_rn((double)h[j], (double)l[j]);
            // (and no overflow of h: FP64 holds what FP32 does not)
            wide |= up_exp(A[j]) - (lo[j] - 150) > 44 || !(A[j] < 1e38f);
        }
        if (__any_sync(0xffffffffu, wide)) {  // magnitudes too far apart: FP64 throughout
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = 0.0;
            for (int t = p; t < end; ++t) {
                float v[4];
                load(__shfl_sync(0xffffffffu, my_id, (t - (int)p0) & 31), true, v);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[j] = __dadd_rn(acc[j], (double)v[j]);
            }
        }
        p = end;
        double* o = up_slot(part, u + c, D);
        uint2* mags = reinterpret_cast<uint2*>(o + D);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int d = d0 + 4 * lane + j;
            if (d < D) {
                o[d] = acc[j];
                mags[d] = make_uint2((uint32_t)lo[j], __float_as_uint(A[j]));
            }
        }
    }
}

// (double)x by integer operations: the conversion would take the FP64 units as
// long as the addition that follows it.
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
    if (m != 0 && m < 0x00800000u) return (double)x;  // subnormal
    const uint32_t hi = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(m << 29));
}

// One CTA per word and 128 dims: the sum of its pieces, the proof that the
// rounded mean is the defined one, and else the chain: one group adds 32 members
// from shared memory while the others bring the next 32.  Its bound is then the
// FP64 units: an addition of a warp has a latency of 64 cycles and takes 19 of
// the SM's.  41,286 x 480 GIST-like rows in 64 uneven words (one of 37,571), 16
// updates: 43.8 ms with one thread loading 32 values and then adding them, or
// with a word's chunks of dims on one SM; 25.0 so.
constexpr int kCbGroups = 4;  // the pieces of a word are read by this many threads per dim
constexpr int kCbRows = 32;   // members staged at once
constexpr int kCbShare = (kCbRows + kCbGroups - 2) / (kCbGroups - 1);  // of them per loading thread
__global__ void __launch_bounds__(128 * kCbGroups) k9_combine(const float* __restrict__ X, int64_t N, int D,
                                                 const int32_t* __restrict__ order,
                                                 const int32_t* __restrict__ gofs, int nb, int W,
                                                 double* __restrict__ part, float* __restrict__ words) {
    __shared__ double gsum[kCbGroups][128];
    __shared__ float gabs[kCbGroups][128];
    __shared__ int glo[kCbGroups][128];
    __shared__ float rows[2][kCbRows][128];
    const int dd = threadIdx.x & 127, g = threadIdx.x >> 7;
    // a word's chunks of dims are neighbours in the grid, which go to different
    // SMs: side by side on one their chains share its FP64 units
    const int chunks = (D + 127) / 128, c = (int)(blockIdx.x / chunks), d = (int)(blockIdx.x % chunks) * 128 + dd;
    const int a = gofs[(int64_t)c * nb], b = c + 1 < W ? gofs[(int64_t)(c + 1) * nb] : (int)N;
    if (b == a) return;  // no members: the word keeps its value (the whole CTA)
    double sum = 0.0;
    const int m = b - a;
    bool open = part == nullptr && g == 0;  // whether this sum has to be the chain's
    if (part != nullptr) {
        int lo = kUpNone;
        float A = 0.f;
        if (d < D) {
#pragma unroll 4
            for (int64_t u = a / kUpRows + g; u <= (b - 1) / kUpRows; u += kCbGroups) {
                const double* o = up_slot(part, u + c, D);
                const uint2 mg = reinterpret_cast<const uint2*>(o + D)[d];
                sum = __dadd_rn(sum, o[d]);
                lo = min(lo, (int)mg.x);
                A = __fadd_ru(A, __uint_as_float(mg.y));
            }
        }
        gsum[g][dd] = sum;
        gabs[g][dd] = A;
        glo[g][dd] = lo;
        __syncthreads();
        if (g == 0) {
#pragma unroll
            for (int q = 1; q < kCbGroups; ++q) {
                sum = __dadd_rn(sum, gsum[q][dd]);
                A = __fadd_ru(A, gabs[q][dd]);
                lo = min(lo, glo[q][dd]);
            }
            // every value is a multiple of 2^(lo - 150) and no partial sum is
            // above A, which past FP32's range is no bound at all (then x and
            // y below differ)
            if (up_exp(A) > 53 + lo - 150 || isinf(A)) {
                // the defined order is within m 2^-53 A, and a little, of the
                // true sum; this one, which adds at most m / 128 + 48 times in
                // a row, nearer
                const double e = ldexp(((double)m * 1.0625 + 64.0) * (double)A, -53);
                const float x = __double2float_rn(__ddiv_rn(sum - e, (double)m));
                const float y = __double2float_rn(__ddiv_rn(sum + e, (double)m));
                open = x != y || x == 0.f;
            }
        }
    }
    if (__syncthreads_or(open)) {
        double s = 0.0;
        for (int t = a - kCbRows; t < b; t += kCbRows) {  // members t .. are added, the next ones brought
            const int buf = ((t - a) / kCbRows) & 1;
            if (g > 0) {
                float v[kCbShare];
#pragma unroll
                for (int q = 0; q < kCbShare; ++q) {
                    const int r = g - 1 + q * (kCbGroups - 1), p = t + kCbRows + r;
                    v[q] = r < kCbRows && p < b && d < D ? __ldg(X + (int64_t)__ldg(order + p) * D + d) : 0.f;
                }
#pragma unroll
                for (int q = 0; q < kCbShare; ++q) {
                    const int r = g - 1 + q * (kCbGroups - 1);
                    if (r < kCbRows) rows[buf ^ 1][r][dd] = v[q];
                }
            } else if (t >= a) {
#pragma unroll
                for (int r = 0; r < kCbRows; ++r)
                    if (t + r < b) s = __dadd_rn(s, widen(rows[buf][r][dd]));
            }
            __syncthreads();
        }
        if (open) sum = s;
    }
    if (g == 0 && d < D) words[(int64_t)c * D + d] = __double2float_rn(__ddiv_rn(sum, (double)m));
}

// words[c] = v_{pos[c]} (the initial words).
__global__ void k9_init_words(const float* __restrict__ X, int D, const int64_t* __restrict__ pos, int W,
                              float* __restrict__ words) {
    const int64_t total = (int64_t)W * D;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(e / D), j = (int)(e - (int64_t)c * D);
        words[e] = X[pos[c] * D + j];
    }
}

// R_i = X_i - W1[c1[i]] (FP32), the stage-2 vectors, written once for all
// of stage 2's iterations.
__global__ void k9_residues(const float* __restrict__ X, int64_t N, int D, const float* __restrict__ W1,
                            const int32_t* __restrict__ c1, float* __restrict__ R) {
    const int64_t total = N * D;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / D;
        R[e] = __fsub_rn(X[e], W1[(int64_t)c1[i] * D + (e - i * D)]);
    }
}

// ---------------------------------------------------------------- index
__global__ void k9_key_count(const int32_t* __restrict__ codes, int64_t n, int W2, int32_t* __restrict__ cnt) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(cnt + (int64_t)codes[2 * e] * W2 + codes[2 * e + 1], 1);
}

// Offsets given by the caller: off[0] >= 0, non-decreasing, off[nk] <= n.
__global__ void k9_check_offsets(const int32_t* __restrict__ off, int64_t nk, int64_t n, int* status) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e <= nk; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = off[e];
        const bool bad = (e == 0 && v < 0) || (e > 0 && v < off[e - 1]) || (e == nk && (int64_t)v > n);
        if (bad) atomicOr(status, kStatusBadInput);
    }
}

// ---------------------------------------------------------------- query tables
__device__ __forceinline__ float dot_canon(const float* __restrict__ a, const float* __restrict__ b, int D) {
    float acc = 0.f;
    for (int j = 0; j < D; ++j) acc = __fmaf_rn(__ldg(a + j), __ldg(b + j), acc);
    return acc;
}

// n1[a] = |w1_a|^2, n2[b] = |w2_b|^2, x12[a][b] = w1_a . w2_b (canonical), and
// the transposed vocabularies w1T (D x W1), w2T (D x W2) for coalesced query
// products.
__global__ void k9_tables(const float* __restrict__ w1, int W1, const float* __restrict__ w2, int W2, int D,
                          float* __restrict__ n1, float* __restrict__ n2, float* __restrict__ x12,
                          float* __restrict__ w1T, float* __restrict__ w2T) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, gs = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = g; e < (int64_t)W1 * W2; e += gs) {
        const int a = (int)(e / W2), b = (int)(e - (int64_t)a * W2);
        x12[e] = dot_canon(w1 + (int64_t)a * D, w2 + (int64_t)b * D, D);
    }
    for (int64_t e = g; e < W1; e += gs) n1[e] = dot_canon(w1 + e * D, w1 + e * D, D);
    for (int64_t e = g; e < W2; e += gs) n2[e] = dot_canon(w2 + e * D, w2 + e * D, D);
    for (int64_t e = g; e < (int64_t)W1 * D; e += gs) {
        const int a = (int)(e / D), j = (int)(e - (int64_t)a * D);
        w1T[(int64_t)j * W1 + a] = w1[e];
    }
    for (int64_t e = g; e < (int64_t)W2 * D; e += gs) {
        const int b = (int)(e / D), j = (int)(e - (int64_t)b * D);
        w2T[(int64_t)j * W2 + b] = w2[e];
    }
}

// ---------------------------------------------------------------- seeds
constexpr int kSdT = 256;

// Ascending bitonic sort of P keys (P a power of two >= 2) in shared memory by
// the whole CTA.  The caller synchronises before; this returns synchronised.
__device__ void block_bitonic(uint64_t* a, int P) {
    for (int k = 2; k <= P; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < P; i += kSdT) {
                const int l = i ^ j;
                if (l > i) {
                    const uint64_t x = a[i], y = a[l];
                    if ((x > y) == ((i & k) == 0)) {
                        a[i] = y;
                        a[l] = x;
                    }
                }
            }
            __syncthreads();
        }
}

// Exclusive scan of one int per thread over the CTA; *total gets the sum.
__device__ int block_excl_scan(int v, int* wsum, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int i = 0; i < kSdT / 32; ++i) {
            const int t = wsum[i];
            wsum[i] = run;
            run += t;
        }
        *total = run;
    }
    __syncthreads();
    return wsum[w] + x - v;
}

size_t seeds_smem(int P, int D) { return (size_t)P * 8 + 256 * 8 + (kSdT / 32 + 1) * 4 + 256 * 4 + (size_t)D * 4; }

// One CTA per query.  P: room for the candidate keys (probe1 * W2 rounded up
// to a power of two, at least kSdT); only those with a non-empty list are
// ranked.
__global__ void __launch_bounds__(kSdT) k9_seeds(const float* __restrict__ w1T, int W1,
                                                const float* __restrict__ w2T, int W2, int D,
                                                const float* __restrict__ n1, const float* __restrict__ n2,
                                                const float* __restrict__ x12, const int32_t* __restrict__ off,
                                                const int32_t* __restrict__ ids, const float* __restrict__ Q,
                                                int p1, int P, int s, int32_t* __restrict__ S,
                                                const int* __restrict__ status) {
    if (*status & kStatusStop) return;  // the caller's offsets failed their check
    extern __shared__ uint64_t smk[];
    uint64_t* cand = smk;                                   // [P]
    uint64_t* t1 = cand + P;                                // [256]
    int* wsum = reinterpret_cast<int*>(t1 + 256);           // [kSdT / 32 + 1]
    float* qw2 = reinterpret_cast<float*>(wsum + kSdT / 32 + 1);  // [256]
    float* q = qw2 + 256;                                   // [D]
    const int tid = threadIdx.x;
    const int64_t qi = blockIdx.x;
    for (int j = tid; j < D; j += kSdT) q[j] = __ldg(Q + qi * D + j);
    __syncthreads();
    float qq = 0.f;  // every thread, the same value
    for (int j = 0; j < D; ++j) qq = __fmaf_rn(q[j], q[j], qq);
    // Eqn. 3's term 1 for every stage-1 word, and q . w2
    uint64_t k1 = kEmptyKey;
    if (tid < W1) {
        float a = 0.f;
        for (int j = 0; j < D; ++j) a = __fmaf_rn(q[j], __ldg(w1T + (int64_t)j * W1 + tid), a);
        const float t = __fadd_rn(__fadd_rn(__fmaf_rn(-2.f, a, qq), __ldg(n1 + tid)), 0.f);
        k1 = make_key(t, (uint32_t)tid);
    }
    t1[tid] = k1;
    if (tid < W2) {
        float a = 0.f;
        for (int j = 0; j < D; ++j) a = __fmaf_rn(q[j], __ldg(w2T + (int64_t)j * W2 + tid), a);
        qw2[tid] = a;
    }
    __syncthreads();
    block_bitonic(t1, 256);
    // term 2 for the kept words' keys, d(q, I) = term 1 + term 2 (Eqn. 2).
    // Keys of empty lists add no seed: only the others are kept (in any
    // order, the sort below fixes it), with their list's start and length.
    __shared__ int nkeep;
    if (tid == 0) nkeep = 0;
    __syncthreads();
    const int nc = p1 * W2;
    for (int e0 = 0; e0 < nc; e0 += kSdT) {
        const int e = e0 + tid;
        uint64_t key = kEmptyKey;
        if (e < nc) {
            const int r = e / W2, b = e - r * W2;
            const uint64_t kk = t1[r];
            const int a = (int)key_id(kk), I = a * W2 + b;
            if (__ldg(off + I + 1) > __ldg(off + I)) {
                const float t2 =
                    __fmaf_rn(-2.f, qw2[b], __fmaf_rn(2.f, __ldg(x12 + (int64_t)a * W2 + b), __ldg(n2 + b)));
                const float d = __fadd_rn(__fadd_rn(key_dist(kk), t2), 0.f);
                key = make_key(d, (uint32_t)I);
            }
        }
        const unsigned ball = __ballot_sync(0xffffffffu, key != kEmptyKey);
        int base = 0;
        if ((tid & 31) == 0 && ball) base = atomicAdd(&nkeep, __popc(ball));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (key != kEmptyKey) cand[base + __popc(ball & ((1u << (tid & 31)) - 1u))] = key;
    }
    __syncthreads();
    const int nk = nkeep;
    int Pk = 2;
    while (Pk < nk) Pk <<= 1;
    for (int e = nk + tid; e < Pk; e += kSdT) cand[e] = kEmptyKey;
    __syncthreads();
    block_bitonic(cand, Pk);
    // the lists in that order: thread t walks keys [t * per, (t + 1) * per)
    const int per = (Pk + kSdT - 1) / kSdT;
    int mine = 0;
    for (int u = 0; u < per; ++u) {
        const int e = tid * per + u;
        if (e >= nk) break;
        const int I = (int)key_id(cand[e]);
        mine += __ldg(off + I + 1) - __ldg(off + I);
    }
    __shared__ int total;
    int pos = block_excl_scan(mine, wsum, &total);
    for (int u = 0; u < per && pos < s; ++u) {
        const int e = tid * per + u;
        if (e >= nk) break;
        const int I = (int)key_id(cand[e]);
        const int a0 = __ldg(off + I), a1 = __ldg(off + I + 1);
        for (int t = a0; t < a1 && pos < s; ++t) S[qi * s + pos++] = __ldg(ids + t);
    }
    for (int p = min(total, s) + tid; p < s; p += kSdT) S[qi * s + p] = -1;
}

// ---------------------------------------------------------------- few seeds
// For up to 32 seeds per query (kSeedFew): the products of all queries and
// words as one blocked FP32 product (k9_dots), the query-independent part of
// every key's distance once (k9_keys), and then one CTA per query picks the
// kept words and the seeds (k9_few_seeds).  Every float operation is
// k9_seeds's own.
constexpr int kSeedFew = 32;
constexpr int kDotRows = 64, kDotCols = 128, kDotDims = 64, kDotStride = kDotDims + 4;
constexpr uint32_t kNoList = 0x7FFFDEADu;  // in place of a key's part of the distance: its list is empty

// out[r][c] = a_r . b_c (canonical: dims ascending, fmaf), self[r] = a_r . a_r.
// 256 threads: 16 row groups x 16 column groups, 4 x 8 products each.
template <bool VEC>
__global__ void __launch_bounds__(256) k9_dots(const float* __restrict__ A, int64_t M, const float* __restrict__ B,
                                              int W, int D, float* __restrict__ out, float* __restrict__ self) {
    extern __shared__ __align__(16) float dt_smem[];
    float* as = dt_smem;                          // [kDotRows][kDotStride]
    float* bs = as + kDotRows * kDotStride;       // [kDotCols][kDotStride]
    const int tid = threadIdx.x, rg = tid % 16, cg = tid / 16;
    const int64_t r0 = (int64_t)blockIdx.x * kDotRows;
    const int c0 = blockIdx.y * kDotCols;
    float acc[4][8], own = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    auto stage = [&](float* dst, const float* src, int rows, int64_t first, int64_t count, int d0) {
        if (VEC) {
            for (int e = tid; e < rows * (kDotDims / 4); e += 256) {
                const int r = e / (kDotDims / 4), c = e % (kDotDims / 4) * 4;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (first + r < count && d0 + c < D)
                    v = __ldg(reinterpret_cast<const float4*>(src + (first + r) * D + d0 + c));
                *reinterpret_cast<float4*>(dst + r * kDotStride + c) = v;
            }
        } else {
#pragma unroll 16  // that many loads in flight
            for (int e = tid; e < rows * kDotDims; e += 256) {
                const int r = e / kDotDims, c = e % kDotDims;
                dst[r * kDotStride + c] = first + r < count && d0 + c < D ? __ldg(src + (first + r) * D + d0 + c) : 0.f;
            }
        }
    };
    for (int d0 = 0; d0 < D; d0 += kDotDims) {
        __syncthreads();
        stage(as, A, kDotRows, r0, M, d0);
        stage(bs, B, kDotCols, c0, W, d0);
        __syncthreads();
        const int dl = (min(kDotDims, D - d0) + 3) & ~3;  // dims past D are zeros: they change no sum
        for (int dq = 0; dq < dl; dq += 4) {
            float4 av[4], bv[8];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                av[i] = *reinterpret_cast<const float4*>(as + (rg + 16 * i) * kDotStride + dq);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                bv[j] = *reinterpret_cast<const float4*>(bs + (cg + 16 * j) * kDotStride + dq);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc[i][j] = __fmaf_rn(av[i].x, bv[j].x, acc[i][j]);
                    acc[i][j] = __fmaf_rn(av[i].y, bv[j].y, acc[i][j]);
                    acc[i][j] = __fmaf_rn(av[i].z, bv[j].z, acc[i][j]);
                    acc[i][j] = __fmaf_rn(av[i].w, bv[j].w, acc[i][j]);
                }
        }
        if (blockIdx.y == 0 && tid < kDotRows) {
            const float* x = as + tid * kDotStride;
            for (int d = 0; d < dl; ++d) own = __fmaf_rn(x[d], x[d], own);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int64_t r = r0 + rg + 16 * i;
            const int c = c0 + cg + 16 * j;
            if (r < M && c < W) out[r * W + c] = acc[i][j];
        }
    if (blockIdx.y == 0 && tid < kDotRows && r0 + tid < M) self[r0 + tid] = own;
}

// The na values of a, then the nb of b (one launch less than two copies).
__global__ void __launch_bounds__(256) k9_stack(const float* __restrict__ a, int64_t na, const float* __restrict__ b,
                                               int64_t nb, float* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < na + nb; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = e < na ? __ldg(a + e) : __ldg(b + e - na);
}

// part[a * W2 + b] = fmaf(2, w1_a . w2_b, |w2_b|^2), or kNoList when the key's
// list is empty.  T, self: products of the stacked words with themselves.
__global__ void k9_keys(const float* __restrict__ T, const float* __restrict__ self, int W1, int W2,
                        const int32_t* __restrict__ off, float* __restrict__ part, const int* __restrict__ status) {
    if (*status & kStatusStop) return;  // the caller's offsets failed their check
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < W1 * W2; e += gridDim.x * blockDim.x) {
        const int a = e / W2, b = e - a * W2;
        part[e] = off[e + 1] > off[e] ? __fmaf_rn(2.f, T[(int64_t)a * (W1 + W2) + W1 + b], self[W1 + b])
                                      : __uint_as_float(kNoList);
    }
}

// One CTA per query; its first warp ranks the words and the seeds, all four
// form and sift the candidates (one warp per query waited for memory most of
// the time: 344 us for 10,000 queries).  Shared memory: 256 keys, the kept
// words, the products with the second words, 256 counters, the threads' least
// distances, the candidate distances (probe1 W2).
constexpr int kFewKeys = 256, kFewT = 128;
size_t few_seeds_smem(int p1, int W2) {
    return (size_t)kFewKeys * 8 + 256 * 8 + 256 * 4 + 260 * 4 + kFewT * 4 + (size_t)p1 * W2 * 4;
}

// VEC: W2 is a multiple of 4.
template <bool VEC>
__global__ void __launch_bounds__(kFewT) k9_few_seeds(const float* __restrict__ dots, const float* __restrict__ qq,
                                                     const float* __restrict__ self, int W1, int W2, int p1,
                                                     const float* __restrict__ part, const int32_t* __restrict__ off,
                                                     const int32_t* __restrict__ ids, int s,
                                                     int32_t* __restrict__ S, const int* __restrict__ status) {
    if (*status & kStatusStop) return;
    extern __shared__ __align__(16) uint64_t fs_smem[];
    uint64_t* keys = fs_smem;                                        // [kFewKeys]
    uint64_t* kept = keys + kFewKeys;                                // [256] (term 1, word), the first p1 kept
    float* qw2 = reinterpret_cast<float*>(kept + 256);               // [256]
    int* hist = reinterpret_cast<int*>(qw2 + 256);                   // [256]
    int* count = hist + 256;                                         // keys taken
    uint32_t* slim = reinterpret_cast<uint32_t*>(count + 1);         // the bound, the least distance
    uint32_t* lmin = reinterpret_cast<uint32_t*>(hist + 260);        // [kFewT]
    uint32_t* cand = lmin + kFewT;                                   // [p1 W2] distances (ord32), ~0: no list
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t qi = blockIdx.x;
    const float* dq = dots + qi * (W1 + W2);
    uint64_t v[8];
    if (warp == 0) {
        // Eqn. 3's term 1 of every stage-1 word; the p1 least are kept
        const float q2 = qq[qi];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int a = 32 * r + lane;
            v[r] = a < W1 ? make_key(__fadd_rn(__fadd_rn(__fmaf_rn(-2.f, dq[a], q2), self[a]), 0.f), (uint32_t)a)
                          : kEmptyKey;
        }
        if (p1 <= 32) {
            uint64_t first[1];
            sort_regs<8>(v);
            warp_select_unique<8, 1>(v, p1, first);  // the keys are distinct
            kept[lane] = first[0];
        } else {
            bitonic_sort_keys<8, 1>(v, nullptr);
#pragma unroll
            for (int r = 0; r < 8; ++r) kept[8 * lane + r] = v[r];
        }
    } else {
        for (int b = tid - 32; b < W2; b += kFewT - 32) qw2[b] = dq[W1 + b];
        for (int e = tid - 32; e < 256; e += kFewT - 32) hist[e] = 0;
        if (tid == 32) *count = 0;
    }
    __syncthreads();
    // d(q, I) of the kept words' keys; each thread's least on the way
    uint32_t least = 0xFFFFFFFFu;
    auto distance = [&](float t1, float qw, float c) -> uint32_t {
        if (__float_as_uint(c) == kNoList) return 0xFFFFFFFFu;
        return min(0xFFFFFFFEu, ord32(__fadd_rn(__fadd_rn(t1, __fmaf_rn(-2.f, qw, c)), 0.f)));
    };
    for (int r = warp; r < p1; r += kFewT / 32) {
        const uint64_t kk = kept[r];
        const float t1 = key_dist(kk);
        const float* pr = part + (int64_t)key_id(kk) * W2;
        if (VEC) {
            for (int b = 4 * lane; b < W2; b += 128) {
                const float4 c = __ldg(reinterpret_cast<const float4*>(pr + b));
                const float4 w = *reinterpret_cast<const float4*>(qw2 + b);
                const uint4 u = make_uint4(distance(t1, w.x, c.x), distance(t1, w.y, c.y), distance(t1, w.z, c.z),
                                           distance(t1, w.w, c.w));
                *reinterpret_cast<uint4*>(cand + r * W2 + b) = u;
                least = min(least, min(min(u.x, u.y), min(u.z, u.w)));
            }
        } else {
            for (int b = lane; b < W2; b += 32) {
                const uint32_t u = distance(t1, qw2[b], __ldg(pr + b));
                cand[r * W2 + b] = u;
                least = min(least, u);
            }
        }
    }
    lmin[tid] = least;
    __syncthreads();
    // The s-th least of the threads' least distances bounds the s-th least of
    // all: only keys up to it can be among the first s (every list gives at
    // least one seed).  The near words of the second stage crowd into few
    // threads, so the bound can be loose: the keys up to it are counted in 256
    // even steps, and the bound becomes the end of the step with the s-th.
    int below = 0;
    uint32_t mn = 0xFFFFFFFFu;
    for (int j = 0; j < kFewT; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(lmin + j);
        mn = min(mn, min(min(o.x, o.y), min(o.z, o.w)));
        below += (o.x < least || (o.x == least && j < tid)) + (o.y < least || (o.y == least && j + 1 < tid)) +
                 (o.z < least || (o.z == least && j + 2 < tid)) + (o.w < least || (o.w == least && j + 3 < tid));
    }
    if (below == s - 1) *slim = min(least, 0xFFFFFFFEu);
    __syncthreads();
    uint32_t lim = *slim;
    const int nc = p1 * W2;
    if (mn <= lim) {  // the same for every thread
        const int sft = max(0, 24 - __clz((int)(lim - mn)));
        auto tally = [&](uint32_t u) {
            if (u <= lim) atomicAdd(hist + ((u - mn) >> sft), 1);
        };
        for (int e = (VEC ? 4 : 1) * tid; e < nc; e += (VEC ? 4 : 1) * kFewT) {
            if (VEC) {
                const uint4 u = *reinterpret_cast<const uint4*>(cand + e);
                tally(u.x);
                tally(u.y);
                tally(u.z);
                tally(u.w);
            } else {
                tally(cand[e]);
            }
        }
        __syncthreads();
        if (warp == 0) {
            int c[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                c[j] = hist[8 * lane + j];
                sum += c[j];
            }
            int run = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, run, o);
                if (lane >= o) run += y;
            }
            const unsigned got = __ballot_sync(0xffffffffu, run >= s);
            run -= sum;
            int step = 8 * lane;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (run + c[j] >= s) break;
                run += c[j];
                ++step;
            }
            if (got && lane == __ffs(got) - 1) {  // else fewer than s keys
                // the step's end may lie past the last 32-bit key
                const uint64_t end = mn + (((uint64_t)step + 1) << sft) - 1;
                *slim = end < lim ? (uint32_t)end : lim;
            }
        }
        __syncthreads();
        lim = *slim;
    }
    auto take = [&](uint32_t u, int e) {
        if (u > lim) return;
        const int at = atomicAdd(count, 1);
        const int r = e / W2;
        if (at < kFewKeys) keys[at] = ((uint64_t)u << 32) | (key_id(kept[r]) * (uint32_t)W2 + (e - r * W2));
    };
    for (int e = (VEC ? 4 : 1) * tid; e < nc; e += (VEC ? 4 : 1) * kFewT) {
        if (VEC) {
            const uint4 u = *reinterpret_cast<const uint4*>(cand + e);
            if (min(min(u.x, u.y), min(u.z, u.w)) > lim) continue;
            take(u.x, e);
            take(u.y, e + 1);
            take(u.z, e + 2);
            take(u.w, e + 3);
        } else {
            take(cand[e], e);
        }
    }
    __syncthreads();
    if (warp > 0) return;
    const int total = *count;
    if (total <= 32) {
        const uint64_t one = warp_sort32(lane < total ? keys[lane] : kEmptyKey);
        __syncwarp();
        keys[lane] = one;
    } else if (total <= 64) {
        uint64_t two[2] = {keys[lane], lane + 32 < total ? keys[lane + 32] : kEmptyKey};
        __syncwarp();
        bitonic_sort_keys<2, 1>(two, nullptr);
        if (lane < 16) {
            keys[2 * lane] = two[0];
            keys[2 * lane + 1] = two[1];
        }
    } else if (total <= kFewKeys) {
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = 32 * r + lane < total ? keys[32 * r + lane] : kEmptyKey;
        __syncwarp();
        bitonic_sort_keys<8, 1>(v, nullptr);
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (8 * lane + r < 32) keys[8 * lane + r] = v[r];
    } else {  // crowded: the least key above the last one, s times
        uint64_t last = 0;
        for (int t = 0; t < 32; ++t) {
            uint64_t m = kEmptyKey;
            for (int e = lane; e < nc; e += 32) {
                const int r = e / W2;
                const uint64_t key = ((uint64_t)cand[e] << 32) | (key_id(kept[r]) * (uint32_t)W2 + (e - r * W2));
                if (cand[e] != 0xFFFFFFFFu && (t == 0 || key > last)) m = min(m, key);
            }
            m = warp_min64(m);
            if (lane == 0) keys[t] = m;
            last = m;
            if (m == kEmptyKey) {
                for (int q = t + lane; q < 32; q += 32) keys[q] = kEmptyKey;
                break;
            }
        }
    }
    __syncwarp();
    // the lists in that order
    const uint64_t key = keys[lane];
    int a0 = 0, len = 0;
    if (key != kEmptyKey) {
        a0 = off[key_id(key)];
        len = min(off[key_id(key) + 1] - a0, s);
    }
    int end = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += y;
    }
    int32_t* out = S + qi * s;
    for (int t = 0, p = end - len; t < len && p < s; ++t, ++p) out[p] = ids[a0 + t];
    const int all = __shfl_sync(0xffffffffu, end, 31);
    for (int p = all + lane; p < s; p += 32) out[p] = -1;
}

int grid_for_count(int64_t count) {
    const int64_t g = (count + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 16));
}

}  // namespace

// ---------------------------------------------------------------- launchers
void launch_rvq_assign(const float* X, int64_t N, int D, const float* W1, const int32_t* c1, int c1_stride,
                       const float* words, int W, int32_t* out, int out_stride, cudaStream_t s) {
    if (N <= 0) return;
    const size_t smem = assign_smem(D);
    const int64_t grid = (N + kAR - 1) / kAR;
    const bool res = W1 != nullptr;
    LaunchScope ls(res ? "k9_assign_res" : "k9_assign", s, (double)N * D * (res ? 8.0 : 4.0) + N * 4.0,
                   (double)N * W * D * 3.0);
    if (res) {
        allow_smem(k9_assign<true>);
        k9_assign<true><<<(unsigned)grid, kAT, smem, s>>>(X, N, D, W1, c1, c1_stride, words, W, out, out_stride);
    } else {
        allow_smem(k9_assign<false>);
        k9_assign<false><<<(unsigned)grid, kAT, smem, s>>>(X, N, D, nullptr, nullptr, 0, words, W, out, out_stride);
    }
}

int digit_sort_blocks(int64_t n) { return (int)std::max<int64_t>(1, (n + kDsTile - 1) / kDsTile); }

size_t digit_sort_hist_ints(int64_t n) { return (size_t)256 * digit_sort_blocks(n); }

void launch_digit_sort(const int32_t* in, int64_t n, const int32_t* key, int kstride, int32_t* out, int32_t* hist,
                       int32_t* gofs, int32_t* scan_tmp, cudaStream_t s) {
    const int nb = digit_sort_blocks(n);
    {
        LaunchScope ls("k9_digit_hist", s, n * (in ? 8.0 : 4.0) + 256.0 * nb * 4, 0);
        k9_digit_hist<<<nb, kDsThreads, 0, s>>>(in, n, key, kstride, hist, nb);
    }
    launch_scan(hist, gofs, (int64_t)256 * nb, scan_tmp, s);
    LaunchScope ls("k9_digit_scatter", s, n * (in ? 12.0 : 8.0) + 256.0 * nb * 4, 0);
    k9_digit_scatter<<<nb, kDsThreads, 0, s>>>(in, n, key, kstride, gofs, nb, out);
}

size_t rvq_update_doubles(int64_t N, int D) { return (size_t)((N + kUpRows - 1) / kUpRows + 256) * 2 * D; }

void launch_rvq_update(const float* X, int64_t N, int D, const int32_t* order, const int32_t* gofs, int nb, int W,
                       double* part, float* words, cudaStream_t s) {
    LaunchScope ls("k9_update", s, (double)N * D * 4.0 + N * 4.0, (double)N * D, 2);
    const int64_t units = (N + kUpRows - 1) / kUpRows;
    const dim3 grid((unsigned)((units + 3) / 4), (unsigned)((D + kUpDims - 1) / kUpDims));
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    if (part && vec) k9_pieces<true><<<grid, 128, 0, s>>>(X, N, D, order, gofs, nb, W, part);
    if (part && !vec) k9_pieces<false><<<grid, 128, 0, s>>>(X, N, D, order, gofs, nb, W, part);
    k9_combine<<<(unsigned)(W * ((D + 127) / 128)), 128 * kCbGroups, 0, s>>>(X, N, D, order, gofs, nb, W, part,
                                                                             words);
}

void launch_rvq_init(const float* X, int D, const int64_t* pos, int W, float* words, cudaStream_t s) {
    LaunchScope ls("k9_init_words", s, (double)W * D * 8.0, 0);
    k9_init_words<<<grid_for_count((int64_t)W * D), 256, 0, s>>>(X, D, pos, W, words);
}

void launch_rvq_residues(const float* X, int64_t N, int D, const float* W1, const int32_t* c1, float* R,
                         cudaStream_t s) {
    if (N <= 0) return;
    LaunchScope ls("k9_residues", s, (double)N * D * 12.0 + N * 4.0, (double)N * D);
    k9_residues<<<grid_for_count(N * D), 256, 0, s>>>(X, N, D, W1, c1, R);
}

void launch_rvq_key_count(const int32_t* codes, int64_t n, int W2, int32_t* cnt, cudaStream_t s) {
    if (n <= 0) return;
    LaunchScope ls("k9_key_count", s, n * 12.0, 0);
    k9_key_count<<<grid_for_count(n), 256, 0, s>>>(codes, n, W2, cnt);
}

void launch_check_offsets(const int32_t* off, int64_t nk, int64_t n, int* status, cudaStream_t s) {
    LaunchScope ls("k9_check_offsets", s, (nk + 1) * 4.0, 0);
    k9_check_offsets<<<grid_for_count(nk + 1), 256, 0, s>>>(off, nk, n, status);
}

void launch_rvq_tables(const float* w1, int W1, const float* w2, int W2, int D, float* n1, float* n2, float* x12,
                       float* w1T, float* w2T, cudaStream_t s) {
    LaunchScope ls("k9_tables", s, (double)(W1 + W2) * D * 12.0 + (double)W1 * W2 * 4.0,
                   (double)(W1 + 1) * (W2 + 1) * D * 2.0);
    k9_tables<<<grid_for_count((int64_t)W1 * W2), 256, 0, s>>>(w1, W1, w2, W2, D, n1, n2, x12, w1T, w2T);
}

// Where few keys are ranked over short words, the general route's two launches
// cost less than this one's five (us, 100 queries): 16 words of
// one dim in both stages 89 and 102, 64 of 16 dims and one kept word 90 and 105,
// 256 of 128 dims 169 and 115; 3,000 queries are even.
bool rvq_few_seeds(int W1, int W2, int D, int64_t m, int probe1, int s_seeds) {
    return s_seeds <= kSeedFew && (probe1 * W2 > 256 || (int64_t)(W1 + W2) * D > 8192 || m > 4096);
}

int64_t rvq_seed_batch(int64_t m) { return std::min<int64_t>(m, 65536); }

namespace {
void launch_dots(const float* A, int64_t M, const float* B, int W, int D, float* out, float* self, cudaStream_t s) {
    LaunchScope ls("k9_dots", s, ((double)M + W) * D * 4.0 + (double)M * W * 4.0, (double)M * W * D * 2.0);
    const dim3 grid((unsigned)((M + kDotRows - 1) / kDotRows), (unsigned)((W + kDotCols - 1) / kDotCols));
    const size_t smem = (size_t)(kDotRows + kDotCols) * kDotStride * 4;
    if (D % 4 == 0 && ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0) {
        allow_smem(k9_dots<true>);
        k9_dots<true><<<grid, 256, smem, s>>>(A, M, B, W, D, out, self);
    } else {
        allow_smem(k9_dots<false>);
        k9_dots<false><<<grid, 256, smem, s>>>(A, M, B, W, D, out, self);
    }
}
}  // namespace

void launch_rvq_few_seeds(const float* w1, int W1, const float* w2, int W2, int D, const int32_t* off,
                          const int32_t* ids, const float* Q, int64_t m, int probe1, int s_seeds,
                          const SeedWork& w, int32_t* S, const int* status, cudaStream_t s) {
    const int W = W1 + W2;
    {
        LaunchScope ls("k9_stack", s, (double)W * D * 8.0, 0);
        k9_stack<<<grid_for_count((int64_t)W * D), 256, 0, s>>>(w1, (int64_t)W1 * D, w2, (int64_t)W2 * D, w.words);
    }
    launch_dots(w.words, W, w.words, W, D, w.table, w.self, s);
    {
        LaunchScope ls("k9_keys", s, (double)W1 * W2 * 16.0, 0);
        k9_keys<<<grid_for_count((int64_t)W1 * W2), 256, 0, s>>>(w.table, w.self, W1, W2, off, w.part, status);
    }
    const size_t smem = few_seeds_smem(probe1, W2);
    auto kernel = W2 % 4 == 0 ? k9_few_seeds<true> : k9_few_seeds<false>;
    allow_smem(kernel);
    const int64_t batch = rvq_seed_batch(m);
    for (int64_t q0 = 0; q0 < m; q0 += batch) {
        const int64_t c = std::min(batch, m - q0);
        launch_dots(Q + q0 * D, c, w.words, W, D, w.dots, w.qq, s);
        LaunchScope ls("k9_seeds", s, (double)c * (W * 4.0 + (double)probe1 * W2 * 4.0 + s_seeds * 8.0), 0);
        kernel<<<(unsigned)c, kFewT, smem, s>>>(w.dots, w.qq, w.self, W1, W2, probe1, w.part, off, ids, s_seeds,
                                                  S + q0 * s_seeds, status);
    }
}

int rvq_seed_keys(int probe1, int W2) {
    int P = kSdT;
    while (P < probe1 * W2) P <<= 1;
    return P;
}

size_t rvq_seeds_smem(int probe1, int W2, int D) { return seeds_smem(rvq_seed_keys(probe1, W2), D); }

void launch_rvq_seeds(const float* w1T, int W1, const float* w2T, int W2, int D, const float* n1, const float* n2,
                      const float* x12, const int32_t* off, const int32_t* ids, const float* Q, int64_t m, int probe1,
                      int s_seeds, int32_t* S, const int* status, cudaStream_t s) {
    if (m <= 0) return;
    const int P = rvq_seed_keys(probe1, W2);
    const size_t smem = seeds_smem(P, D);
    // algorithmic bytes: the query, both vocabularies (cached across queries,
    // counted once per query as a bound), the kept rows of w1.w2, the offsets
    // of the candidate keys and the seeds written
    LaunchScope ls("k9_seeds", s,
                   (double)m * (D * 4.0 + (double)(W1 + W2) * D * 4.0 + (double)probe1 * W2 * 12.0 + s_seeds * 8.0),
                   (double)m * (W1 + W2) * D * 2.0);
    allow_smem(k9_seeds);
    k9_seeds<<<(unsigned)m, kSdT, smem, s>>>(w1T, W1, w2T, W2, D, n1, n2, x12, off, ids, Q, probe1, P, s_seeds, S,
                                             status);
}

}  // namespace knng
