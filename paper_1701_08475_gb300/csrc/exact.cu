// exact.cu -- K7: the exact k nearest neighbours of sampled rows (the
// problem statement of Sec. 1, each sampled point as a query against the
// other n - 1), canonical FP32 distances, ties by id; recall of a graph on
// those rows; and the input check.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace knng {

namespace {

constexpr int kQR = 64;    // query rows per CTA
constexpr int kCT = 128;   // points per column tile
constexpr int kNT = 256;

__host__ __device__ inline void exact_chunk(int D, int* dch, int* stride) {
    const int d4 = (D + 3) & ~3;
    const int cap = (100 * 1024 / ((kQR + kCT) * 4) - 4) & ~3;
    const int c = d4 < cap ? d4 : cap;
    *dch = c;
    *stride = ((c / 4) & 1) ? c : c + 4;
}

// Query rows: row q is sample[q] (or row0 + q without a sample), q = list[r]
// when a list is given (*list_count of them).  gridDim.y > 1 splits the
// columns: split y writes its k best of list slot r to part, merged by
// k7_merge; with one split the lists go straight to out.
template <int NO>
__global__ void __launch_bounds__(kNT) k7_exact(const float* __restrict__ X, int64_t n, int D, int k,
                                               const int32_t* __restrict__ sample, int64_t row0, int64_t s_rows,
                                               const int32_t* __restrict__ list, const int* __restrict__ list_count,
                                               uint64_t* __restrict__ part, uint64_t* __restrict__ out,
                                               const int* __restrict__ status) {
    if (*status & kStatusStop) return;  // a sampled id failed its check
    if (list) s_rows = *list_count;
    if ((int64_t)blockIdx.x * kQR >= s_rows) return;
    extern __shared__ float4 smem4[];
    int dch, stride;
    exact_chunk(D, &dch, &stride);
    float* qs = reinterpret_cast<float*>(smem4);       // [kQR][stride]
    float* cs = qs + kQR * stride;                     // [kCT][stride]
    float* dt = cs + kCT * stride;                     // [kQR][kCT + 1]
    int64_t* qid = reinterpret_cast<int64_t*>(dt + kQR * (kCT + 1));  // [kQR]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = tid % 16, cg = tid / 16;
    const int64_t q0 = (int64_t)blockIdx.x * kQR;
    const int nq = (int)min((int64_t)kQR, s_rows - q0);
    for (int r = tid; r < kQR; r += kNT) {
        const int64_t q = r < nq ? (list ? (int64_t)list[q0 + r] : q0 + r) : -1;
        qid[r] = q < 0 ? -1 : sample ? (int64_t)sample[q] : row0 + q;
    }
    __syncthreads();
    const bool one_chunk = dch >= D;
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    auto load_rows = [&](float* dst, int rows, int64_t first, bool query, int d0) {
        const int dl = min(dch, D - d0);
        if (vec) {  // 16-byte pieces, a row's pieces by consecutive threads
            const int q4 = dch / 4;
            for (int e = tid; e < rows * q4; e += kNT) {
                const int r = e / q4, c = e - r * q4;
                const int64_t row = query ? qid[r] : first + r;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row >= 0 && row < n && 4 * c < dl)
                    v = __ldg(reinterpret_cast<const float4*>(X + row * D + d0) + c);
                *reinterpret_cast<float4*>(dst + r * stride + 4 * c) = v;
            }
            return;
        }
        for (int e = tid; e < rows * dch; e += kNT) {
            const int r = e / dch, dd = e - r * dch;
            const int64_t row = query ? qid[r] : first + r;
            float v = 0.f;
            if (row >= 0 && row < n && dd < dl) v = __ldg(X + row * D + d0 + dd);
            dst[r * stride + dd] = v;
        }
    };
    if (one_chunk) load_rows(qs, kQR, 0, true, 0);
    uint64_t run[8][NO];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr)
#pragma unroll
        for (int o = 0; o < NO; ++o) run[rr][o] = kEmptyKey;

    const int64_t tiles = (n + kCT - 1) / kCT;
    const int64_t t0 = tiles * blockIdx.y / gridDim.y, t1 = tiles * (blockIdx.y + 1) / gridDim.y;
    for (int64_t c0 = t0 * kCT; c0 < min(n, t1 * kCT); c0 += kCT) {
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        for (int d0 = 0; d0 < D; d0 += dch) {
            __syncthreads();
            if (!one_chunk) load_rows(qs, kQR, 0, true, d0);
            load_rows(cs, kCT, c0, false, d0);
            __syncthreads();
            const float* rp = qs + rg * stride;
            const float* cp = cs + cg * stride;
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
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) dt[(rg + 16 * i) * (kCT + 1) + cg + 16 * j] = acc[i][j];
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
            const int r = warp * 8 + rr;
            if (r >= nq) continue;
            uint64_t a[4 + NO];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int64_t col = c0 + lane + 32 * s;
                a[s] = (col < n && col != qid[r]) ? make_key(dt[r * (kCT + 1) + lane + 32 * s], (uint32_t)col)
                                                  : kEmptyKey;
            }
            uint64_t mine = run[rr][0];
#pragma unroll
            for (int o = 1; o < NO; ++o)
                if (o == ((k - 1) >> 5)) mine = run[rr][o];
            const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)mine, (k - 1) & 31);
            const uint32_t hi = __shfl_sync(0xffffffffu, (uint32_t)(mine >> 32), (k - 1) & 31);
            const uint64_t last = ((uint64_t)hi << 32) | lo;
            bool any = false;
#pragma unroll
            for (int s = 0; s < 4; ++s) any |= a[s] < last;
            if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
            for (int o = 0; o < NO; ++o) a[4 + o] = run[rr][o];
            sort_regs<4 + NO>(a);
            warp_select_unique<4 + NO, NO>(a, k, run[rr]);
        }
    }
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        const int r = warp * 8 + rr;
        if (r >= nq) continue;
#pragma unroll
        for (int o = 0; o < NO; ++o)
            if (lane + 32 * o < k) {
                uint64_t* dst = gridDim.y > 1 ? part + ((q0 + r) * gridDim.y + blockIdx.y) * k
                                              : out + (list ? (int64_t)list[q0 + r] : q0 + r) * k;
                dst[lane + 32 * o] = run[rr][o];
            }
    }
}

// One warp per list slot: the k best of its nsplit partial lists.
template <int NO>
__global__ void __launch_bounds__(256) k7_merge(const uint64_t* __restrict__ part, int nsplit, int k, int64_t s_rows,
                                               const int32_t* __restrict__ list, const int* __restrict__ list_count,
                                               uint64_t* __restrict__ out, const int* __restrict__ status) {
    if (*status & kStatusStop) return;
    if (list) s_rows = *list_count;
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= s_rows) return;
    const int lane = threadIdx.x & 31;
    uint64_t run[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) run[o] = kEmptyKey;
    for (int y = 0; y < nsplit; ++y) {
        uint64_t a[2 * NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            const int e = lane + 32 * o;
            a[o] = e < k ? part[(r * nsplit + y) * k + e] : kEmptyKey;
            a[NO + o] = run[o];
        }
        sort_regs<2 * NO>(a);
        warp_select_unique<2 * NO, NO>(a, k, run);
    }
    const int64_t q = list ? (int64_t)list[r] : r;
#pragma unroll
    for (int o = 0; o < NO; ++o)
        if (lane + 32 * o < k) out[q * k + lane + 32 * o] = run[o];
}

__global__ void k_recall(const int32_t* __restrict__ ids, const float* __restrict__ d,
                         const int32_t* __restrict__ gt_ids, const float* __restrict__ gt_d,
                         const int32_t* __restrict__ sample, int64_t s_rows, int k,
                         unsigned long long* __restrict__ counts) {
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= s_rows) return;
    const int lane = threadIdx.x & 31;
    const int64_t i = sample[r];
    const float kth = gt_d[r * k + k - 1];
    int hit = 0, tie = 0;
    for (int e = lane; e < k; e += 32) {
        const int32_t g = ids[i * k + e];
        if (g < 0) continue;
        for (int b = 0; b < k; ++b)
            if (gt_ids[r * k + b] == g) {
                ++hit;
                break;
            }
        tie += d[i * k + e] <= kth;
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        hit += __shfl_xor_sync(0xffffffffu, hit, m);
        tie += __shfl_xor_sync(0xffffffffu, tie, m);
    }
    if (lane == 0) {
        atomicAdd(&counts[0], (unsigned long long)hit);
        atomicAdd(&counts[1], (unsigned long long)tie);
    }
}

// Up to three arrays in one launch.  An array may start at any 4-byte boundary:
// its 16-byte aligned body is read as float4, the few values before and after
// it by the first CTA.
struct FiniteArgs {
    const float* p[3];
    int64_t count[3];
};
__global__ void k_check_finite(const FiniteArgs A, int* __restrict__ status) {
    bool bad = false;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        const int64_t count = A.count[u];
        if (count == 0) continue;
        const float* X = A.p[u];
        const int64_t to16 = (int64_t)((16 - (reinterpret_cast<uintptr_t>(X) & 15)) & 15) / 4;
        const int64_t head = to16 < count ? to16 : count, n4 = (count - head) / 4;
        const float4* X4 = reinterpret_cast<const float4*>(X + head);
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n4;
             e += (int64_t)gridDim.x * blockDim.x) {
            const float4 v = __ldg(X4 + e);
            bad |= !isfinite(v.x) | !isfinite(v.y) | !isfinite(v.z) | !isfinite(v.w);
        }
        if (blockIdx.x == 0) {
            const int64_t t = threadIdx.x;
            if (t < head) bad |= !isfinite(X[t]);
            if (head + 4 * n4 + t < count) bad |= !isfinite(X[head + 4 * n4 + t]);
        }
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(status, kStatusNonFinite);
}

}  // namespace

int exact_splits(int64_t n, int64_t s_rows) {
    // one CTA fits an SM at D >= 128: two waves of CTAs, at least 8 column tiles each
    const int64_t rt = (s_rows + kQR - 1) / kQR, tiles = (n + kCT - 1) / kCT;
    return (int)std::max<int64_t>(1, std::min<int64_t>({(2 * 152 + rt - 1) / rt, tiles / 8, 32}));
}

void launch_exact(const float* X, int64_t n, int D, int k, const int32_t* sample, int64_t row0, int64_t s_rows,
                  const int32_t* list, const int* list_count, int nsplit, uint64_t* part, uint64_t* out,
                  const int* status, cudaStream_t s) {
    int dch, stride;
    exact_chunk(D, &dch, &stride);
    const size_t smem = (size_t)(kQR + kCT) * stride * 4 + (size_t)kQR * (kCT + 1) * 4 + kQR * 8;
    const dim3 grid((unsigned)((s_rows + kQR - 1) / kQR), (unsigned)nsplit);
    // rows taken from a list: how many is known on the device only
    LaunchScope ls("k7_exact", s, list ? 0.0 : (double)grid.x * n * D * 4.0, list ? 0.0 : (double)s_rows * n * 3.0 * D,
                   nsplit > 1 ? 2 : 1);
    const int mgrid = (int)((s_rows * 32 + 255) / 256);
    if (k > 32) {
        allow_smem(k7_exact<2>);
        k7_exact<2><<<grid, kNT, smem, s>>>(X, n, D, k, sample, row0, s_rows, list, list_count, part, out, status);
        if (nsplit > 1)
            k7_merge<2><<<mgrid, 256, 0, s>>>(part, nsplit, k, s_rows, list, list_count, out, status);
    } else {
        allow_smem(k7_exact<1>);
        k7_exact<1><<<grid, kNT, smem, s>>>(X, n, D, k, sample, row0, s_rows, list, list_count, part, out, status);
        if (nsplit > 1)
            k7_merge<1><<<mgrid, 256, 0, s>>>(part, nsplit, k, s_rows, list, list_count, out, status);
    }
}

void launch_recall(const int32_t* ids, const float* d, const int32_t* gt_ids, const float* gt_d,
                   const int32_t* sample, int64_t s_rows, int k, unsigned long long* counts, cudaStream_t s) {
    LaunchScope ls("k_recall", s, (double)s_rows * k * 16.0, 0);
    cudaMemsetAsync(counts, 0, 2 * sizeof(unsigned long long), s);
    if (s_rows == 0) return;
    const int grid = (int)((s_rows * 32 + 255) / 256);
    k_recall<<<grid, 256, 0, s>>>(ids, d, gt_ids, gt_d, sample, s_rows, k, counts);
}

void launch_check_finite(const float* X, int64_t count, int* status, cudaStream_t s, const float* Y, int64_t ycount,
                         const float* Z, int64_t zcount) {
    FiniteArgs A = {{X, Y, Z}, {count, ycount, zcount}};
    const int64_t total = count + ycount + zcount;
    LaunchScope ls("k0_check_finite", s, total * 4.0, 0);
    const int64_t grid = (total / 4 + 255) / 256;
    k_check_finite<<<(int)(grid < 1 ? 1 : grid < 152 * 8 ? grid : 152 * 8), 256, 0, s>>>(A, status);
}

}  // namespace knng
