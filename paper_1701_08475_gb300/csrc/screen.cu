// screen.cu -- exact nearest neighbours found by tensor-core screening: a
// BF16 Gram matrix (tcgen05, TMA-fed, FP32 accumulators in tensor memory)
// says which columns can matter to a row, and only those get their canonical
// FP32 distance.  The error bound makes the result the plain FP32 form's, bit
// for bit; a row the bound cannot serve goes to the FP32 kernel.
//
//   exact lists (Sec. 1)      rows = sampled points, columns = all points
//   nearest word (Sec. 4.1)   rows = vectors, columns = up to 256 words
//
// Bound.  x^ is the BF16 copy, e = ||x - x^|| (rounded up), N = ||x^||^2, g the
// computed x^_i . x^_j.  For the distance d of the FP32 points,
//   |sqrt(d) - sqrt(d~)| <= e_i + e_j        (d~: exact distance of x^)
//   |N_i + N_j - 2 g - d~| <= cD (||x^_i|| + ||x^_j||)^2 <= 2 cD (N_i + N_j)
// with cD the leaf certificate's coefficient, and the canonical FP32 distance
// is within a factor 1 +- gamma, gamma = (D + 8) 2^-23, of d.  A column whose
// canonical distance is at most tau therefore has
//   c_j - 2 g - 2 a_i e_j <= R_i,  c_j = N_j (1 - c) - e_j^2,
//   a_i = sqrt(tau (1 + gamma)) + e_i,  R_i = a_i^2 + N_i (c - 1)
// where c = 2 cD + 2^-19 also covers the test's own FP32 roundings.  When the
// data are integers that BF16 holds exactly (the leaf stage's exactness
// flag), every quantity is an exact integer and e, c and gamma are 0.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace knng {

namespace {

constexpr int kScM = 128;          // rows of a tile (tensor-memory lanes)
constexpr int kScN = 256;          // columns of a tile
constexpr int kScK = 64;           // BF16 elements per 128-byte swizzled row
constexpr int kScStages = 4;
constexpr int kScABytes = kScM * 128, kScBBytes = kScN * 128;
constexpr int kScResident = 4;     // K chunks up to which a row tile stays in shared memory
constexpr int kScEpi = 512;        // epilogue threads: 16 warps, four per tensor-memory quarter
constexpr int kScPart = kScN / 4;  // columns per epilogue warp
constexpr int kScThreads = 64 + kScEpi;  // + a TMA warp and an MMA warp
constexpr int kScGrid = 152;       // one CTA per SM (512 tensor-memory columns, over half of shared memory)
constexpr int kScCand = 2048;      // candidates buffered in shared memory (collect)
constexpr float kScTiny = 1e-17f;  // added to e: squares below FP32's range summed as zero

enum ScreenMode { kScDump = 0, kScCollect = 1, kScArgmin = 2 };

struct ScreenArgs {
    int nk;                // K chunks
    int64_t nrows, ncols;  // rows and columns of the product
    int nrt, nct, nstripe;
    // per row (original row of row r: rid ? rid[r] : rid0 + r)
    const float* rnrm;     // [nrows]
    const float* rerr;
    // per column: column j is row j * cstride of these
    const float* cnrm;
    const float* cerr;
    int64_t cstride;
    float cD2, gamma;      // 2 cD + 2^-19; (D + 8) 2^-23
    const int* flag_r;     // exactness flags of the two operands (may be equal)
    const int* flag_c;
    int* status;
    // dump / collect
    const int32_t* rid;
    int64_t rid0;
    int cap;               // candidates kept per row
    float* cg;             // [nrows][cap] g
    int32_t* cid;          // [nrows][cap] original row of the column (collect)
    int32_t* cnt;          // [nrows]
    const float* rowA;     // [nrows] a_i
    const float* rowR;     // [nrows] R_i
    uint32_t* mask;        // nearest word: [nrows][8] the candidate words of each row
    // re-rank
    const float* X;
    int D;
    bool vec;
};

// The flag bits of the copy (k0_quantize's) plus 8: some squared norm is too
// large for the bound's arithmetic.
__device__ __forceinline__ bool sc_exact(int f) { return (f & 9) == 0 && !((f & 2) && (f & 4)); }

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// Barrier of the epilogue warps; true when every thread passed true.
__device__ __forceinline__ bool epi_all(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 p, %1, 0;\n"
        "barrier.cta.red.and.pred q, 1, 512, p;\n"
        "selp.u32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(r)
        : "r"((uint32_t)ok)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("barrier.cta.sync 1, 512;\n" ::: "memory"); }

struct ScreenSmem {
    size_t a_off, col_off, list_off, row_off, bar_off, total;
    int stage_bytes;
};
__host__ __device__ inline ScreenSmem screen_smem(int nk, int mode) {
    ScreenSmem L;
    const bool res = nk <= kScResident;
    L.stage_bytes = kScBBytes + (res ? 0 : kScABytes);
    L.a_off = (size_t)kScStages * L.stage_bytes;
    L.col_off = L.a_off + (res ? (size_t)nk * kScABytes : 0);
    L.list_off = L.col_off + (mode == kScCollect ? kScEpi / 32 * kScPart : 2 * kScN) * 8;
    L.row_off = L.list_off + (mode == kScCollect ? kScCand * 12 : 0);
    L.bar_off = L.row_off + (mode == kScArgmin ? 2 * 4 * kScM * 4 : 0);
    L.total = L.bar_off + (2 * kScStages + 6) * 8 + 32;
    return L;
}

// The canonical distance of a point to one staged in shared memory.
__device__ __forceinline__ float point_dist(const float* __restrict__ x, const float* q, int D, bool vec) {
    float acc = 0.f;
    if (vec) {
        for (int d = 0; d < D; d += 4) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(x + d));
            const float4 b = *reinterpret_cast<const float4*>(q + d);
            float t = __fsub_rn(a.x, b.x);
            acc = __fmaf_rn(t, t, acc);
            t = __fsub_rn(a.y, b.y);
            acc = __fmaf_rn(t, t, acc);
            t = __fsub_rn(a.z, b.z);
            acc = __fmaf_rn(t, t, acc);
            t = __fsub_rn(a.w, b.w);
            acc = __fmaf_rn(t, t, acc);
        }
        return acc;
    }
    for (int d = 0; d < D; ++d) {
        const float t = __fsub_rn(__ldg(x + d), q[d]);
        acc = __fmaf_rn(t, t, acc);
    }
    return acc;
}

// c_j - 2 g_j - 2 a e_j of two columns (a2 = -2 a), with paired FP32 FMAs.
__device__ __forceinline__ float2 screen_pair(float g0, float g1, float c0, float c1, float e0, float e1, float a2) {
    float2 r;
    asm("{\n"
        ".reg .b64 g, c, e, m, a;\n"
        "mov.b64 g, {%2, %3};\n"
        "mov.b64 c, {%4, %5};\n"
        "mov.b64 e, {%6, %7};\n"
        "mov.b64 m, {%8, %8};\n"
        "mov.b64 a, {%9, %9};\n"
        "fma.rn.f32x2 c, m, g, c;\n"
        "fma.rn.f32x2 c, a, e, c;\n"
        "mov.b64 {%0, %1}, c;\n"
        "}\n"
        : "=f"(r.x), "=f"(r.y)
        : "f"(g0), "f"(g1), "f"(c0), "f"(c1), "f"(e0), "f"(e1), "f"(-2.f), "f"(a2));
    return r;
}
// c_j - 2 g_j of two columns.
__device__ __forceinline__ float2 fma_pair(float g0, float g1, float c0, float c1) {
    float2 r;
    asm("{\n"
        ".reg .b64 g, c, m;\n"
        "mov.b64 g, {%2, %3};\n"
        "mov.b64 c, {%4, %5};\n"
        "mov.b64 m, {%6, %6};\n"
        "fma.rn.f32x2 c, m, g, c;\n"
        "mov.b64 {%0, %1}, c;\n"
        "}\n"
        : "=f"(r.x), "=f"(r.y)
        : "f"(g0), "f"(g1), "f"(c0), "f"(c1), "f"(-2.f));
    return r;
}
__device__ __forceinline__ float min_pair(float2 p, float m) {
    float r;
    asm("min.f32 %0, %1, %2, %3;\n" : "=f"(r) : "f"(p.x), "f"(p.y), "f"(m));
    return r;
}

// An upper bound of the canonical distance of (i, j) from the copies.
__device__ __forceinline__ float screen_ub(float ni, float nj, float g, float ei, float ej, float c, float gamma) {
    const float s = __fadd_ru(ni, nj);
    const float d = __fadd_ru(__fmaf_ru(-2.f, g, s), __fmul_ru(c, s));
    const float r = __fadd_ru(__fsqrt_ru(fmaxf(d, 0.f)), __fadd_ru(ei, ej));
    return __fmul_ru(__fmul_ru(r, r), __fadd_ru(1.f, gamma));
}

// a_i and R_i of a row whose candidates must have canonical distance <= tau.
__device__ __forceinline__ void screen_row(float tau, float ni, float ei, float c, float gamma, bool exact, float& a,
                                           float& R) {
    if (exact) {
        a = 0.f;
        R = __fsub_rn(tau, ni);  // exact integers
        return;
    }
    a = __fadd_ru(__fsqrt_ru(__fmul_ru(tau, __fadd_ru(1.f, gamma))), ei);
    R = __fadd_ru(__fmaf_ru(__fmul_ru(a, a), 1.f + 1.9073486328125e-6f, 1e-30f), __fmul_ru(ni, c - 1.f));
}

// Persistent, warp-specialised screening product: warp 0 issues the TMA loads,
// warp 1 the MMAs (128 x 256 tiles, two accumulators in tensor memory), warps
// 2-17 read finished accumulators (64 columns of 32 rows each; fewer, wider
// warps left the issue slots a third used).  A unit is one row tile against every
// nstripe-th column tile, and units of consecutive row tiles run side by side,
// so that a column tile is read from DRAM once and then from L2.  With up to
// kScResident chunks of K the row tile stays in shared memory for the unit.
template <int MODE>
__global__ void __launch_bounds__(kScThreads, 1) ks_screen(const __grid_constant__ CUtensorMap tma,
                                                          const __grid_constant__ CUtensorMap tmb,
                                                          const ScreenArgs P) {
    extern __shared__ uint8_t smem_raw[];
    if (tc::stopped(P.status)) return;  // whole CTA, before any other barrier or tensor memory
    const ScreenSmem L = screen_smem(P.nk, MODE);
    uint8_t* base = smem_raw + ((1024 - (tc::smem_addr(smem_raw) & 1023)) & 1023);
    const bool res = P.nk <= kScResident;
    float2* colc = reinterpret_cast<float2*>(base + L.col_off);  // (c_j, e_j): [2][kScN], or per warp
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + L.bar_off);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kScStages + 6);
    int* ncand = reinterpret_cast<int*>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t full0 = tc::smem_addr(bars), empty0 = full0 + 8 * kScStages;
    const uint32_t afull = empty0 + 8 * kScStages, aempty = afull + 8, tfull0 = aempty + 8, tempty0 = tfull0 + 16;
    const int nk = P.nk;
    const int units = P.nrt * P.nstripe;

    if (tid == 0) {
        for (int s = 0; s < 2 * kScStages; ++s) tc::mbar_init(full0 + 8 * s, 1);
        tc::mbar_init(afull, 1);
        tc::mbar_init(aempty, 1);
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(tfull0 + 8 * b, 1);
            tc::mbar_init(tempty0 + 8 * b, kScEpi / 32);
        }
        tc::mbar_fence_init();
        ncand[0] = ncand[1] = 0;
    }
    if (warp == 1) {
        tc::tmem_alloc(tc::smem_addr(tmem_slot), 2 * kScN);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int it = 0, uu = 0;
            for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++uu) {
                const int rt = u % P.nrt;
                if (res) {
                    if (!(ok = tc::mbar_wait(aempty, (uint32_t)((uu & 1) ^ 1), P.status))) break;
                    tc::mbar_expect_tx(afull, (uint32_t)(nk * kScABytes));
                    for (int c = 0; c < nk; ++c)
                        tc::tma_load_2d(tc::smem_addr(base + L.a_off + (size_t)c * kScABytes), &tma, c * kScK,
                                        rt * kScM, afull);
                }
                for (int ct = u / P.nrt; ok && ct < P.nct; ct += P.nstripe)
                    for (int c = 0; c < nk; ++c, ++it) {
                        const int s = it % kScStages;
                        if (!(ok = tc::mbar_wait(empty0 + 8 * s, (uint32_t)(((it / kScStages) & 1) ^ 1), P.status)))
                            break;
                        const uint32_t fb = full0 + 8 * s, st = tc::smem_addr(base + (size_t)s * L.stage_bytes);
                        tc::mbar_expect_tx(fb, (uint32_t)L.stage_bytes);
                        tc::tma_load_2d(st, &tmb, c * kScK, ct * kScN, fb);
                        if (!res) tc::tma_load_2d(st + kScBBytes, &tma, c * kScK, rt * kScM, fb);
                    }
            }
            if (!ok) {  // let the loads still in flight land before the CTA can exit
                if (res && uu > 0) tc::mbar_wait(afull, (uint32_t)((uu - 1) & 1), P.status);
                for (int j = std::max(0, it - kScStages); j < it; ++j)
                    tc::mbar_wait(full0 + 8 * (j % kScStages), (uint32_t)((j / kScStages) & 1), P.status);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            bool ok = true;
            int it = 0, uu = 0, t = 0;
            const uint32_t idesc = tc::idesc_f16(true, kScM, kScN);
            for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++uu) {
                if (res && !(ok = tc::mbar_wait(afull, (uint32_t)(uu & 1), P.status))) break;
                for (int ct = u / P.nrt; ok && ct < P.nct; ct += P.nstripe, ++t) {
                    const int buf = t & 1;
                    if (!(ok = tc::mbar_wait(tempty0 + 8 * buf, (uint32_t)(((t >> 1) & 1) ^ 1), P.status))) break;
                    tc::fence_after_sync();
                    const uint32_t acc = tmem + (uint32_t)(buf * kScN);
                    for (int c = 0; c < nk; ++c, ++it) {
                        const int s = it % kScStages;
                        if (!(ok = tc::mbar_wait(full0 + 8 * s, (uint32_t)((it / kScStages) & 1), P.status))) break;
                        tc::fence_after_sync();
                        const uint32_t st = tc::smem_addr(base + (size_t)s * L.stage_bytes);
                        const uint64_t db = tc::sdesc_k128(st);
                        const uint64_t da = tc::sdesc_k128(
                            res ? tc::smem_addr(base + L.a_off + (size_t)c * kScABytes) : st + kScBBytes);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            tc::mma_f16(acc, da + 2 * kk, db + 2 * kk, idesc, (c | kk) != 0);
                        tc::mma_commit(empty0 + 8 * s);
                    }
                    if (ok) tc::mma_commit(tfull0 + 8 * buf);
                }
                if (ok && res) tc::mma_commit(aempty);
            }
        }
    } else {
        const int et = tid - 64;                 // epilogue thread
        const int qd = warp & 3;                 // tensor-memory quarter this warp may read
        const int part = (warp - 2) >> 2;        // columns kScPart part .. of the tile
        const int rl = qd * 32 + lane;           // row of the tile
        const int fr = *P.flag_r, fc = *P.flag_c;
        const bool exact = sc_exact(fr | fc), unsafe = ((fr | fc) & 8) != 0;
        const float c2 = exact ? 0.f : P.cD2, gamma = exact ? 0.f : P.gamma;
        // collect: candidates of the CTA, flushed to the rows' lists
        int32_t* brow = reinterpret_cast<int32_t*>(base + L.list_off);
        int32_t* bid = brow + kScCand;
        float* bg = reinterpret_cast<float*>(bid + kScCand);
        // nearest word: the words' c_j, then e_j, then N_j (1 + c) rounded up
        // (one column tile, loaded once), the greatest e_j, and each part's
        // least value of a row
        float* colf = reinterpret_cast<float*>(colc);
        uint32_t* cmax = reinterpret_cast<uint32_t*>(ncand);
        float* hmin = reinterpret_cast<float*>(base + L.row_off);  // [2][4][kScM]
        int t = 0;
        auto col_const = [&](int64_t col) -> float2 {
            if (col >= P.ncols) return make_float2(__int_as_float(0x7f800000), 0.f);
            const float nj = __ldg(P.cnrm + col * P.cstride);
            if (exact) return make_float2(nj, 0.f);
            const float ej = __ldg(P.cerr + col * P.cstride);
            return make_float2(__fsub_rd(__fmul_rd(nj, 1.f - c2), __fmul_ru(ej, ej)), ej);
        };
        float* wcol = reinterpret_cast<float*>(colc + (warp - 2) * kScPart);  // collect: this warp's c_j, then e_j
        float2 next_col[2];
        auto load_cols = [&](int ct) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
                next_col[q] = col_const((int64_t)ct * kScN + part * kScPart + 32 * q + lane);
        };
        auto append = [&](int64_t row, int64_t own, int64_t id, float g) {
            if (id == own) return;
            const int at = atomicAdd(ncand, 1);
            if (at < kScCand) {
                brow[at] = (int32_t)row;
                bid[at] = (int32_t)id;
                bg[at] = g;
                return;
            }
            // the buffer is full: straight to the row's list
            const int pos = atomicAdd(P.cnt + row, 1);
            if (pos < P.cap) {
                P.cid[row * P.cap + pos] = (int32_t)id;
                P.cg[row * P.cap + pos] = g;
            }
        };
        auto flush = [&](int n) {  // every epilogue thread, uniform n
            n = min(n, kScCand);
            for (int e = et; e < n; e += kScEpi) {
                const int64_t r = brow[e];
                const int pos = atomicAdd(P.cnt + r, 1);
                if (pos < P.cap) {
                    P.cid[r * P.cap + pos] = bid[e];
                    P.cg[r * P.cap + pos] = bg[e];
                }
            }
            epi_sync();
            if (et == 0) *ncand = 0;
            epi_sync();
        };
        if (blockIdx.x < (unsigned)units && MODE == kScCollect) load_cols(blockIdx.x / P.nrt);
        if (MODE == kScArgmin) {
            if (et < kScN) {
                const float2 c = col_const(et);
                colf[et] = c.x;
                colf[kScN + et] = c.y;
                colf[2 * kScN + et] = et < P.ncols ? __fmul_ru(__ldg(P.cnrm + et), __fadd_ru(1.f, c2)) : c.x;
                if (et < P.ncols) atomicMax(cmax, __float_as_uint(c.y));  // at least 0: its bits have its order
            }
            epi_sync();
        }
        bool ok = true;
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
            const int rt = u % P.nrt;
            const int64_t row = (int64_t)rt * kScM + rl;
            const bool live = row < P.nrows;
            float a2 = 0.f, R = __int_as_float(0xff800000), ni = 0.f, ei = 0.f;
            int64_t own = -1;
            if (live) {
                ni = __ldg(P.rnrm + row);
                ei = exact ? 0.f : __ldg(P.rerr + row);
                if (MODE == kScCollect) {
                    a2 = -2.f * P.rowA[row];
                    R = P.rowR[row];
                    own = P.rid ? (int64_t)P.rid[row] : P.rid0 + row;
                }
            }
            for (int ct = u / P.nrt; ct < P.nct; ct += P.nstripe, ++t) {
                const int buf = t & 1;
                if (MODE == kScCollect) {
                    // the warp's own copy of its columns' constants: the
                    // warps share nothing per tile, so one that appends
                    // candidates holds no other back
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        wcol[32 * q + lane] = next_col[q].x;
                        wcol[kScPart + 32 * q + lane] = next_col[q].y;
                    }
                    __syncwarp();
                    // the next tile's load while this one is read
                    int nct = ct + P.nstripe;
                    if (nct >= P.nct) nct = u + gridDim.x < units ? (int)(u + gridDim.x) / P.nrt : -1;
                    if (nct >= 0) load_cols(nct);
                }
                ok = tc::mbar_wait_warp(tfull0 + 8 * buf, (uint32_t)((t >> 1) & 1), P.status);
                if (MODE == kScArgmin) ok = epi_all(ok);  // the waits end for all warps or for none
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t taddr =
                    tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(buf * kScN + part * kScPart);
                if (MODE == kScDump) {
#pragma unroll 1
                    for (int b = 0; b < kScPart / 32; ++b) {
                        float v[32];
                        tc::tmem_ld_32(taddr + b * 32, v);
                        const int64_t col0 = (int64_t)ct * kScN + part * kScPart + b * 32;
                        if (live) {
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                if (col0 + 4 * q < P.ncols)  // cap is a multiple of 4 past the last column
                                    *reinterpret_cast<float4*>(P.cg + row * P.cap + col0 + 4 * q) =
                                        make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                        }
                    }
                } else if (MODE == kScCollect) {
#pragma unroll 1  // one copy of the code: it stays within the instruction cache
                    for (int b = 0; b < kScPart / 32; ++b) {
                        float v[32];
                        tc::tmem_ld_32(taddr + b * 32, v);
                        if (b == kScPart / 32 - 1) {  // the last of it is in registers: hand the accumulator back
                            tc::fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
                        }
                        // two columns per instruction where there is one
                        const float4* c4 = reinterpret_cast<const float4*>(wcol + b * 32);
                        const float4* e4 = reinterpret_cast<const float4*>(wcol + kScPart + b * 32);
                        float mn = __int_as_float(0x7f800000);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 c = c4[q], e = e4[q];
                            mn = min_pair(screen_pair(v[4 * q], v[4 * q + 1], c.x, c.y, e.x, e.y, a2), mn);
                            mn = min_pair(screen_pair(v[4 * q + 2], v[4 * q + 3], c.z, c.w, e.z, e.w, a2), mn);
                        }
                        if (mn <= R) {  // few blocks hold a candidate
                            unsigned hit = 0;
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 c = c4[q], e = e4[q];
                                const float2 x = screen_pair(v[4 * q], v[4 * q + 1], c.x, c.y, e.x, e.y, a2);
                                const float2 y = screen_pair(v[4 * q + 2], v[4 * q + 3], c.z, c.w, e.z, e.w, a2);
                                if (x.x <= R) hit |= 1u << (4 * q);
                                if (x.y <= R) hit |= 2u << (4 * q);
                                if (y.x <= R) hit |= 4u << (4 * q);
                                if (y.y <= R) hit |= 8u << (4 * q);
                            }
                            for (; hit; hit &= hit - 1) {  // v[j] by a chain of selects
                                const int j = __ffs(hit) - 1;
                                float g = v[0];
#pragma unroll
                                for (int q = 1; q < 32; ++q) g = j == q ? v[q] : g;
                                append(row, own, ((int64_t)ct * kScN + part * kScPart + b * 32 + j) * P.cstride, g);
                            }
                        }
                        __syncwarp();
                    }
                } else {
                    // nearest word: the row's least upper bound of a distance
                    // gives tau; every word that could be within tau is a
                    // candidate
                    float va[32], vb[32];
                    tc::tmem_ld_issue(taddr, va);
                    tc::tmem_ld_issue(taddr + 32, vb);
                    tc::tmem_ld_wait(va);
                    tc::tmem_ld_wait(vb);
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
                    const float4* c4 = reinterpret_cast<const float4*>(colf + part * kScPart);
                    const float4* e4 = reinterpret_cast<const float4*>(colf + kScN + part * kScPart);
                    const float4* u4 = reinterpret_cast<const float4*>(colf + 2 * kScN + part * kScPart);
                    float mn = __int_as_float(0x7f800000);
                    auto least = [&](const float (&v)[32], int b) {
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 c = u4[8 * b + q];
                            mn = min_pair(fma_pair(v[4 * q], v[4 * q + 1], c.x, c.y), mn);
                            mn = min_pair(fma_pair(v[4 * q + 2], v[4 * q + 3], c.z, c.w), mn);
                        }
                    };
                    least(va, 0);
                    least(vb, 1);
                    hmin[(buf * 4 + part) * kScM + rl] = mn;
                    epi_sync();
#pragma unroll
                    for (int q = 0; q < 4; ++q) mn = fminf(mn, hmin[(buf * 4 + q) * kScM + rl]);
                    const float ee = __uint_as_float(cmax[0]);
                    float tau = __fadd_rn(ni, mn);
                    if (!exact) {  // mn: N_j (1 + c) - 2 g of some word, its own rounding covered by c's 2^-19
                        const float d = __fadd_ru(mn, __fmul_ru(ni, __fadd_ru(1.f, c2)));
                        const float r = __fadd_ru(__fsqrt_ru(fmaxf(d, 0.f)), __fadd_ru(ei, ee));
                        tau = __fmul_ru(__fmul_ru(r, r), __fadd_ru(1.f, gamma));
                    }
                    float a;
                    screen_row(tau, ni, ei, c2, gamma, exact, a, R);
                    a2 = -2.f * a;
                    auto hits = [&](const float (&v)[32], int b) {
                        unsigned hit = 0;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 c = c4[8 * b + q], e = e4[8 * b + q];
                            const float2 x = screen_pair(v[4 * q], v[4 * q + 1], c.x, c.y, e.x, e.y, a2);
                            const float2 y = screen_pair(v[4 * q + 2], v[4 * q + 3], c.z, c.w, e.z, e.w, a2);
                            if (x.x <= R) hit |= 1u << (4 * q);
                            if (x.y <= R) hit |= 2u << (4 * q);
                            if (y.x <= R) hit |= 4u << (4 * q);
                            if (y.y <= R) hit |= 8u << (4 * q);
                        }
                        return hit;
                    };
                    unsigned h0 = hits(va, 0), h1 = hits(vb, 1);
                    if (unsafe) h0 = h1 = 0xFFFFFFFFu;  // ks_pick drops the columns past the last word
                    if (live) *reinterpret_cast<uint2*>(P.mask + row * 8 + part * 2) = make_uint2(h0, h1);
                }
                if (MODE == kScDump) {  // the accumulator is read: hand it back
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
                }
            }
            if (MODE == kScCollect) {
                ok = epi_all(ok);  // every warp comes here, done with the unit or out of time
                if (!ok) break;
                const int n = *(volatile int*)ncand;
                epi_sync();
                if (n > kScCand / 2 || (n > 0 && u + gridDim.x >= units)) flush(n);
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem, 2 * kScN);
}

// ---------------------------------------------------------------- copies
// BF16 copy of N vectors (rows of X, gathered by perm when given, minus their
// stage-1 word when W1 is given), zero-padded to Dp, with squared norms, error
// bounds and the exactness flags of the leaf stage's k0_quantize plus 8: some
// squared norm is not below 1e30 (the bound's arithmetic could overflow).
// One warp takes 4 rows at once, so that 4 row pieces are in flight per lane.
// status (may be NULL): kStatusNonFinite when a value is not finite.
template <bool VEC>
__global__ void __launch_bounds__(256) ks_copy(const float* __restrict__ X, int64_t N, int D, int Dp,
                                              const float* __restrict__ W1, const int32_t* __restrict__ c1,
                                              int c1_stride, uint16_t* __restrict__ Xq, float* __restrict__ nrm,
                                              float* __restrict__ err, int* __restrict__ flags,
                                              int* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int64_t r0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 4;
    if (r0 >= N) return;
    float red[8];  // squared norms of rows 0-3, then squared errors
    float top = 0.f, low = 0.f;
    bool ints = true;
    int code[4] = {0, 0, 0, 0};
    if (W1) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (r0 + u < N) code[u] = c1[(r0 + u) * c1_stride];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) red[u] = 0.f;
    for (int d0 = lane * 4; d0 < Dp; d0 += 128) {
        float v[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[u][j] = 0.f;
            if (r0 + u < N) {
                const float* x = X + (r0 + u) * D + d0;
                if (VEC) {
                    if (d0 < D) {
                        const float4 f = __ldg(reinterpret_cast<const float4*>(x));
                        v[u][0] = f.x; v[u][1] = f.y; v[u][2] = f.z; v[u][3] = f.w;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (d0 + j < D) v[u][j] = __ldg(x + j);
                }
            }
        }
        if (W1) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (r0 + u < N) {
                    const float* w = W1 + (int64_t)code[u] * D + d0;
                    if (VEC) {
                        if (d0 < D) {
                            const float4 f = __ldg(reinterpret_cast<const float4*>(w));
                            v[u][0] = __fsub_rn(v[u][0], f.x);
                            v[u][1] = __fsub_rn(v[u][1], f.y);
                            v[u][2] = __fsub_rn(v[u][2], f.z);
                            v[u][3] = __fsub_rn(v[u][3], f.w);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (d0 + j < D) v[u][j] = __fsub_rn(v[u][j], __ldg(w + j));
                    }
                }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t h[2];
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                const float x = v[u][j], y = v[u][j + 1];
                const __nv_bfloat162 q = __floats2bfloat162_rn(x, y);
                h[j / 2] = *reinterpret_cast<const uint32_t*>(&q);
                const float b = __uint_as_float(h[j / 2] << 16), c = __uint_as_float(h[j / 2] & 0xFFFF0000u);
                red[u] = __fmaf_rn(b, b, red[u]);
                red[u] = __fmaf_rn(c, c, red[u]);
                const float s = __fsub_rn(x, b), t = __fsub_rn(y, c);  // exact: x and y rounded to fewer bits
                red[4 + u] = __fmaf_rn(s, s, red[4 + u]);
                red[4 + u] = __fmaf_rn(t, t, red[4 + u]);
                // whether a value of magnitude <= 256 is an integer: adding
                // 1.5 * 2^23 rounds it to one
                ints &= __fsub_rn(__fadd_rn(x, 12582912.f), 12582912.f) == x;
                ints &= __fsub_rn(__fadd_rn(y, 12582912.f), 12582912.f) == y;
                top = fmaxf(top, fmaxf(fabsf(x), fabsf(y)));
                low = fminf(low, fminf(x, y));
            }
            if (r0 + u < N) *reinterpret_cast<uint2*>(Xq + (r0 + u) * Dp + d0) = make_uint2(h[0], h[1]);
        }
    }
    // lanes 4 e .. 4 e + 3 end with the warp's sum of red[e]: each exchange
    // halves the sums a lane carries
#pragma unroll
    for (int st = 16, cnt = 4; st >= 4; st >>= 1, cnt >>= 1) {
        const bool hi = (lane & st) != 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u >= cnt) break;
            const float send = hi ? red[u] : red[u + cnt], keep = hi ? red[u + cnt] : red[u];
            red[u] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, st));
        }
    }
    float sum = red[0];
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    const int e = lane >> 2;  // 0-3: squared norms, 4-7: squared errors
    int f = 0;
    if (e < 4) f = (sum >= 8388608.f ? 1 : 0) | (sum >= 4194304.f ? 4 : 0) | (!(sum < 1e30f) ? 8 : 0);
    f |= ((!ints || !(top <= 256.f)) ? 1 : 0) | (low < 0.f ? 2 : 0);
    f = __reduce_or_sync(0xffffffffu, f);
    if ((lane & 3) == 0 && r0 + (e & 3) < N) {
        if (e < 4)
            nrm[r0 + e] = sum;
        else  // rounded up as in k0_quantize, plus what squares below the FP32 range could hide
            err[r0 + e - 4] = __fadd_ru(kScTiny, __fsqrt_ru(__fmul_ru(sum, 1.f + (float)(Dp + 8) * 5.9604645e-8f)));
    }
    // once set, a flag is only read: 250,000 warps' atomics on one word took
    // longer than the copy
    if (lane == 0 && (f & ~*(volatile int*)flags)) atomicOr(flags, f);
    if (status && (f & 8)) {  // a value that is not finite, or only a large norm?
        bool bad = false;
        for (int u = 0; u < 4 && r0 + u < N; ++u)
            for (int d = lane; d < D; d += 32) bad |= !isfinite(X[(r0 + u) * D + d]);
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kStatusNonFinite);
    }
}

// Rows perm[p] of a copy (q 16-byte pieces per row) with their norms and errors.
__global__ void __launch_bounds__(256) ks_gather(const uint4* __restrict__ Xq, const float* __restrict__ nrm,
                                                const float* __restrict__ err, int64_t n, int q,
                                                const int32_t* __restrict__ perm, uint4* __restrict__ out,
                                                float* __restrict__ onrm, float* __restrict__ oerr,
                                                const int* __restrict__ status) {
    if (*status & kStatusStop) return;  // a sampled id failed its check
    const int64_t total = n * q;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = e / q;
        const int c = (int)(e - p * q);
        const int64_t i = perm[p];
        out[e] = __ldg(Xq + i * q + c);
        if (c == 0) {
            onrm[p] = nrm[i];
            oerr[p] = err[i];
        }
    }
}

// ---------------------------------------------------------------- nearest words
// One warp per 32 rows: a row with one candidate word takes it; the others'
// (row, word) pairs are spread over the lanes, which compute canonical
// distances; ties go to the smaller word.  The rows and words of 32 pairs come
// to shared memory kPickDims dims at a time, a row's pieces side by side, and
// each lane walks its own pair there.  (A lane that walked its rows in global
// memory took a sector of its own per 16 bytes: the index of 30,000 x 960 in 64
// words, with 36 candidates a residue, 2.2 ms, staged 1.9; 1.4 with a word's own
// norm in its upper bound instead of the largest, which leaves fewer.)
constexpr int kPickPairs = 512;  // pairs a warp lists at once
constexpr int kPickWarps = 2, kPickDims = 32, kPickStride = kPickDims + 4;

template <bool VEC, bool RES>
__global__ void __launch_bounds__(32 * kPickWarps) ks_pick(const uint32_t* __restrict__ mask, int64_t N, int W,
                                                          const float* __restrict__ X, int D,
                                                          const float* __restrict__ W1,
                                                          const int32_t* __restrict__ c1, int c1_stride,
                                                          const float* __restrict__ words,
                                                          int32_t* __restrict__ out, int out_stride) {
    // staged rows: the vectors, the words and, for residues, the first words
    __shared__ __align__(16) float stage[kPickWarps][RES ? 3 : 2][32 * kPickStride];
    __shared__ uint16_t pairs[kPickWarps][kPickPairs];
    __shared__ unsigned long long best[kPickWarps][32];
    __shared__ int32_t code[kPickWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r0 = ((int64_t)blockIdx.x * kPickWarps + w) * 32, row = r0 + lane;
    if (r0 >= N) return;
    uint32_t m[8];
    int cnt = 0, first = 0;
#pragma unroll
    for (int q = 7; q >= 0; --q) {
        m[q] = row < N && 32 * q < W ? mask[row * 8 + q] : 0;
        if (W < 32 * q + 32 && W > 32 * q) m[q] &= (1u << (W - 32 * q)) - 1u;
        cnt += __popc(m[q]);
        if (m[q]) first = 32 * q + __ffs(m[q]) - 1;
    }
    best[w][lane] = cnt > 1 ? kEmptyKey : (unsigned long long)first;
    if (RES) code[w][lane] = cnt > 1 ? c1[row * c1_stride] : 0;
    __syncwarp();
    int left = cnt > 1 ? cnt : 0;  // pairs still to list
    int q = 0;
    while (__any_sync(0xffffffffu, left > 0)) {
        const int take = min(left, kPickPairs / 32);
        int at = take;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        const int total = __shfl_sync(0xffffffffu, at, 31);
        at -= take;
        for (int t = 0; t < take; ++t) {
            uint32_t cur = 0;
            while (q < 8) {  // the next word of this row's mask
#pragma unroll
                for (int z = 0; z < 8; ++z) cur = z == q ? m[z] : cur;
                if (cur) break;
                ++q;
            }
            const int j = __ffs(cur) - 1;
#pragma unroll
            for (int z = 0; z < 8; ++z)
                if (z == q) m[z] &= m[z] - 1;
            pairs[w][at + t] = (uint16_t)((lane << 8) | (32 * q + j));
        }
        left -= take;
        __syncwarp();
        for (int e = 0; e < total; e += 32) {
            const int np = min(32, total - e);  // pairs of this turn, one per lane
            const uint16_t* list = pairs[w] + e;
            float acc = 0.f;
            for (int d0 = 0; d0 < D; d0 += kPickDims) {
                const int dl = min(kPickDims, D - d0);
                // P pieces per row: a warp's lanes take 32 / P rows side by side
                constexpr int P = VEC ? kPickDims / 4 : 32, S = VEC ? 4 : 1;
                const int c = lane % P * S;
                for (int p = lane / P; p < np; p += 32 / P) {
                    if (c >= dl) continue;
                    const int r = list[p] >> 8;
                    const float* src[3] = {X + (r0 + r) * D, words + (int64_t)(list[p] & 255) * D,
                                           RES ? W1 + (int64_t)code[w][r] * D : nullptr};
#pragma unroll
                    for (int u = 0; u < (RES ? 3 : 2); ++u) {
                        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage[w][u] + p * kPickStride + c);
                        if (VEC)
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src[u] + d0 + c)
                                         : "memory");
                        else
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src[u] + d0 + c)
                                         : "memory");
                    }
                }
                asm volatile("cp.async.wait_all;\n" ::: "memory");
                __syncwarp();
                if (lane < np) {  // the canonical chain: dims ascending
                    const float* x = stage[w][0] + lane * kPickStride;
                    const float* y = stage[w][1] + lane * kPickStride;
                    const float* z = stage[w][RES ? 2 : 0] + lane * kPickStride;
                    auto add = [&](float a, float b, float v) {
                        const float t = __fsub_rn(RES ? __fsub_rn(a, v) : a, b);
                        acc = __fmaf_rn(t, t, acc);
                    };
                    if (VEC) {
#pragma unroll 4
                        for (int d = 0; d < dl; d += 4) {
                            const float4 a = *reinterpret_cast<const float4*>(x + d);
                            const float4 b = *reinterpret_cast<const float4*>(y + d);
                            const float4 v = RES ? *reinterpret_cast<const float4*>(z + d) : a;
                            add(a.x, b.x, v.x);
                            add(a.y, b.y, v.y);
                            add(a.z, b.z, v.z);
                            add(a.w, b.w, v.w);
                        }
                    } else {
                        for (int d = 0; d < dl; ++d) add(x[d], y[d], z[d]);
                    }
                }
                __syncwarp();  // the next stage overwrites
            }
            if (lane < np)
                atomicMin(&best[w][list[lane] >> 8], (unsigned long long)make_key(acc, (uint32_t)(list[lane] & 255)));
        }
        __syncwarp();
    }
    if (row < N) out[row * out_stride] = (int32_t)key_id(best[w][lane]);
}

// ---------------------------------------------------------------- thresholds and re-rank
constexpr int kRrThreads = 256;

// The value of rank `rank` (from 0) among u[0 .. c), by 8-bit digits from the
// top.  Called by the whole CTA; u is read only; synchronised on return.
__device__ uint32_t block_select32(const uint32_t* u, int c, int rank, int* hist, int* sh) {
    uint32_t prefix = 0;
    for (int sft = 24; sft >= 0; sft -= 8) {
        hist[threadIdx.x] = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < c; e += kRrThreads)
            if (sft == 24 || (u[e] >> (sft + 8)) == (prefix >> (sft + 8))) atomicAdd(hist + ((u[e] >> sft) & 255), 1);
        __syncthreads();
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = hist[threadIdx.x];
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh[w] = x;
        __syncthreads();
        int before = x - v;
        for (int q = 0; q < w; ++q) before += sh[q];
        if (before <= rank && rank < before + v) {
            sh[8] = (int)threadIdx.x;
            sh[9] = before;
        }
        __syncthreads();
        prefix |= (uint32_t)sh[8] << sft;
        rank -= sh[9];
        __syncthreads();
    }
    return prefix;
}

// One CTA per row: the row's candidates (dump: every column of the last
// product; else its collected list) give tau, an upper bound of its k-th least
// canonical distance.  FINAL = false: stores a_i and R_i of tau for the next,
// denser set of columns.  FINAL = true: the candidates that tau cannot exclude
// get their canonical distance and the k least (distance, id) are written.  A
// row whose list overflowed, or that the bound cannot serve, is listed for the
// FP32 kernel (fb_list, fb_count) and takes no further part.
template <bool FINAL>
__global__ void __launch_bounds__(kRrThreads) k7_rank(ScreenArgs P, bool dump, int k, float* __restrict__ rowA,
                                                     float* __restrict__ rowR, int* __restrict__ fb_flag,
                                                     int32_t* __restrict__ fb_list, int* __restrict__ fb_count,
                                                     uint64_t* __restrict__ out) {
    extern __shared__ uint64_t rk_smem[];
    __shared__ int hist[256], sh[10], ns_sh;
    if (*P.status & kStatusStop) return;
    const int64_t r = blockIdx.x;
    if (fb_flag[r]) return;  // listed already (its R_i excludes every column)
    uint32_t* u = reinterpret_cast<uint32_t*>(rk_smem);
    const int f = *P.flag_r;
    const bool exact = sc_exact(f);
    const float c2 = exact ? 0.f : P.cD2, gamma = exact ? 0.f : P.gamma;
    const int64_t own = P.rid ? (int64_t)P.rid[r] : P.rid0 + r;
    const int found = dump ? (int)P.ncols : P.cnt[r];
    const int c = min(found, P.cap);
    const float ni = P.rnrm[r], ei = exact ? 0.f : P.rerr[r];
    const float* cg = P.cg + r * P.cap;
    const int32_t* cid = P.cid + r * P.cap;
    const uint32_t kNone = 0xFFFFFFFFu;
    for (int e = threadIdx.x; e < c; e += kRrThreads) {
        const int64_t id = dump ? (int64_t)e * P.cstride : cid[e];
        uint32_t v = kNone;
        if (id != own) {
            const float ub = screen_ub(ni, P.cnrm[id], cg[e], ei, exact ? 0.f : P.cerr[id], c2, gamma);
            if (ub < __int_as_float(0x7f800000)) v = ord32(ub);
        }
        u[e] = v;
    }
    __syncthreads();
    const uint32_t sel = c >= k ? block_select32(u, c, k - 1, hist, sh) : kNone;
    if ((f & 8) || found > P.cap || sel == kNone) {
        if (threadIdx.x == 0) {
            fb_flag[r] = 1;
            fb_list[atomicAdd(fb_count, 1)] = (int32_t)r;
            atomicAdd(P.status + 1, 1);  // over all batches (statistics)
            rowA[r] = 0.f;
            rowR[r] = __int_as_float(0xff800000);
        }
        return;
    }
    float a, R;
    screen_row(unord32(sel), ni, ei, c2, gamma, exact, a, R);
    if (!FINAL) {
        if (threadIdx.x == 0) {
            rowA[r] = a;
            rowR[r] = R;
        }
        return;
    }
    uint64_t* keys = rk_smem;                                        // [cap] over u
    int32_t* sid = reinterpret_cast<int32_t*>(rk_smem + P.cap);      // [cap]
    float* q = reinterpret_cast<float*>(sid + P.cap);                // [D rounded up to 4]
    if (threadIdx.x == 0) ns_sh = 0;
    for (int d = threadIdx.x; d < P.D; d += kRrThreads) q[d] = P.X[own * P.D + d];
    __syncthreads();
    for (int e = threadIdx.x; e < c; e += kRrThreads) {
        const int64_t id = dump ? (int64_t)e * P.cstride : cid[e];
        const float nj = P.cnrm[id], ej = exact ? 0.f : P.cerr[id];
        const float cj = exact ? nj : __fsub_rd(__fmul_rd(nj, 1.f - c2), __fmul_ru(ej, ej));
        if (id != own && __fmaf_rn(-2.f * a, ej, __fmaf_rn(-2.f, cg[e], cj)) <= R) sid[atomicAdd(&ns_sh, 1)] = (int32_t)id;
    }
    __syncthreads();
    const int ns = ns_sh;
    int Pk = 2;
    while (Pk < ns) Pk <<= 1;
    for (int e = threadIdx.x; e < Pk; e += kRrThreads)
        keys[e] = e < ns ? make_key(point_dist(P.X + (int64_t)sid[e] * P.D, q, P.D, P.vec), (uint32_t)sid[e])
                         : kEmptyKey;
    __syncthreads();
    for (int kk = 2; kk <= Pk; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < Pk; i += kRrThreads) {
                const int l = i ^ j;
                if (l > i) {
                    const uint64_t x = keys[i], y = keys[l];
                    if ((x > y) == ((i & kk) == 0)) {
                        keys[i] = y;
                        keys[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    for (int e = threadIdx.x; e < k; e += kRrThreads) out[r * k + e] = e < Pk ? keys[e] : kEmptyKey;
}

// ---------------------------------------------------------------- host
// 2 cD + 2^-19 for the BF16 copy.
float screen_c(int D) { return 2.f * lp_cert_coeff(D, 1) + 1.9073486328125e-6f; }

void launch_screen_copy(const float* X, int64_t N, int D, const float* W1, const int32_t* c1, int c1_stride,
                        uint16_t* Xq, float* nrm, float* err, int* flags, int* status, cudaStream_t s) {
    const int Dp = lp_dim(D);
    LaunchScope ls("ks_copy", s, (double)N * (D * 4.0 + Dp * 2.0 + 8.0), 0);
    const unsigned grid = (unsigned)((N + 31) / 32);
    if (D % 4 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(W1)) & 15) == 0)
        ks_copy<true><<<grid, 256, 0, s>>>(X, N, D, Dp, W1, c1, c1_stride, Xq, nrm, err, flags, status);
    else
        ks_copy<false><<<grid, 256, 0, s>>>(X, N, D, Dp, W1, c1, c1_stride, Xq, nrm, err, flags, status);
}

bool screen_map(CUtensorMap* m, const uint16_t* p, int64_t rows, int Dp, int64_t stride, int box_rows) {
    const cuuint64_t gdim[2] = {(cuuint64_t)Dp, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)Dp * 2 * (cuuint64_t)stride};
    const cuuint32_t box[2] = {(cuuint32_t)kScK, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    return tensor_map_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p, gdim, gstride, box, estride);
}

template <int MODE>
bool launch_screen(const uint16_t* A, const uint16_t* B, int Dp, ScreenArgs& P, const char* name, cudaStream_t s) {
    CUtensorMap ta, tb;
    if (!screen_map(&ta, A, P.nrows, Dp, 1, kScM) || !screen_map(&tb, B, P.ncols, Dp, P.cstride, kScN)) return false;
    P.nk = Dp / kScK;
    P.nrt = (int)((P.nrows + kScM - 1) / kScM);
    P.nct = (int)((P.ncols + kScN - 1) / kScN);
    // one unit per CTA, or, with many tiles, about four, so that the last wave
    // is short
    const bool many = (int64_t)P.nrt * P.nct >= 64 * kScGrid;
    P.nstripe = std::max(1, std::min(P.nct, many ? (4 * kScGrid + P.nrt - 1) / P.nrt : kScGrid / P.nrt));
    const size_t smem = screen_smem(P.nk, MODE).total + 1024;
    const int64_t units = (int64_t)P.nrt * P.nstripe;
    LaunchScope ls(name, s, (double)(P.nrows + P.ncols) * (Dp * 2.0 + 8.0), (double)P.nrows * P.ncols * 2.0 * Dp);
    allow_smem(ks_screen<MODE>);
    ks_screen<MODE><<<(int)std::min<int64_t>(units, kScGrid), kScThreads, smem, s>>>(ta, tb, P);
    return true;
}

}  // namespace

// ---------------------------------------------------------------- nearest words
// The FP32 kernel takes about 0.19 us a dim, tile of 128 words and wave of 9,728
// vectors, the screen 25 us of short launches, plus rows of at least 64 dims to
// copy and read.  Index of 10,000 vectors, two assignments, FP32 against the
// screen (us): 64 words 16 dims 161 and 203, 64 dims 189 and 207, 128 dims 218 and
// 225, 300 dims 324 and 302; 256 words 64 dims 231 and 213; 100,000 vectors, 16
// dims: 64 words 222 and 248, 256 words 277 and 264.  With hardly more vectors than
// words the vectors are the words, and most distances of the residues are ties
// (300 x 300, 256 words: 418 and 1,800).
bool assign_screened(int64_t N, int D, int W) {
    const double tiles = (W + 127) / 128, waves = std::max(1.0, (double)N / 9728.0);
    return N >= 4 * (int64_t)W && D * tiles * waves >= 140.0 * std::max(1.0, 32.0 / D);
}

void launch_screen_copy(const float* X, int64_t N, int D, const float* W1, const int32_t* c1, int c1_stride,
                        const AssignWork& w, int* status, cudaStream_t s) {
    cudaMemsetAsync(w.flags, 0, sizeof(int), s);
    launch_screen_copy(X, N, D, W1, c1, c1_stride, w.Xq, w.nrm, w.err, w.flags, status, s);
}

bool launch_assign_screened(const float* X, int64_t N, int D, const float* W1, const int32_t* c1, int c1_stride,
                            const float* words, int W, const AssignWork& w, int32_t* out, int out_stride, int* status,
                            cudaStream_t s) {
    const int Dp = lp_dim(D);
    cudaMemsetAsync(w.flags + 1, 0, sizeof(int), s);
    launch_screen_copy(words, W, D, nullptr, nullptr, 0, w.Wq, w.wnrm, w.werr, w.flags + 1, nullptr, s);
    ScreenArgs P{};
    P.nrows = N;
    P.ncols = W;
    P.rnrm = w.nrm;
    P.rerr = w.err;
    P.cnrm = w.wnrm;
    P.cerr = w.werr;
    P.cstride = 1;
    P.cD2 = screen_c(D);
    P.gamma = (float)(D + 8) * 1.1920928955078125e-7f;
    P.flag_r = w.flags;
    P.flag_c = w.flags + 1;
    P.status = status;
    P.mask = w.mask;
    if (!launch_screen<kScArgmin>(w.Xq, w.Wq, Dp, P, W1 ? "ks_assign_res" : "ks_assign", s)) return false;
    const bool vec = D % 4 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(words) |
                                     reinterpret_cast<uintptr_t>(W1)) & 15) == 0;
    LaunchScope ls("ks_pick", s, (double)N * 36.0, 0);
    const auto pick = W1 ? (vec ? ks_pick<true, true> : ks_pick<false, true>)
                         : (vec ? ks_pick<true, false> : ks_pick<false, false>);
    constexpr int kRows = 32 * kPickWarps;
    pick<<<(unsigned)((N + kRows - 1) / kRows), kRows, 0, s>>>(w.mask, N, W, X, D, W1, c1, c1_stride, words, out,
                                                              out_stride);
    return true;
}

// ---------------------------------------------------------------- exact lists
// The FP32 kernel spends two instructions per pair and dim and a long chain
// per CTA, the screen one tensor-core product and about twelve short launches.
// Measured (GB300): n = 500, D = 128, 15 rows 195 us against 95; n = 20,000,
// D = 64, 7 rows 456 against 143; n = 1 M, D = 128, 1 row 5.7 ms against
// 0.55, 2,000 rows 189 ms against 1.33 (0.94 of it the products).  Below one
// column tile there is nothing to screen; a few rows of few values take the
// FP32 kernel less time than the launches (1 row of 256 x 32 93 us against 101,
// of 300 x 2 85 against 104; 256 rows of 256 x 32 124 against 109).
bool exact_screened(int64_t n, int D, int64_t s_rows) { return n >= kScN && (s_rows > 4 || n * D > 8192); }

int64_t exact_batch(int64_t s_rows) { return std::min<int64_t>(s_rows, 8192); }

bool launch_exact_screened(const float* X, int64_t n, int D, int k, const int32_t* sample, int64_t s_rows,
                           const ScreenWork& w, uint64_t* out, int* status, cudaStream_t s) {
    const int Dp = lp_dim(D);
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    cudaMemsetAsync(w.flags, 0, 2 * sizeof(int), s);
    launch_screen_copy(X, n, D, nullptr, nullptr, 0, w.Xq, w.nrm, w.err, w.flags, status, s);
    // column sets: every st0-th row (at most kScreenCap of them, all kept),
    // then 4 times as many each time, up to every row.  A set's k-th least
    // upper bound bounds the row's k-th distance, so about 4 k columns of the
    // next one stay below it.
    constexpr int64_t kGrow = 4;
    int64_t st0 = 1;
    while ((n + st0 - 1) / st0 > kScreenCap) st0 *= kGrow;
    const int64_t batch = exact_batch(s_rows);
    const int nsplit = exact_splits(n, batch);
    const size_t rank_smem = (size_t)kScreenCap * 12 + ((size_t)D + 3) / 4 * 16;
    allow_smem(k7_rank<true>);
    for (int64_t q0 = 0; q0 < s_rows; q0 += batch) {
        const int64_t rows = std::min(batch, s_rows - q0);
        ScreenArgs P{};
        const uint16_t* A;
        if (sample) {
            LaunchScope ls("ks_gather", s, (double)rows * (Dp * 4.0 + 16.0), 0);
            const int64_t pieces = rows * (Dp / 8);
            ks_gather<<<(unsigned)std::min<int64_t>((pieces + 255) / 256, kScGrid * 16), 256, 0, s>>>(
                reinterpret_cast<const uint4*>(w.Xq), w.nrm, w.err, rows, Dp / 8, sample + q0,
                reinterpret_cast<uint4*>(w.Qq), w.qn, w.qe, status);
            A = w.Qq;
            P.rnrm = w.qn;
            P.rerr = w.qe;
            P.rid = sample + q0;
        } else {
            A = w.Xq + q0 * Dp;
            P.rnrm = w.nrm + q0;
            P.rerr = w.err + q0;
            P.rid0 = q0;
        }
        P.nrows = rows;
        P.cnrm = w.nrm;
        P.cerr = w.err;
        P.cD2 = screen_c(D);
        P.gamma = (float)(D + 8) * 1.1920928955078125e-7f;
        P.flag_r = P.flag_c = w.flags;
        P.status = status;
        P.cap = kScreenCap;
        P.cg = w.cg;
        P.cid = w.cid;
        P.cnt = w.cnt;
        P.rowA = w.rowA;
        P.rowR = w.rowR;
        P.X = X;
        P.D = D;
        P.vec = vec;
        cudaMemsetAsync(w.fb_flag, 0, sizeof(int32_t) * rows, s);
        cudaMemsetAsync(w.flags + 1, 0, sizeof(int), s);
        for (int64_t st = st0;; st /= kGrow) {
            P.cstride = st;
            P.ncols = (n + st - 1) / st;
            const bool dump = st == st0, last = st == 1;
            if (dump) {
                if (!launch_screen<kScDump>(A, w.Xq, Dp, P, "ks_screen", s)) return false;
            } else {
                cudaMemsetAsync(w.cnt, 0, sizeof(int32_t) * rows, s);
                if (!launch_screen<kScCollect>(A, w.Xq, Dp, P, "ks_screen", s)) return false;
            }
            LaunchScope ls("k7_rank", s, 0, 0);
            if (last) {
                k7_rank<true><<<(unsigned)rows, kRrThreads, rank_smem, s>>>(P, dump, k, w.rowA, w.rowR, w.fb_flag,
                                                                            w.fb_list, w.flags + 1, out + q0 * k);
                break;
            }
            k7_rank<false><<<(unsigned)rows, kRrThreads, kScreenCap * 4, s>>>(P, dump, k, w.rowA, w.rowR, w.fb_flag,
                                                                              w.fb_list, w.flags + 1, nullptr);
        }
        launch_exact(X, n, D, k, sample ? sample + q0 : nullptr, q0, rows, w.fb_list, w.flags + 1, nsplit, w.part,
                     out + q0 * k, status, s);
    }
    return true;
}

}  // namespace knng
