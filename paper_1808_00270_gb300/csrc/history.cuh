// history.cuh -- kernels of the history convolution shared by k_history.cu
// (whole sums, batches) and k_history_blk.cu (sums resumed from the parts of a
// block of steps).
#pragma once

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include <cuda_bf16.h>

#include "launch.h"

namespace gld {

// The step is number t of its block (len steps; t < 0: no parts).
struct BlockPos {
    const float* part;
    int t, len;
};

// A launch decision, cached per (device, columns, slots) for each
// instantiation: the occupancy queries cost far more host time than a launch.
struct Shape {
    int kind;  // 0: one column per thread, 1: general kernel
    int block, G;
    unsigned grid;
};

namespace {

constexpr int kThreads = 256;     // largest block; the launch picks 64 .. 256
constexpr int kUnroll = 8;         // loads issued together per thread

template <bool KAHAN>
__device__ __forceinline__ void acc1(float& s, float& comp, float c, float v)
{
    if (KAHAN) {
        const float y = fmaf(c, v, -comp);
        const float t = s + y;
        comp = (t - s) - y;
        s = t;
    } else {
        s = fmaf(c, v, s);
    }
}

template <int NACC>
__device__ __forceinline__ void stage_coefs(float* cs, const float* __restrict__ coef, int M, int H,
                                            long long n, int from = 0)
{
    int r0 = (int)((n - 1) % H);  // slot s holds m = ((n - 1 - s) mod H) + 1
    if (r0 < 0) r0 += H;
    for (int s = from + threadIdx.x; s < H; s += blockDim.x) {
        const int r = r0 - s;
        const int m = (r < 0 ? r + H : r) + 1;
#pragma unroll
        for (int a = 0; a < NACC; ++a) cs[s * NACC + a] = __ldg(coef + a * M + m);
    }
    __syncthreads();
}

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Blocks of steps.  Within a block of `len` steps that starts at step n0 only
// the slots h0 .. h0 + len - 1 (mod H), h0 = n0 mod H, are rewritten.  A
// column's sum runs over a range [lo, hi) of slots in a fixed order, so the
// terms before the range's first such slot are the same chain of FMAs for
// every step that the full sum would start with: conv_pre forms them for all
// steps of the block in one pass over those rows, and each step resumes its
// chain there -- the same bits as the full sum.
__device__ __forceinline__ int first_rewritten(int lo, int hi, int h0, int len, int H)
{
    const int over = h0 + len - H;              // slots [0, over) are rewritten too
    if (lo < over || (lo >= h0 && lo < h0 + len)) return lo;
    return h0 >= lo && h0 < hi ? h0 : hi;
}

// Row of the parts [G][len][nacc][planes][3 n_pad] (planes: 2 with compensation).
__device__ __forceinline__ size_t part_row(int g, int t, int a, int plane, int len, int nacc, int planes)
{
    return (((size_t)g * len + t) * nacc + a) * planes + plane;
}

__device__ __forceinline__ int step_slot(long long n, int H)
{
    const long long r = n % H;
    return (int)(r < 0 ? r + H : r);
}

template <bool BF16>
struct Col {
    using V = typename std::conditional<BF16, uint4, float4>::type;
    static constexpr int W = BF16 ? 8 : 4;  // values per 16-byte column
};

template <bool BF16>
__device__ __forceinline__ void unpack(const typename Col<BF16>::V v, float (&x)[Col<BF16>::W])
{
    if constexpr (BF16) {
        x[0] = bf_lo(v.x); x[1] = bf_hi(v.x); x[2] = bf_lo(v.y); x[3] = bf_hi(v.y);
        x[4] = bf_lo(v.z); x[5] = bf_hi(v.z); x[6] = bf_lo(v.w); x[7] = bf_hi(v.w);
    } else {
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    }
}

// Sums (and compensations) of a column as the block's parts hold them.
template <int NACC, bool KAHAN, int VW>
__device__ __forceinline__ void load_part(const BlockPos& bp, int g, long long cols, long long q, float (&acc)[NACC][VW],
                                          float (&cmp)[KAHAN ? NACC : 1][VW])
{
    constexpr int PL = KAHAN ? 2 : 1;
    const long long cols4 = cols * (VW / 4);
    const float4* b = (const float4*)bp.part + part_row(g, bp.t, 0, 0, bp.len, NACC, PL) * cols4 + q * (VW / 4);
#pragma unroll
    for (int a = 0; a < NACC; ++a)
#pragma unroll
        for (int h = 0; h < VW / 4; ++h) {
            const float4 f = __ldcs(b + (a * PL) * cols4 + h);
            acc[a][4 * h] = f.x; acc[a][4 * h + 1] = f.y; acc[a][4 * h + 2] = f.z; acc[a][4 * h + 3] = f.w;
            if constexpr (KAHAN) {
                const float4 k = __ldcs(b + (a * PL + 1) * cols4 + h);
                cmp[a][4 * h] = k.x; cmp[a][4 * h + 1] = k.y; cmp[a][4 * h + 2] = k.z; cmp[a][4 * h + 3] = k.w;
            }
        }
}

// One 16-byte column per thread over all slots, one wave (the common case;
// the lean form keeps the register count at 44 for two FP32 accumulators).
// Two FP32 accumulators fit in 40 registers: 6 CTAs of 256 threads per SM,
// enough for one wave of the 262144-particle suspension (768 CTAs).
// PART: the chain is resumed from the block's parts.
template <int NACC, bool KAHAN, bool BF16, bool PART>
__global__ void __launch_bounds__(kThreads, (NACC * Col<BF16>::W * (KAHAN ? 2 : 1) <= 8) ? 6 : 1)
    hist_conv_col(const typename Col<BF16>::V* __restrict__ ring, long long cols, int H,
                  const float* __restrict__ coef, int M, const long long* __restrict__ nstep, long long step,
                  float* __restrict__ out, const BlockPos bp)
{
    using V = typename Col<BF16>::V;
    constexpr int VW = Col<BF16>::W;
    extern __shared__ float cs[];
    const long long n = nstep ? *nstep : step;
    const int s_first = PART ? first_rewritten(0, H, step_slot(n - bp.t, H), bp.len, H) : 0;
    stage_coefs<NACC>(cs, coef, M, H, n, s_first);
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= cols) return;
    float acc[NACC][VW];
    float cmp[KAHAN ? NACC : 1][VW];
#pragma unroll
    for (int a = 0; a < NACC; ++a)
#pragma unroll
        for (int e = 0; e < VW; ++e) acc[a][e] = 0.f;
#pragma unroll
    for (int a = 0; a < (KAHAN ? NACC : 1); ++a)
#pragma unroll
        for (int e = 0; e < VW; ++e) cmp[a][e] = 0.f;
    const V* p = ring + q;
    if (PART && s_first > 0) load_part<NACC, KAHAN, VW>(bp, 0, cols, q, acc, cmp);
    int s = s_first;
    for (; s + kUnroll <= H; s += kUnroll) {
        V v[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) v[u] = __ldcs(p + (long long)(s + u) * cols);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            float x[VW];
            unpack<BF16>(v[u], x);
#pragma unroll
            for (int a = 0; a < NACC; ++a) {
                const float cf = cs[(s + u) * NACC + a];
#pragma unroll
                for (int e = 0; e < VW; ++e) acc1<KAHAN>(acc[a][e], cmp[KAHAN ? a : 0][e], cf, x[e]);
            }
        }
    }
    for (; s < H; ++s) {
        float x[VW];
        unpack<BF16>(__ldcs(p + (long long)s * cols), x);
#pragma unroll
        for (int a = 0; a < NACC; ++a) {
            const float cf = cs[s * NACC + a];
#pragma unroll
            for (int e = 0; e < VW; ++e) acc1<KAHAN>(acc[a][e], cmp[KAHAN ? a : 0][e], cf, x[e]);
        }
    }
    float4* o = (float4*)out;
    const long long cols4 = cols * (VW / 4);
#pragma unroll
    for (int a = 0; a < NACC; ++a)
#pragma unroll
        for (int h = 0; h < VW / 4; ++h) {
            float r[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) r[e] = KAHAN ? acc[a][4 * h + e] - cmp[KAHAN ? a : 0][4 * h + e] : acc[a][4 * h + e];
            o[a * cols4 + q * (VW / 4) + h] = make_float4(r[0], r[1], r[2], r[3]);
        }
}

// One 16-byte column (4 FP32 or 8 BF16 values) per thread and slot group.
// The G threads of a column split its slots into G contiguous ranges and are
// combined in shared memory in a fixed order.  Loads run as a rolling
// pipeline: a register is refilled with the slot kUnroll ahead as soon as it
// is consumed, so kUnroll loads per thread stay in flight.
template <int NACC, bool KAHAN, bool BF16>
__global__ void __launch_bounds__(kThreads)
    hist_conv(const typename Col<BF16>::V* __restrict__ ring, long long cols, int H, const float* __restrict__ coef,
              int M, const long long* __restrict__ nstep, long long step, float* __restrict__ out, int G)
{
    using V = typename Col<BF16>::V;
    constexpr int VW = Col<BF16>::W;
    extern __shared__ float cs[];
    __shared__ float4 red[kThreads * (BF16 ? 2 : 1)];
    const long long n = nstep ? *nstep : step;
    stage_coefs<NACC>(cs, coef, M, H, n);
    const int per = blockDim.x / G;  // columns per block
    const int g = threadIdx.x / per, c = threadIdx.x - g * per;
    const int s_lo = (int)((long long)g * H / G), s_hi = (int)((long long)(g + 1) * H / G);
    for (long long qb = (long long)blockIdx.x * per; qb < cols; qb += (long long)gridDim.x * per) {
        const long long q = qb + c;
        float acc[NACC][VW];
        float cmp[KAHAN ? NACC : 1][VW];
#pragma unroll
        for (int a = 0; a < NACC; ++a)
#pragma unroll
            for (int e = 0; e < VW; ++e) acc[a][e] = 0.f;
#pragma unroll
        for (int a = 0; a < (KAHAN ? NACC : 1); ++a)
#pragma unroll
            for (int e = 0; e < VW; ++e) cmp[a][e] = 0.f;
        if (q < cols) {
            const V* p = ring + q;
            int s = s_lo;
            for (; s + kUnroll <= s_hi; s += kUnroll) {
                V v[kUnroll];
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) v[u] = __ldcs(p + (long long)(s + u) * cols);
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    float x[VW];
                    unpack<BF16>(v[u], x);
#pragma unroll
                    for (int a = 0; a < NACC; ++a) {
                        const float cf = cs[(s + u) * NACC + a];
#pragma unroll
                        for (int e = 0; e < VW; ++e) acc1<KAHAN>(acc[a][e], cmp[KAHAN ? a : 0][e], cf, x[e]);
                    }
                }
            }
            for (; s < s_hi; ++s) {
                float x[VW];
                unpack<BF16>(__ldcs(p + (long long)s * cols), x);
#pragma unroll
                for (int a = 0; a < NACC; ++a) {
                    const float cf = cs[s * NACC + a];
#pragma unroll
                    for (int e = 0; e < VW; ++e) acc1<KAHAN>(acc[a][e], cmp[KAHAN ? a : 0][e], cf, x[e]);
                }
            }
            if constexpr (KAHAN) {
#pragma unroll
                for (int a = 0; a < NACC; ++a)
#pragma unroll
                    for (int e = 0; e < VW; ++e) acc[a][e] -= cmp[a][e];  // compensated value
            }
        }
        float4* o = (float4*)out;
        const long long cols4 = cols * (VW / 4);  // float4 per accumulator row
        if (G == 1) {
            if (q < cols)
#pragma unroll
                for (int a = 0; a < NACC; ++a)
#pragma unroll
                    for (int h = 0; h < VW / 4; ++h)
                        o[a * cols4 + q * (VW / 4) + h] =
                            make_float4(acc[a][4 * h], acc[a][4 * h + 1], acc[a][4 * h + 2], acc[a][4 * h + 3]);
        } else {
            // fixed-order combine of the G slot ranges, one accumulator at a time
#pragma unroll
            for (int a = 0; a < NACC; ++a) {
#pragma unroll
                for (int h = 0; h < VW / 4; ++h)
                    red[threadIdx.x * (VW / 4) + h] =
                        make_float4(acc[a][4 * h], acc[a][4 * h + 1], acc[a][4 * h + 2], acc[a][4 * h + 3]);
                __syncthreads();
                if (g == 0 && q < cols) {
#pragma unroll
                    for (int h = 0; h < VW / 4; ++h) {
                        float4 t = red[c * (VW / 4) + h];
                        for (int gg = 1; gg < G; ++gg) {
                            const float4 y = red[(gg * per + c) * (VW / 4) + h];
                            t.x += y.x; t.y += y.y; t.z += y.z; t.w += y.w;
                        }
                        o[a * cols4 + q * (VW / 4) + h] = t;
                    }
                }
                __syncthreads();
            }
        }
    }
}

__host__ __device__ constexpr int pre_len(int kahan, int G) { return kahan || G > 1 ? 8 : 16; }

// Calls f(std::integral_constant<int, nacc>, bool_constant<kahan>) for 1 <= nacc <= kMaxAcc.
template <class F>
cudaError_t by_nacc(int nacc, bool kahan, F&& f)
{
#define GLD_NACC(N)                                                          \
    case N:                                                                  \
        return kahan ? f(std::integral_constant<int, N>{}, std::true_type{}) \
                     : f(std::integral_constant<int, N>{}, std::false_type{});
    switch (nacc) {
        GLD_NACC(1) GLD_NACC(2) GLD_NACC(3) GLD_NACC(4) GLD_NACC(5) GLD_NACC(6) GLD_NACC(7) GLD_NACC(8) GLD_NACC(9)
    default: return cudaErrorInvalidValue;
    }
#undef GLD_NACC
}

}  // namespace

// k_history_blk.cu: a step whose chains are resumed from the parts.
cudaError_t launch_hist_conv_part(const Shape& sh, int nacc, int kahan, const void* ring, int bf16, int n_pad, int M,
                                  const long long* nstep, long long step, const float* coef, float* out,
                                  const BlockPos& bp, cudaStream_t st);

}  // namespace gld
