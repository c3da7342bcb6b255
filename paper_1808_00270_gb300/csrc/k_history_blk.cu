// k_history_blk.cu -- the history convolution over blocks of steps: the parts of
// a block (conv_pre) and the steps that resume their sums from them.
//
// A step of the streaming convolution reads the whole ring (12 H bytes per
// particle).  Within a block of 8 or 16 steps only 8 or 16 slots are
// rewritten; the chain of FMAs over the slots before the first of them is the
// same for all steps, so it is formed once per block for all of its steps --
// bound by the FP32 pipes, 2 x 16 FMAs per value read -- and each step streams
// only the rest of the ring.  Sums keep their order, and with it every bit.
#include "history.cuh"

namespace gld {

namespace {

// ---- parts of a block of steps ----------------------------------------------
// Chains of the slots before each range's first rewritten one, for the LEN
// steps of the block that starts at step n0: one thread per two or four
// streams, NA accumulators and LEN outputs, so one load feeds 64 FMAs with two
// accumulators (bound by the FP32 pipes, not by HBM).
// Eight rows are in flight; the weights of 8 rows x LEN steps are LEN + 7
// values of one accumulator (row s + 1 has the weights of row s shifted by
// one), read from shared memory as broadcasts.
constexpr int kPreThreads = 128;

// VB bytes of a ring row (4, 8 or 16), streamed.  A group of rows is loaded
// before the first is used: the address of the group's weights is made to
// depend on the last load (`& none`, none = 0 at run time).  Left to itself the
// compiler interleaved loads and sums in about half of the instances (32 to 40
// registers where the loads in flight alone need 32) and lost most of the
// bandwidth (batch step: 139 us where the whole sum took 114 us).
template <int VB>
struct Row {
    uint32_t w[VB / 4];
};

template <int VB>
__device__ __forceinline__ Row<VB> load_row(const char* p)
{
    Row<VB> r;
    if constexpr (VB == 16)
        asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]) : "l"(p));
    else if constexpr (VB == 8)
        asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(r.w[0]), "=r"(r.w[1]) : "l"(p));
    else
        asm volatile("ld.global.cs.u32 %0, [%1];" : "=r"(r.w[0]) : "l"(p));
    return r;
}

template <int VB, bool BF16>
__device__ __forceinline__ void values(const Row<VB>& r, float (&x)[VB / (BF16 ? 2 : 4)])
{
#pragma unroll
    for (int k = 0; k < VB / 4; ++k) {
        if constexpr (BF16) {
            x[2 * k] = bf_lo(r.w[k]);
            x[2 * k + 1] = bf_hi(r.w[k]);
        } else {
            x[k] = __uint_as_float(r.w[k]);
        }
    }
}

// Streams per thread: 64 sums (and their compensations) in registers with two
// accumulators.
__host__ __device__ constexpr int pre_streams(int len, bool kahan) { return len == 8 && !kahan ? 4 : 2; }

template <int NA, int LEN, bool KAHAN, bool BF16>
__device__ __forceinline__ void pre_body(const void* __restrict__ ring, int n_pad, int H, int M,
                                         const float* __restrict__ coef, int nacc, long long n0, float* __restrict__ part,
                                         int a0, int g, int G, int blk)
{
    extern __shared__ float cs[];  // [NA][rows + LEN - 1]: weight of row s at step t: cs[last - s + t]
    constexpr int PL = KAHAN ? 2 : 1;
    const int lo = (int)((long long)g * H / G), hi = (int)((long long)(g + 1) * H / G);
    const int e = first_rewritten(lo, hi, step_slot(n0, H), LEN, H);
    const int rows = e - lo, nw = rows + LEN - 1;
    if (rows <= 0) return;  // uniform over the block
    const int m_last = step_slot(n0 - 1 - (e - 1), H) + 1;  // m of slot e - 1 at step n0
    for (int x = threadIdx.x; x < NA * nw; x += blockDim.x) {
        const int a = x / nw, m = m_last + x - a * nw;
        cs[x] = m <= H ? __ldg(coef + (size_t)(a0 + a) * M + m) : 0.f;
    }
    __syncthreads();
    constexpr int W = pre_streams(LEN, KAHAN), VB = W * (BF16 ? 2 : 4);
    const int C = 3 * n_pad / W, q = blk * kPreThreads + (int)threadIdx.x;
    if (q >= C) return;
    const size_t stride = (size_t)C * VB;
    const char* p = (const char*)ring + (size_t)lo * stride + (size_t)q * VB;
    const uint32_t none = (uint32_t)H >> 16;  // 0: H < 4096
    float acc[NA][LEN][W], cmp[KAHAN ? NA : 1][LEN][W];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int t = 0; t < LEN; ++t)
#pragma unroll
            for (int k = 0; k < W; ++k) {
                acc[a][t][k] = 0.f;
                if (KAHAN) cmp[KAHAN ? a : 0][t][k] = 0.f;
            }
    int s = lo;
    for (; s + 8 <= e; s += 8) {
        Row<VB> r[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            r[u] = load_row<VB>(p);
            p += stride;
        }
        float x[8][W];
#pragma unroll
        for (int u = 0; u < 8; ++u) values<VB, BF16>(r[u], x[u]);
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            float w[LEN + 7];
            const float* c = cs + a * nw + (e - 1 - s - 7) + (r[7].w[0] & none);
#pragma unroll
            for (int v = 0; v < LEN + 7; ++v) w[v] = c[v];
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int t = 0; t < LEN; ++t)
#pragma unroll
                    for (int k = 0; k < W; ++k)
                        acc1<KAHAN>(acc[a][t][k], cmp[KAHAN ? a : 0][t][k], w[7 - u + t], x[u][k]);
        }
    }
    for (; s < e; ++s) {
        float x[W];
        values<VB, BF16>(load_row<VB>(p), x);
        p += stride;
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int t = 0; t < LEN; ++t) {
                const float w = cs[a * nw + (e - 1 - s) + t];
#pragma unroll
                for (int k = 0; k < W; ++k) acc1<KAHAN>(acc[a][t][k], cmp[KAHAN ? a : 0][t][k], w, x[k]);
            }
    }
    using F = typename std::conditional<W == 4, float4, float2>::type;
    F* o = (F*)part + q;
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int t = 0; t < LEN; ++t) {
            auto pack = [](const float (&v)[W]) {
                if constexpr (W == 4) return make_float4(v[0], v[1], v[2], v[3]);
                else return make_float2(v[0], v[1]);
            };
            o[part_row(g, t, a0 + a, 0, LEN, nacc, PL) * C] = pack(acc[a][t]);
            if constexpr (KAHAN) o[part_row(g, t, a0 + a, 1, LEN, nacc, PL) * C] = pack(cmp[a][t]);
        }
}

template <int NA, int LEN, bool KAHAN, bool BF16>
__global__ void __launch_bounds__(kPreThreads)
    conv_pre(const void* __restrict__ ring, int n_pad, int H, int M, const float* __restrict__ coef, int nacc,
             const long long* __restrict__ nstep, float* __restrict__ part, int a0, int G)
{
    pre_body<NA, LEN, KAHAN, BF16>(ring, n_pad, H, M, coef, nacc, *nstep, part, a0 + NA * (int)blockIdx.z,
                                   (int)blockIdx.y, G, (int)blockIdx.x);
}

template <int NA, int LEN, bool KAHAN, bool BF16>
__global__ void __launch_bounds__(kPreThreads)
    b_conv_pre(const SysDesc* __restrict__ D, const Tile* __restrict__ tiles, int a0)
{
    const Tile t = tiles[blockIdx.x];
    const SysDesc& d = D[t.m];
    pre_body<NA, LEN, KAHAN, BF16>(d.B.ring, d.P.n_pad, d.P.H, d.P.m_max, d.coef, d.P.nacc, d.B.ctrl->step, d.B.part,
                                   a0 + NA * (int)blockIdx.z, 0, 1, t.b);
}

template <int NA, int LEN, bool KAHAN, bool BF16>
cudaError_t pre_launch(const void* ring, int n_pad, int M, const float* coef, int nacc, const long long* nstep,
                       float* part, int a0, int passes, int G, cudaStream_t st)
{
    const size_t smem = sizeof(float) * (size_t)NA * (M + LEN);
    auto k = conv_pre<NA, LEN, KAHAN, BF16>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    const int C = 3 * n_pad / pre_streams(LEN, KAHAN);
    const dim3 grid((unsigned)((C + kPreThreads - 1) / kPreThreads), (unsigned)G, (unsigned)passes);
    k<<<grid, kPreThreads, smem, st>>>(ring, n_pad, M - 1, M, coef, nacc, nstep, part, a0, G);
    return cudaGetLastError();
}

template <int NA, int LEN, bool KAHAN, bool BF16>
cudaError_t b_pre_launch(const BatchPlan& bp, int a0, int passes, cudaStream_t st)
{
    const size_t smem = sizeof(float) * (size_t)NA * (bp.max_H + 1 + LEN);
    auto k = b_conv_pre<NA, LEN, KAHAN, BF16>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    k<<<dim3((unsigned)bp.n_pre, 1u, (unsigned)passes), kPreThreads, smem, st>>>(bp.desc, bp.pre, a0);
    return cudaGetLastError();
}

// f(NA, LEN, KAHAN, BF16 as constants, first accumulator, passes): the
// accumulators in pairs, an odd last one alone.
template <class F>
cudaError_t by_pre(int nacc, int kahan, int bf16, int len, F&& f)
{
    auto na = [&](auto n, int a0, int passes) -> cudaError_t {
        if (passes == 0) return cudaSuccess;
        using I8 = std::integral_constant<int, 8>;
        using I16 = std::integral_constant<int, 16>;
        if (kahan) return bf16 ? f(n, I8{}, std::true_type{}, std::true_type{}, a0, passes)
                               : f(n, I8{}, std::true_type{}, std::false_type{}, a0, passes);
        if (len == 8) return bf16 ? f(n, I8{}, std::false_type{}, std::true_type{}, a0, passes)
                                  : f(n, I8{}, std::false_type{}, std::false_type{}, a0, passes);
        return bf16 ? f(n, I16{}, std::false_type{}, std::true_type{}, a0, passes)
                    : f(n, I16{}, std::false_type{}, std::false_type{}, a0, passes);
    };
    const cudaError_t e = na(std::integral_constant<int, 2>{}, 0, nacc / 2);
    return e != cudaSuccess ? e : na(std::integral_constant<int, 1>{}, nacc & ~1, nacc & 1);
}

// ---- a step resumed from the parts -------------------------------------------
// One thread per VB bytes of a row: the slots of a column are split into G
// ranges; a range without rewritten slots is complete in the parts, the one or
// two others go on from their first rewritten slot; the ranges are added in
// the order of the whole sum (((R_0 + R_1) + R_2) + R_3).  The whole sum's G
// threads per 16-byte column would leave all but the threads of those ranges
// idle; here a thread takes its bytes through all ranges, and VB is the
// largest of 16, 8 and 4 that still gives every SM 512 threads.
__host__ __device__ constexpr int tail_unroll(int vb) { return vb == 16 ? 8 : 16; }

template <int NACC, bool KAHAN, bool BF16, int VB>
__device__ __forceinline__ void tail_body(float* cs, const void* __restrict__ ring, int n_pad, int H, int M,
                                          const float* __restrict__ coef, long long n, const BlockPos& bp, int G,
                                          float* __restrict__ out, int q0, int qstride)
{
    constexpr int W = VB / (BF16 ? 2 : 4), PL = KAHAN ? 2 : 1, U = tail_unroll(VB);
    const int h0 = step_slot(n - bp.t, H);
    const int C = 3 * n_pad / W;
    auto lo_of = [&](int g) { return (int)((unsigned)(g * H) / (unsigned)G); };
    // first rewritten slot of a range (its end: none)
    auto first_of = [&](int lo, int hi) { return bp.t < 0 ? lo : first_rewritten(lo, hi, h0, bp.len, H); };
    int from = H;
    for (int g = G - 1; g >= 0; --g) {
        const int f = first_of(lo_of(g), lo_of(g + 1));
        if (f < lo_of(g + 1)) from = f;
    }
    stage_coefs<NACC>(cs, coef, M, H, n, from);
    const size_t stride = (size_t)C * VB, S = (size_t)C * W;
    const uint32_t none = (uint32_t)H >> 16;  // 0: H < 4096
    for (int q = q0 + (int)threadIdx.x; q < C; q += qstride) {
        float tot[NACC][W], cmp[KAHAN ? NACC : 1][W];
#pragma unroll 1
        for (int g = 0; g < G; ++g) {
            const int lo = lo_of(g), hi = lo_of(g + 1), first = first_of(lo, hi);
            float acc[NACC][W];
            if (first > lo) {
                const float* b = bp.part + part_row(g, bp.t, 0, 0, bp.len, NACC, PL) * S + (size_t)q * W;
#pragma unroll
                for (int a = 0; a < NACC; ++a)
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        acc[a][w] = __ldg(b + (size_t)(a * PL) * S + w);
                        if (KAHAN) cmp[KAHAN ? a : 0][w] = __ldg(b + (size_t)(a * PL + 1) * S + w);
                    }
            } else {
#pragma unroll
                for (int a = 0; a < NACC; ++a)
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        acc[a][w] = 0.f;
                        if (KAHAN) cmp[KAHAN ? a : 0][w] = 0.f;
                    }
            }
            auto term = [&](const float* c0, int u, const Row<VB>& r) {
                float x[W];
                values<VB, BF16>(r, x);
#pragma unroll
                for (int a = 0; a < NACC; ++a) {
                    const float c = c0[u * NACC + a];
#pragma unroll
                    for (int w = 0; w < W; ++w) acc1<KAHAN>(acc[a][w], cmp[KAHAN ? a : 0][w], c, x[w]);
                }
            };
            int s = first;
            const char* p = (const char*)ring + (size_t)s * stride + (size_t)q * VB;
            for (; s + U <= hi; s += U) {
                Row<VB> r[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    r[u] = load_row<VB>(p);
                    p += stride;
                }
                const float* c0 = cs + s * NACC + (r[U - 1].w[0] & none);
#pragma unroll
                for (int u = 0; u < U; ++u) term(c0, u, r[u]);
            }
            if (s < hi) {  // the last rows, in flight together too (past the end: the last row again, unused)
                Row<VB> r[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    r[u] = load_row<VB>(p);
                    if (s + u + 1 < hi) p += stride;
                }
                const float* c0 = cs + s * NACC + (r[U - 1].w[0] & none);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (s + u < hi) term(c0, u, r[u]);
            }
#pragma unroll
            for (int a = 0; a < NACC; ++a)
#pragma unroll
                for (int w = 0; w < W; ++w) tot[a][w] = g == 0 ? acc[a][w] : tot[a][w] + acc[a][w];
        }
#pragma unroll
        for (int a = 0; a < NACC; ++a)
#pragma unroll
            for (int w = 0; w < W; ++w)
                out[(size_t)a * S + (size_t)q * W + w] = KAHAN ? tot[a][w] - cmp[KAHAN ? a : 0][w] : tot[a][w];
    }
}

template <int NACC, bool KAHAN, bool BF16, int VB>
__global__ void __launch_bounds__(kThreads)
    conv_tail(const void* __restrict__ ring, int n_pad, int H, int M, const float* __restrict__ coef,
              const long long* __restrict__ nstep, long long step, const BlockPos bp, int G, float* __restrict__ out)
{
    extern __shared__ float cs[];
    tail_body<NACC, KAHAN, BF16, VB>(cs, ring, n_pad, H, M, coef, nstep ? *nstep : step, bp, G, out,
                                     (int)(blockIdx.x * blockDim.x), (int)(gridDim.x * blockDim.x));
}

// Batch convolution of step t of the block: tile (member, block of 16-byte
// columns).  A member without parts (P.cblk = 0) streams its whole ring.
template <int NACC, bool KAHAN, bool BF16>
__global__ void __launch_bounds__(kBatchConvCols)
    b_conv(const SysDesc* __restrict__ D, const Tile* __restrict__ tiles, int t_blk)
{
    extern __shared__ float cs[];
    const Tile t = tiles[blockIdx.x];
    const SysDesc& d = D[t.m];
    const BlockPos bp{d.B.part, d.P.cblk ? t_blk : -1, pre_len(KAHAN, 1)};
    tail_body<NACC, KAHAN, BF16, 16>(cs, d.B.ring, d.P.n_pad, d.P.H, d.P.m_max, d.coef, d.B.ctrl->step, bp, 1, d.B.conv,
                                     t.b * (int)blockDim.x, t.nb * (int)blockDim.x);
}

template <int NACC, bool KAHAN>
cudaError_t launch_b_conv_t(const BatchPlan& bp, int t, cudaStream_t st)
{
    const size_t smem = sizeof(float) * (size_t)bp.max_H * NACC;
    auto k = bp.bf16 ? b_conv<NACC, KAHAN, true> : b_conv<NACC, KAHAN, false>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    k<<<bp.n_conv, bp.conv_block, smem, st>>>(bp.desc, bp.conv, t);
    return cudaGetLastError();
}

template <int NACC, bool KAHAN, bool BF16>
cudaError_t part_launch(const Shape& sh, const void* ring, int n_pad, int M, const long long* nstep, long long step,
                        const float* coef, float* out, const BlockPos& bp, cudaStream_t st)
{
    const int H = M - 1;
    const size_t smem = sizeof(float) * (size_t)H * NACC;
    const long long bytes = 3LL * n_pad * (BF16 ? 2 : 4);
    // One range, one wave of 16-byte columns.  Compensated sums have one range
    // at every size and are chains of four dependent operations a term: below
    // 384 threads per SM narrower columns hide them better (us per step, 16-byte
    // / narrower: 20.3 / 12.3 at 4096 particles in BF16, 29.9 / 20.0 at 10007 and
    // 48.2 / 42.5 at 50000 in FP32, 68.3 / 58.6 at 100003 in BF16; above it
    // 68.8 / 75.4 at 100003 in FP32).
    if (sh.kind == 0 && !(KAHAN && bytes / 16 < 384LL * kChipSms)) {
        auto k = hist_conv_col<NACC, KAHAN, BF16, true>;
        const cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        k<<<sh.grid, sh.block, smem, st>>>((const typename Col<BF16>::V*)ring, 3LL * n_pad / Col<BF16>::W, H, coef, M,
                                           nstep, step, out, bp);
    } else {
        const int vb = bytes / 16 >= 512LL * kChipSms ? 16 : bytes / 8 >= 512LL * kChipSms ? 8 : 4;
        auto k = vb == 16 ? conv_tail<NACC, KAHAN, BF16, 16>
                          : vb == 8 ? conv_tail<NACC, KAHAN, BF16, 8> : conv_tail<NACC, KAHAN, BF16, 4>;
        const cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        const int C = (int)(bytes / vb), block = vb == 4 ? 128 : kThreads;
        k<<<(unsigned)((C + block - 1) / block), block, smem, st>>>(ring, n_pad, H, M, coef, nstep, step, bp, sh.G, out);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_hist_conv_part(const Shape& sh, int nacc, int kahan, const void* ring, int bf16, int n_pad, int M,
                                  const long long* nstep, long long step, const float* coef, float* out,
                                  const BlockPos& bp, cudaStream_t st)
{
    return by_nacc(nacc, kahan != 0, [&](auto na, auto ka) {
        constexpr int N = decltype(na)::value;
        constexpr bool K = decltype(ka)::value;
        return bf16 ? part_launch<N, K, true>(sh, ring, n_pad, M, nstep, step, coef, out, bp, st)
                    : part_launch<N, K, false>(sh, ring, n_pad, M, nstep, step, coef, out, bp, st);
    });
}

cudaError_t launch_batch_conv(const BatchPlan& bp, int step, cudaStream_t st)
{
    if (!bp.n_conv) return cudaSuccess;
    const int len = pre_len(bp.kahan, 1), t = step < 0 ? -1 : step % len;
    if (bp.n_pre && t == 0) {
        const cudaError_t e = by_pre(bp.nacc, bp.kahan, bp.bf16, len, [&](auto na, auto ln, auto ka, auto bf, int a0, int p) {
            return b_pre_launch<decltype(na)::value, decltype(ln)::value, decltype(ka)::value, decltype(bf)::value>(
                bp, a0, p, st);
        });
        if (e != cudaSuccess) return e;
    }
    return by_nacc(bp.nacc, bp.kahan != 0, [&](auto na, auto ka) {
        return launch_b_conv_t<decltype(na)::value, decltype(ka)::value>(bp, t, st);
    });
}

// (two streams per thread: the batch's blocks have 16 steps, or compensated sums)
int batch_pre_tiles(int n_pad) { return (3 * n_pad / 2 + kPreThreads - 1) / kPreThreads; }
static_assert(pre_streams(16, false) == 2 && pre_streams(8, true) == 2, "tiles of a batch");

// (pairs of accumulators in one launch, an odd last one in another)
int conv_pre_launches(int nacc) { return (nacc > 1) + (nacc & 1); }

cudaError_t launch_conv_pre(const void* ring, int bf16, int n_pad, int m_max, const long long* nstep, const float* coef,
                            int nacc, float* part, int G, int len, int kahan, cudaStream_t st)
{
    return by_pre(nacc, kahan, bf16, len, [&](auto na, auto ln, auto ka, auto bf, int a0, int p) {
        return pre_launch<decltype(na)::value, decltype(ln)::value, decltype(ka)::value, decltype(bf)::value>(
            ring, n_pad, m_max, coef, nacc, nstep, part, a0, p, G, st);
    });
}

}  // namespace gld
