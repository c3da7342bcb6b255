// k_history.cu -- the history convolution of Eq. dissipative_force2.
//
// For every particle i and component c the dissipative force needs
//   S_i      = sum_{m=1}^{m_max-1} K^s_m       dR_{i,n-m}     (self term)
//   P_{i,q}  = sum_{m=1}^{m_max-1} g_q[m]      dR_{i,n-m}     (pair terms)
//   Ps_{i,q} = sum_{m=1}^{m_max-1} gs_q[m]     dR_{i,n-m}     (dK^s terms)
// With separable kernels K^p_m(r) = sum_q f_q(r) g_q[m] the pair sums of
// Eq. dissipative_force2 become sum_j f_q(r_ij) e e^T P_{j,q}, so the history
// ring is streamed at most once per step, here (inside a block of steps only
// the part of it from the first rewritten slot on: k_history_blk.cu).  This is
// the step that sets the cost: 12 (m_max-1) bytes per particle (FP32) against ~2 flops per
// byte per accumulator -- bound by HBM bandwidth, so no tensor cores.
//
// Layout: ring[slot][3][n_pad], slot = k mod (m_max-1) for dR_k.  Every slot
// is one contiguous row of 3 n_pad values; a thread owns one 16-byte column
// (4 consecutive values) and walks all slots with 8 loads in flight, so each
// warp reads 512 contiguous bytes per slot.  The ring is never rotated: the
// coefficients are (slot s holds m = ((n - s - 1) mod (m_max-1)) + 1),
// staged in shared memory.
//
// Launch shape: the block size is picked from the occupancy of the
// instantiation so that every column gets its own thread in ONE wave; a
// second partial wave would leave a handful of CTAs streaming alone at the
// end (measured: 768 CTAs on 760 resident slots cost +50 % at 262144
// particles).  Only when the columns exceed one full wave does the grid
// become persistent, each thread taking columns q, q + grid, ...
#include "history.cuh"

namespace gld {

namespace {

// Launch shape (see the header).  Registers are allocated per warp, so small
// blocks can use every warp slot the registers allow (44 registers: 42 warps
// per SM, but only 40 in 128-thread blocks).  Returns the largest block size
// among 256..64 with which one wave of `kern` covers `items` threads, or 0.
template <class K>
cudaError_t one_wave_block(K kern, long long items, size_t smem, int* block, long long* best_cap, int* best_b)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    *block = 0;
    for (int b : {256, 128, 96, 64}) {
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, b, smem);
        if (e != cudaSuccess) return e;
        const long long cap = (long long)occ * sms * b;  // resident threads
        if (cap > *best_cap) {
            *best_cap = cap;
            *best_b = b;
        }
        if (cap >= items && *block == 0) *block = b;
    }
    return cudaSuccess;
}

template <int NACC, bool KAHAN, bool BF16>
cudaError_t choose_shape(long long cols, int H, size_t smem, Shape* out)
{
    // (the kernels without parts decide: the split of a column's slots, and so
    // the order of its sum, does not depend on whether the step is in a block)
    auto kc = hist_conv_col<NACC, KAHAN, BF16, false>;
    auto kg = hist_conv<NACC, KAHAN, BF16>;
    cudaError_t e = allow_smem(kc, smem);
    if (e == cudaSuccess) e = allow_smem(kg, smem);
    if (e != cudaSuccess) return e;
    int b1 = 0, bcap_b = kThreads;
    long long bcap = 0;
    e = one_wave_block(kc, cols, smem, &b1, &bcap, &bcap_b);
    if (e != cudaSuccess) return e;
    // Room for twice the threads in one wave: split each column's slots (not
    // with compensated sums, which stay one sequence over all m).
    int G = 1, bg = 0, gcap_b = kThreads;
    long long gcap = 0;
    for (int g = 4; g >= 2 && b1 && !KAHAN; g /= 2) {
        if (H < 16 * g) continue;
        int b = 0;
        gcap = 0;
        if ((e = one_wave_block(kg, cols * g, smem, &b, &gcap, &gcap_b)) != cudaSuccess) return e;
        if (b && b / g >= 32) {
            G = g;
            bg = b;
            break;
        }
    }
    if (G > 1) {
        const int per = bg / G;
        *out = Shape{1, bg, G, (unsigned)((cols + per - 1) / per)};
    } else if (b1) {
        *out = Shape{0, b1, 1, (unsigned)((cols + b1 - 1) / b1)};
    } else {
        // more columns than one wave: a persistent grid of the resident CTAs
        long long cap = 0;
        int b = 0, cb = kThreads;
        if ((e = one_wave_block(kg, cols, smem, &b, &cap, &cb)) != cudaSuccess) return e;
        *out = Shape{1, cb, 1, (unsigned)std::max(1LL, cap / cb)};
    }
    return cudaSuccess;
}

template <int NACC, bool KAHAN, bool BF16>
cudaError_t shape_of(int n_pad, int M, Shape* out)
{
    static std::mutex mu;
    static std::map<std::tuple<int, long long, int>, Shape> cache;
    const int H = M - 1;
    const long long cols = 3LL * n_pad / Col<BF16>::W;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find({dev, cols, H});
    if (it == cache.end()) {
        Shape sh{};
        if ((e = choose_shape<NACC, KAHAN, BF16>(cols, H, sizeof(float) * (size_t)H * NACC, &sh)) != cudaSuccess)
            return e;
        it = cache.emplace(std::make_tuple(dev, cols, H), sh).first;
    }
    *out = it->second;
    return cudaSuccess;
}

template <int NACC, bool KAHAN, bool BF16>
cudaError_t launch_tb(const void* ring, int n_pad, int M, const long long* nstep, long long step, const float* coef,
                      float* out, const BlockPos& bp, cudaStream_t st)
{
    Shape sh{};
    const cudaError_t e = shape_of<NACC, KAHAN, BF16>(n_pad, M, &sh);
    if (e != cudaSuccess) return e;
    if (bp.t >= 0) return launch_hist_conv_part(sh, NACC, KAHAN, ring, BF16, n_pad, M, nstep, step, coef, out, bp, st);
    using V = typename Col<BF16>::V;
    const int H = M - 1;
    const size_t smem = sizeof(float) * (size_t)H * NACC;
    const long long cols = 3LL * n_pad / Col<BF16>::W;
    if (sh.kind == 0)
        hist_conv_col<NACC, KAHAN, BF16, false><<<sh.grid, sh.block, smem, st>>>((const V*)ring, cols, H, coef, M, nstep,
                                                                                 step, out, bp);
    else
        hist_conv<NACC, KAHAN, BF16><<<sh.grid, sh.block, smem, st>>>((const V*)ring, cols, H, coef, M, nstep, step, out,
                                                                      sh.G);
    return cudaGetLastError();
}

template <int NACC, bool KAHAN>
cudaError_t launch_t(const void* ring, int bf16, int n_pad, int M, const long long* nstep, long long step,
                     const float* coef, float* out, const BlockPos& bp, cudaStream_t st)
{
    return bf16 ? launch_tb<NACC, KAHAN, true>(ring, n_pad, M, nstep, step, coef, out, bp, st)
                : launch_tb<NACC, KAHAN, false>(ring, n_pad, M, nstep, step, coef, out, bp, st);
}

cudaError_t dispatch(int nacc, int kahan, const void* ring, int bf16, int n_pad, int M, const long long* nstep,
                     long long step, const float* coef, float* out, const BlockPos& bp, cudaStream_t st)
{
    return by_nacc(nacc, kahan != 0, [&](auto na, auto ka) {
        return launch_t<decltype(na)::value, decltype(ka)::value>(ring, bf16, n_pad, M, nstep, step, coef, out, bp, st);
    });
}

cudaError_t shape_for(int bf16, int n_pad, int m_max, int nacc, int kahan, Shape* sh)
{
    return by_nacc(nacc, kahan != 0, [&](auto na, auto ka) {
        return bf16 ? shape_of<decltype(na)::value, decltype(ka)::value, true>(n_pad, m_max, sh)
                    : shape_of<decltype(na)::value, decltype(ka)::value, false>(n_pad, m_max, sh);
    });
}

}  // namespace

cudaError_t conv_block_shape(int bf16, int n_pad, int m_max, int nacc, int kahan, int* G, int* len, size_t* bytes)
{
    *G = *len = 0;
    *bytes = 0;
    if (m_max - 1 < (kahan ? 2 : 1) * kMinBlockedSlots) return cudaSuccess;
    Shape sh{};
    const cudaError_t e = shape_for(bf16, n_pad, m_max, nacc, kahan, &sh);
    if (e != cudaSuccess) return e;
    *G = sh.G;
    *len = pre_len(kahan, sh.G);
    const int rows = std::max(sh.G * *len, pre_len(kahan, 1));  // alone, and in a batch (one range)
    *bytes = sizeof(float) * (size_t)rows * nacc * (kahan ? 2 : 1) * 3 * n_pad;
    return cudaSuccess;
}

// A system alone runs the convolution beside its list build and F^C, so blocks
// have to save more than their parts' launch: the ring must be long, the longer
// the fewer its columns.  Time per step with whole sums over time with blocks at
// H slots (one pair term, graphs; 3 and 11 neighbours in a list):
//   FP32            4097: 0.95-0.98 at 160, 1.00-1.08 at 200    8192: 0.98-1.01 at 128, 1.05-1.08 at 160
//                  16384: 0.96-1.07 at 100, 0.99-1.14 at 128   40000: 1.00-1.02 at 80, 1.03-1.07 at 100
//                  65536: 1.00-1.09 at 64, 1.05-1.16 at 100   262144: 1.03 at 32, 1.11 at 64, 1.22 at 128
//                 600000: 0.98 at 49, 1.06 at 64, 1.18 at 128
//   BF16            8192: 0.98-1.00 at 128, 1.05-1.10 at 160   20000: 1.01 at 128, 1.11 at 160
//                 100000: 1.02 at 128, 1.07-1.08 at 160       160000: 0.99 at 80, 1.01 at 100, 1.04 at 128
//                 262144: 1.00 at 49, 1.03 at 64              600000: 0.98 at 49, 1.03 at 64
// Compensated sums have one range at every size and are bound by operations once
// their columns fill the chip; blocks save loads, not operations.
//   FP32            8192: 0.98 at 80, 1.04 at 100              20000: 1.01 at 128, 1.08 at 160
//                  40000: 0.93-1.01 at 128, 0.98-1.09 at 160  160000: 0.98 at 49, 1.02 at 64, 1.09 at 128
//   BF16           20000: 1.02 at 80, 1.16 at 100              40000: 0.96-1.04 at 80, 1.07-1.17 at 100
//                 100000: 0.99-1.00 at 160, 1.06 at 200       262144: 0.96 at 32, 0.93 at 160, 0.95 at 300
bool conv_blocks_alone(int bf16, int n_pad, int m_max, int nacc, int kahan)
{
    const int H = m_max - 1;
    if (H < kMinBlockedSlots) return false;
    Shape sh{};
    if (shape_for(bf16, n_pad, m_max, nacc, kahan, &sh) != cudaSuccess) return false;
    const long long per_sm = 3LL * n_pad / (bf16 ? 8 : 4) / kChipSms;  // 16-byte columns
    if (kahan) {
        if (per_sm >= 512) return !bf16 && H >= 64;
        return H >= (bf16 ? (per_sm >= 192 ? 192 : 96) : per_sm >= 64 ? 160 : 96);
    }
    if (sh.G == 1) return H >= (sh.kind == 0 ? 32 : 56);  // (columns of one wave, or more)
    if (sh.G == 2) return H >= (bf16 ? 96 : 56);
    return H >= (bf16 ? 144 : per_sm >= 56 ? 96 : per_sm >= 32 ? 144 : 192);
}

cudaError_t launch_hist_conv(const void* ring, int bf16, int n_pad, int m_max, const Ctrl* ctrl,
                             long long step, const float* coef, int nacc, float* out, int kahan,
                             cudaStream_t st, const float* part, int t, int len)
{
    if (m_max < 2 || n_pad <= 0 || n_pad % 32 != 0 || nacc < 1 || nacc > kMaxAcc) return cudaErrorInvalidValue;
    const long long* nstep = ctrl ? &ctrl->step : nullptr;
    return dispatch(nacc, kahan, ring, bf16, n_pad, m_max, nstep, step, coef, out, BlockPos{part, t, len}, st);
}

cudaError_t launch_hist_conv_next(const void* ring, int bf16, int n_pad, int m_max, const Ctrl* ctrl,
                                  const float* coef, int nacc, float* out, int kahan, cudaStream_t st,
                                  const float* part, int t, int len)
{
    if (m_max < 2 || n_pad <= 0 || n_pad % 32 != 0 || nacc < 1 || nacc > kMaxAcc || !ctrl) return cudaErrorInvalidValue;
    return dispatch(nacc, kahan, ring, bf16, n_pad, m_max, &ctrl->conv_step, 0, coef, out, BlockPos{part, t, len}, st);
}

}  // namespace gld
