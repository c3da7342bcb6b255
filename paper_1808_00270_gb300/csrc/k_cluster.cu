// k_cluster.cu -- whole steps of a small system inside one kernel.
//
// A step of a few thousand particles is bound by latency: its kernels run 8 to
// 12 us each whatever the size, and a conditional graph node costs another 7
// us (29 us per step at 64 particles, 33 us at 4096).  Here one thread-block
// cluster (1 to 16 CTAs, hardware cluster barriers) takes a system through all
// steps of a noise block: per step two barriers, none of the launches,
//   conv    memory sums of the step (parts of a block of steps, then the rest
//           of the ring; one particle's three streams per thread)
//   -- barrier --
//   pair    F^D, R_{n+1}, the displacement into the ring, rebuild request
//   -- barrier --
//   (lists  when requested: cells by counting, neighbour lists; three barriers)
//   force   F^C_{n+1}, V_{n+1}, VACF terms
// A thread keeps its particles, so own data needs no barrier; positions swap
// between two buffers, so nothing that others read is overwritten before the
// next barrier.  All sums run in the order of the kernels for single systems
// (k_particles.cu, k_history*.cu): the same bits.  Batches keep their tile kernels:
// a cluster per small member left the chip's other SMs waiting for the longest
// member (226 to 300 us per step of 64 systems against 192).
//
// Arrays that other CTAs write during the kernel are read by plain loads
// behind the cluster barrier (release / acquire), never through the read-only
// path.
#include <algorithm>
#include <cmath>

#include <cuda_bf16.h>

#include "cluster_fit.h"
#include "history.cuh"
#include "neighbours.cuh"

namespace gld {

namespace {

// (Without .aligned: the barriers stand behind loops that lanes leave one by one,
// and nothing obliges the compiler to bring a warp together before inline
// assembly.  us per step without / with it: 7.42 / 7.40 at 64 particles, 15.94 /
// 15.91 at 2048, 18.75 / 18.78 at 4096.)
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Data written by other CTAs: plain loads.
__device__ __forceinline__ float4 ld4(const float4* p) { return LdPlain::f4(p); }
__device__ __forceinline__ float ld1(const float* p) { return LdPlain::f1(p); }
__device__ __forceinline__ int ldi(const int* p) { return LdPlain::i1(p); }

struct ClSched {  // the VACF's view of a step (vacf_schedule in k_particles.cu)
    int on, nact, slot0, origin, lag0, buf, pending;
    int pv_nact, pv_lag0, pv_buf;
};

__device__ __forceinline__ void cl_schedule(const StepParams& P, ClSched& c, long long t)
{
    c.pv_nact = c.pending ? c.nact : 0;
    c.pv_lag0 = c.lag0;
    c.pv_buf = c.buf;
    c.pending = 0;
    c.buf ^= 1;
    if (t < P.vacf_burnin) {
        c.on = 0;
        return;
    }
    const long long rel = t - P.vacf_burnin;
    const long long o_now = rel / P.vacf_stride;
    const int lag0 = (int)(rel - o_now * P.vacf_stride);
    int n_act = 0;
    for (int j = 0; j < P.n_os; ++j)
        if (o_now - j >= 0 && lag0 + (long long)j * P.vacf_stride < P.vacf_len) n_act = j + 1;
    c.on = 1;
    c.nact = n_act;
    c.slot0 = (int)(o_now % P.n_os);
    c.origin = lag0 == 0;
    c.lag0 = lag0;
}

__device__ __forceinline__ float cl_warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void cl_two_sum(float a, float b, float& s, float& e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void cl_df_add(float& hi, float& lo, float bhi, float blo)
{
    float s, e;
    cl_two_sum(hi, bhi, s, e);
    e += lo + blo;
    hi = s + e;
    lo = e - (hi - s);
}

// Exclusive scan over the CTA; returns the total.
__device__ int cl_scan(int v, int* excl)
{
    __shared__ int tot[kClThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tot[w] = x;
    __syncthreads();
    int base = 0, all = 0;
    for (int k = 0; k < kClThreads / 32; ++k) {
        if (k < w) base += tot[k];
        all += tot[k];
    }
    __syncthreads();
    *excl = base + x - v;
    return all;
}

// vacf_fold of one origin by one warp: block partials b = 32 w + lane < 256 in
// the tree of warp w, the eight warps' sums in order.
__device__ __forceinline__ void cl_fold(const float* base, int nblk, double* csum, long long* ccnt)
{
    const int lane = threadIdx.x & 31;
    const double s0 = __ldcg(csum);
    const long long k0 = __ldcg(ccnt);
    float h = 0.f, l = 0.f;
    for (int w = 0; 32 * w < nblk; ++w) {  // (a warp without partials adds exactly nothing)
        const int b = 32 * w + lane;
        float hi = b < nblk ? ld1(base + b) : 0.f, lo = 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
            cl_df_add(hi, lo, h2, l2);
        }
        cl_df_add(h, l, hi, lo);
    }
    if (lane == 0) {
        __stcg(csum, s0 + ((double)h + (double)l));
        __stcg(ccnt, k0 + 1);
    }
}

// The VACF terms of V_t (the fused form of cforce_vacf): folds the previous
// time's partials, then the partial sums of blocks of 256 particles (8 warps).
__device__ __forceinline__ void cl_vacf(const StepParams& P, const ParticleBuffers& B, ClSched& vs, long long t, int rank,
                                        int ncta)
{
    __shared__ float wsum[kClThreads / 32][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = P.n, nblk = B.vacf_gx;
    cl_schedule(P, vs, t);
    for (int q = rank + ncta * warp; q < vs.pv_nact; q += ncta * (kClThreads / 32)) {
        const int lg = vs.pv_lag0 + q * P.vacf_stride;
        cl_fold(B.vpartial + ((size_t)vs.pv_buf * P.n_os + q) * nblk, nblk, B.csum + lg, B.ccnt + lg);
    }
    if (!vs.on) return;
    vs.pending = 1;
    if (vs.origin && rank == 0 && tid == 0) *B.norig += 1;
    float* out = B.vpartial + (size_t)vs.buf * P.n_os * nblk;
    // (block of 256 particles, 8 origins) by groups of 256 threads
    const int og = (vs.nact + 7) / 8, items = nblk * max(og, 1), grp = 2 * rank + (tid >> 8);
    for (int k0 = 0; k0 < items; k0 += 2 * ncta) {  // the same rounds for all threads
        const int k = k0 + grp, blk = k < items ? k % nblk : 0, q0 = k < items ? k / nblk * 8 : 0;
        const int i = blk * 256 + (tid & 255), left = k < items ? min(8, vs.nact - q0) : 0;
        const bool valid = i < n && k < items;
        const float4 v = valid ? ld4(B.vel + i) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = q0 + q;
            const int sl = vs.slot0 - j < 0 ? vs.slot0 - j + P.n_os : vs.slot0 - j;
            const bool use = valid && q < left && !(j == 0 && vs.origin);
            w[q] = use ? ld4(B.vorig + (size_t)sl * n + i) : v;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float dv = valid && q < left ? fmaf(v.x, w[q].x, fmaf(v.y, w[q].y, v.z * w[q].z)) : 0.f;
            const float sq = cl_warp_sum(dv);
            if (lane == 0) wsum[warp][q] = sq;
        }
        __syncthreads();
        if ((tid & 255) < left) {
            float sb = 0.f;
            for (int w2 = 0; w2 < 8; ++w2) sb += wsum[(warp & ~7) + w2][tid & 255];
            out[(size_t)(q0 + (tid & 255)) * nblk + blk] = sb;
        }
        __syncthreads();
        if (vs.origin && valid && q0 == 0) B.vorig[(size_t)vs.slot0 * n + i] = v;
    }
}

// Neighbour lists at R (the lists of nbr_build: ids within r_c + skin, sorted)
// by one cluster, L lanes per particle; lists: scratch [kClThreads / L][maxnb].
// A thread-per-particle walk of the 27 cells is a chain of some 60 dependent
// loads (40 to 50 us whatever the size); here cells keep their particles in
// the order of a scan, so the stencil is nine or ten ranges, shared by lanes.
template <int L>
__device__ __forceinline__ void cl_rebuild(const StepParams& P, const ParticleBuffers& B, const float4* nxt, int* lists,
                                           int rank, int ncta)
{
    __shared__ int lcnt[kClThreads / L], cbase[kClMaxCtas];
    Ctrl* ctrl = B.ctrl;
    const int n = P.n, tid = threadIdx.x, np = P.n_pad;
    const int lane = tid & (L - 1), grp = tid / L;
    const unsigned gmask = ((1u << L) - 1u) << ((tid & 31) & ~(L - 1));
    const int pstride = ncta * (kClThreads / L), p0 = rank * (kClThreads / L) + grp;
    const int iters = (n + pstride - 1) / pstride;
    const int cthreads = ncta * kClThreads, g0 = rank * kClThreads + tid;
    int shift = 0;  // cells per CTA: 2^shift
    while ((ncta << shift) < B.ncells) ++shift;
    auto barrier = [&]() {
        if (ncta == 1) __syncthreads();
        else cluster_barrier();
    };
    // particles counted into cells; their rank in the cell
    for (int i = g0; i < n; i += cthreads)
        B.cell_next[i] = atomicAdd(B.cell_count + cell_of(ld4(nxt + i), P), 1);
    if (g0 == 0) ctrl->rebuilds += 1;
    barrier();
    // starts within the CTA's 2^shift cells, and the CTA's total
    const int c0 = rank << shift, c1 = min(B.ncells, c0 + (1 << shift));
    int run = 0;
    for (int cb = c0; cb < c0 + (1 << shift); cb += kClThreads) {  // uniform over the CTA
        const int c = cb + tid, k = c < c1 ? ldi(B.cell_count + c) : 0;
        int excl;
        const int tot = cl_scan(k, &excl);
        if (c < c1) {
            B.cell_start[c] = run + excl;
            B.cell_count[c] = 0;
        }
        run += tot;
    }
    if (tid == 0) B.chunk_sum[rank] = run;
    barrier();
    if (tid < 32) {  // particles in earlier CTAs' cells
        int v = tid < ncta ? ldi(B.chunk_sum + tid) : 0, x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (tid >= o) x += y;
        }
        if (tid < ncta) cbase[tid] = x - v;
    }
    __syncthreads();
    auto start = [&](int c) { return c < B.ncells ? ldi(B.cell_start + c) + cbase[c >> shift] : n; };
    for (int i = g0; i < n; i += cthreads) {
        const float4 x = ld4(nxt + i);
        B.pos_sorted[start(cell_of(x, P)) + B.cell_next[i]] = make_float4(x.x, x.y, x.z, __int_as_float(i));
    }
    barrier();
    // a row of three cells along x is one range of particles, or two at
    // the box's faces; lane l takes the rows l, l + L, ... of the nine
    // (one cell: its particles l, l + L, ...); candidates meet in shared
    // memory and go to the place of their id's rank
    int* list = lists + grp * P.maxnb;
    for (int it = 0; it < iters; ++it) {
        const int i = p0 + it * pstride;
        if (i >= n) break;  // uniform over the lanes of a particle
        if (lane == 0) lcnt[grp] = 0;
        __syncwarp(gmask);
        const float4 pi = ld4(nxt + i);
        const int nc = P.nc;
        auto test = [&](const float4 pj) {
            const int jd = __float_as_int(pj.w);
            const float dx = min_image(pi.x, pj.x, P.box, P.half_box);
            const float dy = min_image(pi.y, pj.y, P.box, P.half_box);
            const float dz = min_image(pi.z, pj.z, P.box, P.half_box);
            if (jd != i && dist2(dx, dy, dz) < P.rl2) {
                const int k = atomicAdd(lcnt + grp, 1);
                if (k < P.maxnb) list[k] = jd;
            }
        };
        if (nc == 1) {
            for (int q = lane; q < n; q += L) test(ld4(B.pos_sorted + q));
        } else {
            constexpr int R = (9 + L - 1) / L;  // rows of a lane
            const int cx = cell_coord(pi.x, P.inv_cell, nc), cy = cell_coord(pi.y, P.inv_cell, nc),
                      cz = cell_coord(pi.z, P.inv_cell, nc);
            int b0[R], n0[R], b1[R], n1[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int o = lane + r * L;
                int z = cz + o / 3 - 1, y = cy + o % 3 - 1;
                z = z < 0 ? z + nc : (z >= nc ? z - nc : z);
                y = y < 0 ? y + nc : (y >= nc ? y - nc : y);
                const int base = (z * nc + y) * nc;
                const int xa = max(cx - 1, 0), xb = min(cx + 1, nc - 1);       // the row inside the box
                const int xw = cx == 0 ? nc - 1 : cx == nc - 1 ? 0 : -1;       // the cell across a face
                b0[r] = n0[r] = b1[r] = n1[r] = 0;
                if (o < 9) {
                    b0[r] = start(base + xa);
                    n0[r] = start(base + xb + 1) - b0[r];
                    if (xw >= 0) {
                        b1[r] = start(base + xw);
                        n1[r] = start(base + xw + 1) - b1[r];
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                for (int q = 0; q < n0[r] + n1[r]; q += 4) {
                    float4 pj[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int k = q + u < n0[r] + n1[r] ? q + u : q;
                        pj[u] = ld4(B.pos_sorted + (k < n0[r] ? b0[r] + k : b1[r] + k - n0[r]));
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (q + u < n0[r] + n1[r]) test(pj[u]);
                }
        }
        __syncwarp(gmask);
        int c = lcnt[grp];
        if (c > P.maxnb) {
            if (lane == 0) atomicOr(&ctrl->err, kErrNbrOverflow);
            c = P.maxnb;
        }
        for (int s = lane; s < c; s += L) {
            const int v = list[s];
            int r = 0;
            for (int k = 0; k < c; ++k) r += list[k] < v;
            B.nbr[(size_t)r * np + i] = v;
        }
        if (lane == 0) {
            B.nbr_cnt[i] = c;
            B.disp_build[i] = ld4(B.disp + i);
        }
        __syncwarp(gmask);  // the scratch is read before the next particle's; the lists before the forces
    }
}

// Two adjacent streams of a ring row.
template <bool BF16>
__device__ __forceinline__ uint2 ring_pair(const char* p)
{
    uint2 r;
    if constexpr (BF16) {
        uint32_t w;
        asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
        r = make_uint2(w << 16, w & 0xffff0000u);
    } else {
        asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p) : "memory");
    }
    return r;
}

// Memory sums of the step that writes slot h (tail_body and pre_body of
// k_history_blk.cu, two streams per thread): fresh forms the parts of the block
// that starts here; t is the step's number in its block (-1: no parts).
// cs: weights [m][NACC], zero past H.
template <int NACC, bool BF16>
__device__ __forceinline__ void cl_conv(const StepParams& P, const ParticleBuffers& B, const float* cs, int h, bool fresh,
                                        int t, int G, int len, int q0, int qstride)
{
    constexpr int U = 16;
    const int H = P.H, C = 3 * P.n_pad / 2;
    const size_t rowb = (size_t)C * (BF16 ? 4 : 8);  // bytes of a ring row
    const uint32_t none = (uint32_t)H >> 16;         // 0 (see k_history_blk.cu)
    const int hb = t > 0 ? (h - t < 0 ? h - t + H : h - t) : h;  // slot of the block's first step
    for (int q = q0; q < C; q += qstride) {
        const char* ring = (const char*)B.ring + (size_t)q * (BF16 ? 4 : 8);
        float2* part = (float2*)B.part + q;
        if (fresh)
#pragma unroll 1
            for (int g = 0; g < G; ++g) {
                const int lo = (int)((unsigned)(g * H) / (unsigned)G), hi = (int)((unsigned)((g + 1) * H) / (unsigned)G);
                const int e = first_rewritten(lo, hi, h, len, H);
                if (e <= lo) continue;
                int ml = h - (e - 1);  // weight of slot e - 1 at the block's first step
                if (ml <= 0) ml += H;
#pragma unroll 1
                for (int t0 = 0; t0 < len; t0 += 8) {
                    float2 acc[NACC][8];
#pragma unroll
                    for (int a = 0; a < NACC; ++a)
#pragma unroll
                        for (int v = 0; v < 8; ++v) acc[a][v] = make_float2(0.f, 0.f);
                    const char* p = ring + (size_t)lo * rowb;
                    const float* wr = cs + (ml + t0) * NACC;  // row s, step t0 + v: wr[(e - 1 - s + v) NACC + a]
                    int s = lo;
                    for (; s + 8 <= e; s += 8) {
                        uint2 x[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            x[u] = ring_pair<BF16>(p);
                            p += rowb;
                        }
                        const float* w0 = wr + (e - 1 - s - 7) * NACC + (x[7].x & none);
#pragma unroll
                        for (int a = 0; a < NACC; ++a) {
                            float w[15];
#pragma unroll
                            for (int v = 0; v < 15; ++v) w[v] = w0[v * NACC + a];
#pragma unroll
                            for (int u = 0; u < 8; ++u)
#pragma unroll
                                for (int v = 0; v < 8; ++v) {
                                    acc[a][v].x = fmaf(w[7 - u + v], __uint_as_float(x[u].x), acc[a][v].x);
                                    acc[a][v].y = fmaf(w[7 - u + v], __uint_as_float(x[u].y), acc[a][v].y);
                                }
                        }
                    }
                    for (; s < e; ++s) {
                        const uint2 x = ring_pair<BF16>(p);
                        p += rowb;
#pragma unroll
                        for (int a = 0; a < NACC; ++a)
#pragma unroll
                            for (int v = 0; v < 8; ++v) {
                                const float w = wr[(e - 1 - s + v) * NACC + a];
                                acc[a][v].x = fmaf(w, __uint_as_float(x.x), acc[a][v].x);
                                acc[a][v].y = fmaf(w, __uint_as_float(x.y), acc[a][v].y);
                            }
                    }
#pragma unroll
                    for (int a = 0; a < NACC; ++a)
#pragma unroll
                        for (int v = 0; v < 8; ++v) part[part_row(g, t0 + v, a, 0, len, NACC, 1) * C] = acc[a][v];
                }
            }
        float2 tot[NACC];
#pragma unroll 1
        for (int g = 0; g < G; ++g) {
            const int lo = (int)((unsigned)(g * H) / (unsigned)G), hi = (int)((unsigned)((g + 1) * H) / (unsigned)G);
            const int first = t < 0 ? lo : first_rewritten(lo, hi, hb, len, H);
            float2 acc[NACC];
#pragma unroll
            for (int a = 0; a < NACC; ++a)
                acc[a] = first > lo ? part[part_row(g, t, a, 0, len, NACC, 1) * C] : make_float2(0.f, 0.f);
            // slot s holds dR_{n-m}, m = h - s before slot h and h - s + H from it on
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                int s = half ? max(first, h) : first;
                const int end = half ? hi : min(hi, h);
                if (s >= end) continue;
                const char* p = ring + (size_t)s * rowb;
                const float* w = cs + (half ? h - s + H : h - s) * NACC;
                for (; s + U <= end; s += U) {
                    uint2 x[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        x[u] = ring_pair<BF16>(p);
                        p += rowb;
                    }
                    const float* w0 = w + (x[U - 1].x & none);
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int a = 0; a < NACC; ++a) {
                            acc[a].x = fmaf(w0[a - u * NACC], __uint_as_float(x[u].x), acc[a].x);
                            acc[a].y = fmaf(w0[a - u * NACC], __uint_as_float(x[u].y), acc[a].y);
                        }
                    w -= U * NACC;
                }
                if (s < end) {  // the last rows in flight together too (past the end: the last row again, unused)
                    uint2 x[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        x[u] = ring_pair<BF16>(p);
                        if (s + u + 1 < end) p += rowb;
                    }
                    const float* w0 = w + (x[U - 1].x & none);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (s + u < end)
#pragma unroll
                            for (int a = 0; a < NACC; ++a) {
                                acc[a].x = fmaf(w0[a - u * NACC], __uint_as_float(x[u].x), acc[a].x);
                                acc[a].y = fmaf(w0[a - u * NACC], __uint_as_float(x[u].y), acc[a].y);
                            }
                }
            }
#pragma unroll
            for (int a = 0; a < NACC; ++a)
                tot[a] = g == 0 ? acc[a] : make_float2(tot[a].x + acc[a].x, tot[a].y + acc[a].y);
        }
#pragma unroll
        for (int a = 0; a < NACC; ++a) ((float2*)B.conv)[(size_t)a * C + q] = tot[a];
    }
}

// Steps of one system.  NACC 1: self kernel only; 2: one separable pair term.
// L lanes share a particle (neighbours.cuh).
// The convolution's blocks have G ranges and len steps; rel0 is the number of
// the first step in its block (> 0: the block's parts are formed).
template <int NACC, bool BF16, int L>
__device__ __forceinline__ void cl_steps(const SysDesc& d, int nsteps, int rel0, int G, int len, int rank,
                                         int ncta)
{
    constexpr int E = L >= 8 ? 2 : 4;
    extern __shared__ float cs[];  // weights [M + len][NACC]: w_a[m], zero past H; then list scratch
    const StepParams& P = d.P;
    const ParticleBuffers& B = d.B;
    Ctrl* ctrl = B.ctrl;
    const int H = P.H, M = P.m_max, n = P.n, tid = threadIdx.x, np = P.n_pad;
    const int ncs = M + len;
    for (int x = tid; x < NACC * ncs; x += kClThreads) {
        const int m = x / NACC, a = x - m * NACC;
        cs[x] = m >= 1 && m <= H ? __ldg(d.coef + (size_t)a * M + m) : 0.f;
    }
    int* lists = (int*)(cs + NACC * ncs);  // [kClThreads / L][maxnb]
    const Lanes<L> ln;
    const int lane = ln.lane, grp = tid / L;
    const int pstride = ncta * (kClThreads / L), p0 = rank * (kClThreads / L) + grp;
    const int iters = (n + pstride - 1) / pstride;
    const int cthreads = ncta * kClThreads, g0 = rank * kClThreads + tid;
    const size_t S = 3 * (size_t)np;
    long long step = ctrl->step;
    int h = (int)ctrl->hslot;
    const long long noise_n0 = ctrl->noise_n0;
    ClSched vs{};
    const bool vacf = P.vacf_len > 0;
    if (vacf) {
        vs.on = ctrl->vacf_on;
        vs.nact = ctrl->vacf_nact;
        vs.slot0 = ctrl->vacf_slot0;
        vs.origin = ctrl->vacf_origin;
        vs.lag0 = ctrl->vacf_lag0;
        vs.buf = ctrl->vacf_buf;
        vs.pending = ctrl->vacf_pending;
    }
    float4 *cur = B.pos, *nxt = B.pos_next;
    static_assert(sizeof(Ctrl::rebuild) == 2 * sizeof(int), "requests of even and odd steps");
    int* flags = ctrl->rebuild;
    const float g00 = NACC > 1 ? __ldg(B.g0) : 0.f;
    int rel = rel0;
    auto barrier = [&]() {
        if (ncta == 1) __syncthreads();
        else cluster_barrier();
    };
    __syncthreads();

    for (int st = 0; st < nsteps; ++st, ++step) {
        // ---- memory sums ---------------------------------------------------
        cl_conv<NACC, BF16>(P, B, cs, h, P.cblk && rel == 0, P.cblk ? rel : -1, G, len, g0, cthreads);
        barrier();

        // ---- VACF of V_n; F^D, position update (pair_force_integrate) -------
        if (vacf && st > 0) cl_vacf(P, B, vs, step, rank, ncta);
        const int par = (int)(step & 1);
        if (rank == 0 && tid == 0) flags[par ^ 1] = 0;  // read by all before the last barrier
        const long long row = step - noise_n0;
        const bool row_ok = row >= 0 && row < P.T;
        if (!row_ok && rank == 0 && tid == 0) atomicOr(&ctrl->err, kErrNoise);
        for (int it = 0; it < iters; ++it) {
            const int i = p0 + it * pstride;
            if (i >= n) break;  // uniform over the lanes of a particle
            const float4 pi = ld4(cur + i);
            // the finishing lane's own data, loaded ahead of the neighbours'
            float4 vi, fci, dd, db;
            float fr[3] = {0.f, 0.f, 0.f}, sx[3];
            if (lane == 0) {
                vi = ld4(B.vel + i);
                fci = ld4(B.fc + i);
                dd = ld4(B.disp + i);
                db = ld4(B.disp_build + i);
                const float* f = B.frblock + (size_t)row * S + i;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if (row_ok) fr[c] = ld1(f + c * np);
                    sx[c] = ld1(B.conv + c * np + i);
                }
            }
            float f0x = 0.f, f0y = 0.f, f0z = 0.f, fhx = 0.f, fhy = 0.f, fhz = 0.f;
            if (NACC > 1) {
                float f0[3] = {0.f, 0.f, 0.f}, fh[3] = {0.f, 0.f, 0.f};
                pair_sums<LdPlain, L, E>(P, ln, cur, B.vel, B.conv + S, B.nbr + i, B.nbr_cnt + i, i, pi, B.ftab, g00, f0, fh);
                f0x = f0[0]; f0y = f0[1]; f0z = f0[2];
                fhx = fh[0]; fhy = fh[1]; fhz = fh[2];
            }
            if (lane != 0) continue;
            const float fdx = fmaf(fhx - sx[0], P.inv_dt, f0x);
            const float fdy = fmaf(fhy - sx[1], P.inv_dt, f0y);
            const float fdz = fmaf(fhz - sx[2], P.inv_dt, f0z);
            const float frx = fr[0], fry = fr[1], frz = fr[2];
            const float dRx = fmaf(P.pos_f, fci.x + fdx + frx, P.pos_v * vi.x);
            const float dRy = fmaf(P.pos_f, fci.y + fdy + fry, P.pos_v * vi.y);
            const float dRz = fmaf(P.pos_f, fci.z + fdz + frz, P.pos_v * vi.z);
            if (BF16) {
                __nv_bfloat16* hr = (__nv_bfloat16*)B.ring + (size_t)h * S + i;
                hr[0] = __float2bfloat16_rn(dRx);
                hr[np] = __float2bfloat16_rn(dRy);
                hr[2 * np] = __float2bfloat16_rn(dRz);
            } else {
                float* hr = (float*)B.ring + (size_t)h * S + i;
                hr[0] = dRx;
                hr[np] = dRy;
                hr[2 * np] = dRz;
            }
            nxt[i] = make_float4(wrap_box(__fadd_rn(pi.x, dRx), P.box), wrap_box(__fadd_rn(pi.y, dRy), P.box),
                                 wrap_box(__fadd_rn(pi.z, dRz), P.box), 0.f);
            B.vhalf[i] = make_float4(fmaf(P.vh_f, fdx + frx, fmaf(P.vh_fc, fci.x, P.vh_v * vi.x)),
                                     fmaf(P.vh_f, fdy + fry, fmaf(P.vh_fc, fci.y, P.vh_v * vi.y)),
                                     fmaf(P.vh_f, fdz + frz, fmaf(P.vh_fc, fci.z, P.vh_v * vi.z)), 0.f);
            B.fd[i] = make_float4(fdx, fdy, fdz, 0.f);
            const float4 dn = make_float4(dd.x + dRx, dd.y + dRy, dd.z + dRz, 0.f);
            B.disp[i] = dn;
            const float mx = dn.x - db.x, my = dn.y - db.y, mz = dn.z - db.z;
            if (mx * mx + my * my + mz * mz > P.trig2) atomicOr(flags + par, 1);
            if (!(isfinite(dRx) && isfinite(dRy) && isfinite(dRz))) {
                atomicOr(&ctrl->err, kErrNonFinite);
                atomicOr(flags + par, 1);
            }
        }
        barrier();

        // ---- neighbour lists at R_{n+1}, when requested ---------------------
        if (__ldcg(flags + par) != 0) {  // the same for the whole cluster
            cl_rebuild<L>(P, B, nxt, lists, rank, ncta);
        }

        // ---- F^C_{n+1}, V_{n+1} (cforce) ------------------------------------
        for (int it = 0; it < iters; ++it) {
            const int i = p0 + it * pstride;
            if (i >= n) break;
            const float4 pi = ld4(nxt + i);
            float4 vh;
            if (lane == 0) vh = ld4(B.vhalf + i);
            float f[3] = {0.f, 0.f, 0.f};
            cforce_sums<LdPlain, L, E>(P, ln, nxt, B.nbr + i, B.nbr_cnt + i, i, pi, B.fctab, f);
            const float fx = f[0], fy = f[1], fz = f[2];
            if (lane != 0) continue;
            B.fc[i] = make_float4(fx, fy, fz, 0.f);
            B.vel[i] = make_float4(fmaf(P.vf_fc, fx, vh.x), fmaf(P.vf_fc, fy, vh.y), fmaf(P.vf_fc, fz, vh.z), 0.f);
        }
        float4* sw = cur;
        cur = nxt;
        nxt = sw;
        h = h + 1 == H ? 0 : h + 1;
        rel = rel + 1 == len ? 0 : rel + 1;
    }
    barrier();  // V_n complete; all have read the flags and the step
    if (vacf) cl_vacf(P, B, vs, step, rank, ncta);
    // both position buffers hold R; control block as the step kernels leave it
    for (int i = g0; i < n; i += cthreads) nxt[i] = ld4(cur + i);
    if (rank == 0 && tid == 0) {
        flags[0] = flags[1] = 0;
        ctrl->step = step;
        ctrl->conv_step = step;
        ctrl->hslot = h;
        if (vacf) {
            ctrl->vacf_on = vs.on;
            ctrl->vacf_nact = vs.nact;
            ctrl->vacf_slot0 = vs.slot0;
            ctrl->vacf_origin = vs.origin;
            ctrl->vacf_lag0 = vs.lag0;
            ctrl->vacf_buf = vs.buf;
            ctrl->vacf_pending = vs.pending;
            ctrl->pv_nact = vs.pv_nact;
            ctrl->pv_lag0 = vs.pv_lag0;
            ctrl->pv_buf = vs.pv_buf;
        }
    }
}

__device__ __forceinline__ int cluster_rank()
{
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

template <int NACC, bool BF16, int L>
__global__ void __launch_bounds__(kClThreads, 1)
    steps_cluster(const __grid_constant__ SysDesc d, int nsteps, int rel0, int G, int len)
{
    cl_steps<NACC, BF16, L>(d, nsteps, rel0, G, len, cluster_rank(), (int)gridDim.x);
}

constexpr int kRebLanes = 4;

__global__ void __launch_bounds__(kClThreads, 1)
    rebuild_cluster(const __grid_constant__ StepParams P, const __grid_constant__ ParticleBuffers B)
{
    extern __shared__ int rlists[];
    if (B.ctrl->rebuild[0] == 0) return;  // the same for the whole cluster
    cl_rebuild<kRebLanes>(P, B, B.pos_next, rlists, cluster_rank(), (int)gridDim.x);
}

// A launch of one cluster of `ctas` CTAs.
struct ClusterLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    ClusterLaunch(int ctas, size_t smem, cudaStream_t st)
    {
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)ctas;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }
    ClusterLaunch(const ClusterLaunch&) = delete;
};

template <class... P, class... A>
cudaError_t launch_cluster(void (*kern)(P...), int ctas, size_t smem, cudaStream_t st, const A&... args)
{
    const cudaError_t e = allow_smem(kern, smem, true);
    if (e != cudaSuccess) return e;
    ClusterLaunch l(ctas, smem, st);
    return cudaLaunchKernelEx(&l.cfg, kern, args...);
}

template <class... P>
bool cluster_fits(void (*kern)(P...), int ctas, size_t smem)
{
    static ClusterFit fit;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return fit(dev, (const void*)kern, ctas, smem, [&](size_t bytes) {
        int active = 0;
        cudaError_t e = allow_smem(kern, bytes, true);
        if (e == cudaSuccess) {
            ClusterLaunch l(ctas, bytes, nullptr);
            e = cudaOccupancyMaxActiveClusters(&active, kern, &l.cfg);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return active;
    });
}

using StepsKernel = void (*)(const SysDesc, int, int, int, int);

// The instantiation, CTAs and shared memory for the steps of a system: eight
// lanes per particle, in up to 16 CTAs.
StepsKernel steps_kernel(const StepParams& P, int* ctas, size_t* smem)
{
    *ctas = cluster_ctas(P.n, 8);
    const int lanes = cluster_lanes(P.n, *ctas);
    *smem = sizeof(float) * P.nacc * (size_t)(P.m_max + pre_len(0, 1)) +  // (no block is longer)
            sizeof(int) * (size_t)(kClThreads / lanes) * (size_t)P.maxnb;
    auto of = [&](auto na, auto bf) -> StepsKernel {
        constexpr int N = decltype(na)::value;
        constexpr bool B = decltype(bf)::value;
        return lanes == 8 ? steps_cluster<N, B, 8> : lanes == 4 ? steps_cluster<N, B, 4> : steps_cluster<N, B, 2>;
    };
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    if (P.nacc == 1) return P.hist_bf16 ? of(I1{}, std::true_type{}) : of(I1{}, std::false_type{});
    return P.hist_bf16 ? of(I2{}, std::true_type{}) : of(I2{}, std::false_type{});
}

size_t rebuild_smem(const StepParams& P) { return sizeof(int) * (kClThreads / kRebLanes) * (size_t)P.maxnb; }

}  // namespace

bool cluster_ok(const StepParams& P, int kahan)
{
    if (P.n > kClusterMaxN || P.maxnb > 128 || kahan || P.perp || P.Qs > 0 || P.Q > 1 || P.nmodes > 0 || P.pn_deg > 0 ||
        P.pn_kry || P.pc_nbins > 0 || P.T != kMaxNoiseBlock)
        return false;
    int ctas = 0;
    size_t smem = 0;
    const StepsKernel kern = steps_kernel(P, &ctas, &smem);
    // long lists: the chip's other SMs win over the launches they cost (launch.h)
    const double list = P.n / ((double)P.box * P.box * P.box) * 4.18879020478639 * std::pow((double)P.rl2, 1.5);
    const int lanes = cluster_lanes(P.n, ctas);
    if (lanes < 8 && list > (lanes == 4 ? 24.0 : 8.0)) return false;
    return cluster_fits(kern, ctas, smem);
}

cudaError_t launch_steps_cluster(const SysDesc& d, int nsteps, int rel0, int G, int len, cudaStream_t st)
{
    if (!d.P.cblk) {  // no parts: whole sums, in the ranges of the step kernels (one for memories too short for blocks)
        len = 1;
        G = std::max(G, 1);
    }
    int ctas = 0;
    size_t smem = 0;
    const StepsKernel kern = steps_kernel(d.P, &ctas, &smem);
    return launch_cluster(kern, ctas, smem, st, d, nsteps, rel0, G, len);
}

bool rebuild_in_cluster(const StepParams& P)
{
    return P.n <= kClusterRebuildMaxN && P.maxnb <= 128 &&
           cluster_fits(rebuild_cluster, cluster_ctas(P.n, kRebLanes), rebuild_smem(P));
}

cudaError_t launch_rebuild_cluster(const StepParams& P, const ParticleBuffers& B, cudaStream_t st)
{
    return launch_cluster(rebuild_cluster, cluster_ctas(P.n, kRebLanes), rebuild_smem(P), st, P, B);
}

}  // namespace gld
