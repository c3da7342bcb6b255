// neighbours.cuh -- neighbour sums with L lanes per particle.
//
// One thread per particle walks its list four entries at a time; up to some
// 100000 particles that leaves the chip idle behind a chain of loads (8 to 12
// us per kernel whatever the size).  Here lane l of a round takes the E entries
// from l E on, so a list of up to L E entries costs one chain; every lane then
// adds the terms in list order (shuffles), the additions a single thread would
// make: the same bits.  A term outside the cutoff adds exactly nothing.
#pragma once

#include "gld_internal.cuh"

namespace gld {

// Loads of data that other CTAs write during the kernel (plain), and of data
// that is constant during it (read-only path).
struct LdPlain {
    static __device__ __forceinline__ float4 f4(const float4* p)
    {
        float4 v;
        asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ float f1(const float* p)
    {
        float v;
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ int i1(const int* p)
    {
        int v;
        asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
};
struct LdConst {
    static __device__ __forceinline__ float4 f4(const float4* p) { return __ldg(p); }
    static __device__ __forceinline__ float f1(const float* p) { return __ldg(p); }
    static __device__ __forceinline__ int i1(const int* p) { return __ldg(p); }
};

__device__ __forceinline__ float nb_dot3(float ax, float ay, float az, float bx, float by, float bz)
{
    return fmaf(ax, bx, fmaf(ay, by, az * bz));
}

// Lanes of one particle: lane in the group and the group's mask in the warp.
template <int L>
struct Lanes {
    int lane;
    unsigned mask;
    __device__ __forceinline__ Lanes()
    {
        lane = threadIdx.x & (L - 1);
        mask = (L == 32 ? 0xffffffffu : ((1u << L) - 1u)) << ((threadIdx.x & 31) & ~(L - 1));
    }
    __device__ __forceinline__ float get(float v, int l) const { return __shfl_sync(mask, v, l, L); }
};

// Walks the list nb[s * stride], s < *cnt, of particle i in rounds of L E
// entries: load(u, j) for the E entries of this lane (j = i past the list),
// then form(u, valid), then add(l, u) for the round's entries in list order.
// The first round's entries load beside the count (past the list they are
// stale ids, still valid indices); each next round's during the gathers.
template <class LD, int L, int E, class Load, class Form, class Add>
__device__ __forceinline__ void walk_list(const Lanes<L>& ln, const int* nb, const int* pcnt, int stride, int maxnb, int i,
                                          Load&& load, Form&& form, Add&& add)
{
    int jn[E];
#pragma unroll
    for (int u = 0; u < E; ++u) jn[u] = ln.lane * E + u < maxnb ? LD::i1(nb + (size_t)(ln.lane * E + u) * stride) : i;
    const int cnt = LD::i1(pcnt);
    for (int s = 0; s < cnt; s += L * E) {
        int j[E];
#pragma unroll
        for (int u = 0; u < E; ++u) j[u] = s + ln.lane * E + u < cnt ? jn[u] : i;
#pragma unroll
        for (int u = 0; u < E; ++u) load(u, j[u]);
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int e = s + L * E + ln.lane * E + u;
            jn[u] = e < cnt ? LD::i1(nb + (size_t)e * stride) : i;
        }
#pragma unroll
        for (int u = 0; u < E; ++u) form(u, j[u] != i);
        const int left = min(L, (cnt - s + E - 1) / E);
        for (int l = 0; l < left; ++l)
#pragma unroll
            for (int u = 0; u < E; ++u) add(l, u);
    }
}

// One separable pair term: F^D's instantaneous and history sums f0, fh (the
// one-term form of pair_force_integrate).
template <class LD, int L, int E>
__device__ __forceinline__ void pair_sums(const StepParams& P, const Lanes<L>& ln, const float4* pos, const float4* vel,
                                          const float* pj0, const int* nb, const int* pcnt, int i, const float4 pi,
                                          const float* __restrict__ ftab, float g00, float (&f0)[3], float (&fh)[3])
{
    const size_t np = P.n_pad;
    float4 pj[E], vj[E];
    float qx[E], qy[E], qz[E], inst[E], hist[E], ex[E], ey[E], ez[E];
    walk_list<LD, L, E>(
        ln, nb, pcnt, P.n_pad, P.maxnb, i,
        [&](int u, int j) {
            pj[u] = LD::f4(pos + j);
            vj[u] = LD::f4(vel + j);
            qx[u] = LD::f1(pj0 + j);
            qy[u] = LD::f1(pj0 + np + j);
            qz[u] = LD::f1(pj0 + 2 * np + j);
        },
        [&](int u, bool listed) {
            const float dx = min_image_fma(pi.x, pj[u].x, P.box, P.inv_box);
            const float dy = min_image_fma(pi.y, pj[u].y, P.box, P.inv_box);
            const float dz = min_image_fma(pi.z, pj[u].z, P.box, P.inv_box);
            const float r2 = dist2(dx, dy, dz);
            inst[u] = hist[u] = ex[u] = ey[u] = ez[u] = 0.f;
            if (!listed || !(r2 < P.rc2)) return;
            const float inv_r = rsqrtf(r2);  // listed pairs are distinct particles: r2 > 0
            const float r = r2 * inv_r;
            ex[u] = dx * inv_r;
            ey[u] = dy * inv_r;
            ez[u] = dz * inv_r;
            const float x = fmaxf(r, P.rc_min) * P.inv_dr;
            const float evj = nb_dot3(ex[u], ey[u], ez[u], vj[u].x, vj[u].y, vj[u].z);
            const float fq = table_at(ftab, P.nr, x);
            const float epj = nb_dot3(ex[u], ey[u], ez[u], qx[u], qy[u], qz[u]);
            inst[u] = fmaf(fq * g00, evj, 0.f);
            hist[u] = fmaf(fq, epj, 0.f);
        },
        [&](int l, int u) {
            const float in = ln.get(inst[u], l), hi = ln.get(hist[u], l);
            const float x = ln.get(ex[u], l), y = ln.get(ey[u], l), z = ln.get(ez[u], l);
            f0[0] = fmaf(-in, x, f0[0]); f0[1] = fmaf(-in, y, f0[1]); f0[2] = fmaf(-in, z, f0[2]);
            fh[0] = fmaf(-hi, x, fh[0]); fh[1] = fmaf(-hi, y, fh[1]); fh[2] = fmaf(-hi, z, fh[2]);
        });
}

// Any pair and self-difference terms, with perpendicular factors (the general
// form of pair_force_integrate); ps: the own history sums of the
// self-difference terms.
template <class LD, int L>
__device__ __forceinline__ void pair_sums_general(const StepParams& P, const Lanes<L>& ln, const float4* pos,
                                                  const float4* vel, const float* conv, const int* nb, const int* pcnt,
                                                  int i, const float4 pi, const float4 vi, const float (&ps)[kMaxQ][3],
                                                  const float* __restrict__ ftab, const float* __restrict__ fptab,
                                                  const float* __restrict__ g0, float (&f0)[3], float (&fh)[3])
{
    const size_t np = P.n_pad;
    float4 pj, vj;
    int jd = 0;
    float inst, hist, ex, ey, ez, ai[3], ah[3];  // ai, ah: the perpendicular parts' additions
    walk_list<LD, L, 1>(
        ln, nb, pcnt, P.n_pad, P.maxnb, i,
        [&](int, int j) {
            jd = j;
            pj = LD::f4(pos + j);
            vj = LD::f4(vel + j);
        },
        [&](int, bool listed) {
            const float dx = min_image_fma(pi.x, pj.x, P.box, P.inv_box);
            const float dy = min_image_fma(pi.y, pj.y, P.box, P.inv_box);
            const float dz = min_image_fma(pi.z, pj.z, P.box, P.inv_box);
            const float r2 = dist2(dx, dy, dz);
            inst = hist = ex = ey = ez = 0.f;
#pragma unroll
            for (int c = 0; c < 3; ++c) ai[c] = ah[c] = 0.f;
            if (!listed || !(r2 < P.rc2)) return;
            const float r = sqrtf(r2);
            const float inv_r = 1.0f / r;
            ex = dx * inv_r;
            ey = dy * inv_r;
            ez = dz * inv_r;
            const float x = fmaxf(r, P.rc_min) * P.inv_dr;
            const float evj = nb_dot3(ex, ey, ez, vj.x, vj.y, vj.z);
            const float evi = nb_dot3(ex, ey, ez, vi.x, vi.y, vi.z);
            for (int q = 0; q < P.Q; ++q) {
                const float fq = table_at(ftab + q * P.nr, P.nr, x);
                const float* p = conv + (size_t)(1 + q) * 3 * np + jd;
                const float epj = nb_dot3(ex, ey, ez, LD::f1(p), LD::f1(p + np), LD::f1(p + 2 * np));
                inst = fmaf(fq * __ldg(g0 + q), evj, inst);
                hist = fmaf(fq, epj, hist);
            }
            for (int q = 0; q < P.Qs; ++q) {
                const float fq = table_at(ftab + (P.Q + q) * P.nr, P.nr, x);
                const float epi = nb_dot3(ex, ey, ez, ps[q][0], ps[q][1], ps[q][2]);
                inst = fmaf(fq * __ldg(g0 + P.Q + q), evi, inst);
                hist = fmaf(fq, epi, hist);
            }
            if (P.perp) {
                // perpendicular parts act through 1 - e e^T: on X they give
                // fp (X - (e.X) e), X = V_j, P_j (pair) or V_i, P_i (self-difference)
                float cvj = 0.f, cvi = 0.f, hpe = 0.f, hpx = 0.f, hpy = 0.f, hpz = 0.f;
                for (int q = 0; q < P.Q; ++q) {
                    const float fp = table_at(fptab + q * P.nr, P.nr, x);
                    const float* p = conv + (size_t)(1 + q) * 3 * np + jd;
                    const float px = LD::f1(p), py = LD::f1(p + np), pz = LD::f1(p + 2 * np);
                    cvj = fmaf(fp, __ldg(g0 + q), cvj);
                    hpe = fmaf(fp, nb_dot3(ex, ey, ez, px, py, pz), hpe);
                    hpx = fmaf(fp, px, hpx); hpy = fmaf(fp, py, hpy); hpz = fmaf(fp, pz, hpz);
                }
                for (int q = 0; q < P.Qs; ++q) {
                    const float fp = table_at(fptab + (P.Q + q) * P.nr, P.nr, x);
                    cvi = fmaf(fp, __ldg(g0 + P.Q + q), cvi);
                    hpe = fmaf(fp, nb_dot3(ex, ey, ez, ps[q][0], ps[q][1], ps[q][2]), hpe);
                    hpx = fmaf(fp, ps[q][0], hpx); hpy = fmaf(fp, ps[q][1], hpy); hpz = fmaf(fp, ps[q][2], hpz);
                }
                const float ipe = fmaf(cvj, evj, cvi * evi);
                ai[0] = fmaf(ipe, ex, -fmaf(cvj, vj.x, cvi * vi.x));
                ai[1] = fmaf(ipe, ey, -fmaf(cvj, vj.y, cvi * vi.y));
                ai[2] = fmaf(ipe, ez, -fmaf(cvj, vj.z, cvi * vi.z));
                ah[0] = fmaf(hpe, ex, -hpx); ah[1] = fmaf(hpe, ey, -hpy); ah[2] = fmaf(hpe, ez, -hpz);
            }
        },
        [&](int l, int) {
            const float in = ln.get(inst, l), hi = ln.get(hist, l);
            const float x = ln.get(ex, l), y = ln.get(ey, l), z = ln.get(ez, l);
            f0[0] = fmaf(-in, x, f0[0]); f0[1] = fmaf(-in, y, f0[1]); f0[2] = fmaf(-in, z, f0[2]);
            fh[0] = fmaf(-hi, x, fh[0]); fh[1] = fmaf(-hi, y, fh[1]); fh[2] = fmaf(-hi, z, fh[2]);
            if (P.perp) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    f0[c] += ln.get(ai[c], l);
                    fh[c] += ln.get(ah[c], l);
                }
            }
        });
}

// F^C (soft repulsion or the table) as cforce sums it.
template <class LD, int L, int E>
__device__ __forceinline__ void cforce_sums(const StepParams& P, const Lanes<L>& ln, const float4* pos, const int* nb,
                                            const int* pcnt, int i, const float4 pi, const float* __restrict__ fctab,
                                            float (&f)[3])
{
    float4 pj[E];
    float sc[E], dx[E], dy[E], dz[E];
    walk_list<LD, L, E>(
        ln, nb, pcnt, P.n_pad, P.maxnb, i, [&](int u, int j) { pj[u] = LD::f4(pos + j); },
        [&](int u, bool listed) {
            dx[u] = min_image_fma(pi.x, pj[u].x, P.box, P.inv_box);
            dy[u] = min_image_fma(pi.y, pj[u].y, P.box, P.inv_box);
            dz[u] = min_image_fma(pi.z, pj[u].z, P.box, P.inv_box);
            const float r2 = dist2(dx[u], dy[u], dz[u]);
            if (listed && r2 < P.rc2) {
                const float inv_r = rsqrtf(r2);  // listed pairs are distinct particles: r2 > 0
                const float r = r2 * inv_r;
                sc[u] = (P.fc_nr > 0 ? table_at(fctab, P.fc_nr, r * P.fc_inv_dr) : P.fc_mag * (1.0f - r * P.inv_rc)) * inv_r;
            } else {
                sc[u] = dx[u] = dy[u] = dz[u] = 0.f;
            }
        },
        [&](int l, int u) {
            const float k = ln.get(sc[u], l);
            f[0] = fmaf(k, ln.get(dx[u], l), f[0]);
            f[1] = fmaf(k, ln.get(dy[u], l), f[1]);
            f[2] = fmaf(k, ln.get(dz[u], l), f[2]);
        });
}

}  // namespace gld
