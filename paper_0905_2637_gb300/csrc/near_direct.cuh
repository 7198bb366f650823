// near_direct.cuh -- the mixed path's leaf pairs summed directly, one thread
// per target: the sums of k_near_direct (p2p.cu) and of the smooth near
// field's small leaf pairs (smooth.cu).
#pragma once
#include <cfloat>

#include "common.cuh"

namespace petfmm {

__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_ftz(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_full(float x) {  // subnormal x too
    float y;
    asm("lg2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// kappa g(q) by the polynomial fitted on the host, in t = log2 e^-q
template <int DEG>
__device__ __forceinline__ float near_poly(const float (&a)[DEG + 1], float t) {
    float g = a[DEG];
#pragma unroll
    for (int k = DEG - 1; k >= 0; --k) g = fmaf(g, t, a[k]);
    return g;
}

// Four sources' factors gamma kappa g: GENERAL, most pairs of a narrow core lie
// beyond the polynomial and take (1 - e^-q) / rho^2, two special-function
// operations; below q = kDirectQ the subtraction loses more than the polynomial
// does, which takes over behind one test for the four.
template <int DEG, bool GENERAL>
__device__ __forceinline__ void near_four(const float4 (&r)[4], float xt, float yt,
                                          const float (&a)[DEG + 1], float split, float ek,
                                          float &u, float &v) {
    float dx[4], dy[4], r2[4], t[4], f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        dx[i] = xt - r[i].x;
        dy[i] = yt - r[i].y;
        r2[i] = fmaf(dx[i], dx[i], dy[i] * dy[i]);
        t[i] = ek * r2[i];
        if (GENERAL) {
            f[i] = r[i].z * rcp_ftz(r2[i]);
            f[i] = fmaf(-ex2_ftz(t[i]), f[i], f[i]);
        } else {
            f[i] = r[i].z * near_poly<DEG>(a, t[i]);
        }
    }
    if (GENERAL && fminf(fminf(r2[0], r2[1]), fminf(r2[2], r2[3])) < split) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (r2[i] < split) f[i] = r[i].z * near_poly<DEG>(a, t[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        u = fmaf(-dy[i], f[i], u);
        v = fmaf(dx[i], f[i], v);
    }
}

// Sources summed before the partial sum joins the total: a single running
// FP32 sum over the thousands of sources of dense leaves loses three times the
// accuracy (349,185 clustered blobs, 4,800 sources a target: 1.0e-6 against
// 3.7e-7 of the FP64 path).
constexpr int NEAR_RUN = 64;

// The leaves a target sums directly: the neighbours in the 9-bit mask (bit
// (dy + 1) 3 + dx + 1) of leaf (ix, iy) that lie in the domain and are not
// summed pairwise with it (n blobs; both of at least pmin).
struct NearLeaves {
    const InstDesc *d;
    const uint32_t *st;
    int ix, iy;
    uint32_t mask, n, pmin;
};

// Calls four(records, x, y) for the sources of those leaves, four at a time
// (places past a leaf's end repeat the first of the four, with no strength),
// x, y the target in the source leaf's frame, and next() after every leaf and
// NEAR_RUN sources.  Returns the number of sources in the mask's leaves.  One
// loop body for the nine leaves: unrolled it spilled registers and left the
// instruction cache.
template <typename F, typename G>
__device__ __forceinline__ uint32_t near_sources(const NearLeaves &q, const float4 *__restrict__ rec,
                                                 float x, float y, F &&four, G &&next) {
    const InstDesc &d = *q.d;
    const int nside = 1 << d.L;
    uint32_t total = 0;
#pragma unroll 1
    for (int o = 0; o < 9; ++o) {
        const int dy = o < 3 ? -1 : o < 6 ? 0 : 1, dx = o - 3 * dy - 4;
        const int lx = q.ix + dx, ly = q.iy + dy;
        if (!((q.mask >> o) & 1u) || lx < 0 || ly < 0 || lx >= nside || ly >= nside) continue;
        const uint32_t nm = morton_key(uint32_t(lx), uint32_t(ly));
        const uint32_t s0 = q.st[nm], s1 = q.st[nm + 1];
        if (!(PF_IN(int64_t(s0) - d.poff, d.n + 1) && PF_IN(int64_t(s1) - d.poff, d.n + 1)))
            continue;
        total += s1 - s0;
        if (q.n >= q.pmin && s1 - s0 >= q.pmin) continue;
        const float xt = x - float(dx), yt = y - float(dy);
        const float4 *s = rec + s0;
        int n = int(s1 - s0);
        float4 r[4];
        while (n > 0) {
            const int run = min(n, NEAR_RUN);
            const float4 *e = s + (run & ~3);
            for (; s < e; s += 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) r[i] = __ldg(s + i);
                four(r, xt, yt);
            }
            const int rest = run & 3;  // (only in the last run of a leaf)
            if (rest) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    r[i] = __ldg(s + (i < rest ? i : 0));
                    if (i >= rest) r[i].z = 0.f;
                }
                four(r, xt, yt);
            }
            n -= run;
            next();
        }
    }
    return total;
}

// Sum of gamma_j (-d_eta, d_xi) kappa g(kappa rho^2) over the leaves, target
// (x, y) in its leaf's frame.
template <int DEG, bool GENERAL>
__device__ __forceinline__ float2 near_vortex(const NearLeaves &q, const float4 *__restrict__ rec,
                                              float x, float y, uint32_t &total) {
    const InstDesc &d = *q.d;
    float a[DEG + 1];
#pragma unroll
    for (int k = 0; k <= DEG; ++k) a[k] = d.polyt[k];
    const float split = d.direct_rho2;
    const float ek = -1.44269504f * d.kappa;  // e^-q = 2^(ek rho^2)
    float u = 0.f, v = 0.f, pu = 0.f, pv = 0.f;
    total = near_sources(
        q, rec, x, y,
        [&](const float4(&r)[4], float xt, float yt) {
            near_four<DEG, GENERAL>(r, xt, yt, a, split, ek, pu, pv);
        },
        [&] {
            u += pu;
            v += pv;
            pu = pv = 0.f;
        });
    return make_float2(u, v);
}

// ... by the instance's degree and range
__device__ __forceinline__ float2 near_vortex_of(const NearLeaves &q, const float4 *__restrict__ rec,
                                                 float x, float y, uint32_t &total) {
    // (5: the degree of the default tolerance)
    if (q.d->general)
        return q.d->deg <= 5 ? near_vortex<5, true>(q, rec, x, y, total)
                             : near_vortex<12, true>(q, rec, x, y, total);
    return q.d->deg <= 6 ? near_vortex<6, false>(q, rec, x, y, total)
                         : near_vortex<12, false>(q, rec, x, y, total);
}

// Laplace kernel: sum of q_j log r over the leaves (global units, logw the
// log of the leaf width), coincident pairs excluded: log r = ln 2 / 2 log2
// rho^2 + logw, the constant taken out of the sum.  Pairs so close that rho^2
// is subnormal (the flushing logarithm would take them for coincident, log 0)
// stand apart with those, behind one test for the four; coincident ones have no
// strength there (a logarithm that cancels the constant leaves its rounding).
__device__ __forceinline__ float near_laplace(const NearLeaves &q, const float4 *__restrict__ rec,
                                              float x, float y, float logw, uint32_t &total) {
    float s = 0.f, qs = 0.f, ps = 0.f, pq = 0.f;
    total = near_sources(
        q, rec, x, y,
        [&](const float4(&r)[4], float xt, float yt) {
            float r2[4], l[4], z[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float dx = xt - r[i].x, dy = yt - r[i].y;
                r2[i] = fmaf(dx, dx, dy * dy);
                l[i] = lg2_ftz(r2[i]);
                z[i] = r[i].z;
            }
            if (fminf(fminf(r2[0], r2[1]), fminf(r2[2], r2[3])) < FLT_MIN) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (r2[i] < FLT_MIN) {
                        l[i] = r2[i] > 0.f ? lg2_full(r2[i]) : 0.f;
                        if (!(r2[i] > 0.f)) z[i] = 0.f;
                    }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ps = fmaf(z[i], l[i], ps);
                pq += z[i];
            }
        },
        [&] {
            s += ps;
            qs += pq;
            ps = pq = 0.f;
        });
    return fmaf(0.34657359f, s, logw * qs);
}

// sum_k c_k (x + i y)^k, k < p, FAR_CHUNK coefficients requested at a time:
// all threads of a leaf read the same ones, so the latency of the loads, not
// their number, is what a loop of dependent steps waits for.  (Final pass and
// scatters of 16.8M clustered blobs, p = 17: one chunk of 18 676 us, 9 688,
// 6 702, 4 719; an ordinary loop 715.)
constexpr int FAR_CHUNK = 9;
__device__ __forceinline__ float2 far_series(const float2 *__restrict__ c, int p, float x, float y) {
    float2 z = make_float2(0.f, 0.f);
    for (int k = (p - 1) / FAR_CHUNK * FAR_CHUNK; k >= 0; k -= FAR_CHUNK) {
        float2 ck[FAR_CHUNK];
#pragma unroll
        for (int i = 0; i < FAR_CHUNK; ++i)
            ck[i] = k + i < p ? __ldg(c + k + i) : make_float2(0.f, 0.f);
#pragma unroll
        for (int i = FAR_CHUNK - 1; i >= 0; --i)
            z = make_float2(fmaf(z.x, x, fmaf(-z.y, y, ck[i].x)),
                            fmaf(z.x, y, fmaf(z.y, x, ck[i].y)));
    }
    return z;
}

}  // namespace petfmm
