// near_direct.cuh -- the mixed path's leaf pairs summed directly, one thread
// per target: the sums of k_near_direct (p2p.cu) and of the smooth near
// field's small leaf pairs (smooth.cu).
#pragma once
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

// Source ranges of the neighbours in the 9-bit mask (bit (dy + 1) 3 + dx + 1)
// of leaf (ix, iy); the others empty.
__device__ __forceinline__ void near_ranges(uint32_t mask, const InstDesc &d,
                                            const uint32_t *__restrict__ st, int ix, int iy,
                                            uint32_t (&s0)[9], uint32_t (&s1)[9]) {
#pragma unroll
    for (int o = 0; o < 9; ++o) {
        s0[o] = s1[o] = 0;
        if ((mask >> o) & 1u) {
            const uint32_t nm = morton_key(uint32_t(ix + o % 3 - 1), uint32_t(iy + o / 3 - 1));
            s0[o] = st[nm];
            s1[o] = st[nm + 1];
            if (!(PF_IN(int64_t(s0[o]) - d.poff, d.n + 1) &&
                  PF_IN(int64_t(s1[o]) - d.poff, d.n + 1)))
                s1[o] = s0[o];
        }
    }
}

// kappa g(kappa rho^2) by the polynomial fitted on the host
template <int DEG>
__device__ __forceinline__ float near_poly(const float (&a)[DEG + 1], float r2, float kappa) {
    float g = a[DEG];
#pragma unroll
    for (int k = DEG - 1; k >= 0; --k) g = fmaf(g, r2, a[k]);
    return kappa * g;
}

// Four sources' factors gamma kappa g: GENERAL, most pairs of a narrow core lie
// beyond the polynomial and take (1 - e^-q) / rho^2, two special-function
// operations; the polynomial only where q is so small that the subtraction
// would lose the fit's tolerance (InstDesc::direct_rho2), behind one test for
// the four.
template <int DEG, bool GENERAL>
__device__ __forceinline__ void near_four(const float4 (&r)[4], float xt, float yt,
                                          const float (&a)[DEG + 1], float kappa, float split,
                                          float ek, float &u, float &v) {
    float dx[4], dy[4], r2[4], f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        dx[i] = xt - r[i].x;
        dy[i] = yt - r[i].y;
        r2[i] = fmaf(dx[i], dx[i], dy[i] * dy[i]);
        if (GENERAL) {
            f[i] = r[i].z * rcp_ftz(r2[i]);
            f[i] = fmaf(-ex2_ftz(ek * r2[i]), f[i], f[i]);
        } else {
            f[i] = r[i].z * near_poly<DEG>(a, r2[i], kappa);
        }
    }
    if (GENERAL && fminf(fminf(r2[0], r2[1]), fminf(r2[2], r2[3])) < split) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (r2[i] < split) f[i] = r[i].z * near_poly<DEG>(a, r2[i], kappa);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        u = fmaf(-dy[i], f[i], u);
        v = fmaf(dx[i], f[i], v);
    }
}

// Sum of gamma_j (-d_eta, d_xi) kappa g(kappa rho^2) over the ranges, target
// (x, y) in its leaf's frame.
template <int DEG, bool GENERAL>
__device__ __forceinline__ float2 near_vortex(const uint32_t (&s0)[9], const uint32_t (&s1)[9],
                                              const InstDesc &d, const float4 *__restrict__ rec,
                                              float x, float y) {
    float a[DEG + 1];
#pragma unroll
    for (int k = 0; k <= DEG; ++k) a[k] = d.poly[k];
    const float kappa = d.kappa, split = d.direct_rho2;
    const float ek = -1.44269504f * kappa;  // e^-q = 2^(ek rho^2)
    float u = 0.f, v = 0.f;
#pragma unroll
    for (int o = 0; o < 9; ++o) {
        const float xt = x - float(o % 3 - 1), yt = y - float(o / 3 - 1);
        const float4 *s = rec + s0[o];
        int n = int(s1[o] - s0[o]);
        float4 r[4];
        for (; n >= 4; n -= 4, s += 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = __ldg(s + i);
            near_four<DEG, GENERAL>(r, xt, yt, a, kappa, split, ek, u, v);
        }
        if (n > 0) {  // the rest: places past the end repeat the first, without strength
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                r[i] = __ldg(s + (i < n ? i : 0));
                if (i >= n) r[i].z = 0.f;
            }
            near_four<DEG, GENERAL>(r, xt, yt, a, kappa, split, ek, u, v);
        }
    }
    return make_float2(u, v);
}

// ... by the instance's degree and range
__device__ __forceinline__ float2 near_vortex_of(const uint32_t (&s0)[9], const uint32_t (&s1)[9],
                                                 const InstDesc &d, const float4 *__restrict__ rec,
                                                 float x, float y) {
    if (d.general)
        return d.deg <= 6 ? near_vortex<6, true>(s0, s1, d, rec, x, y)
                          : near_vortex<12, true>(s0, s1, d, rec, x, y);
    return d.deg <= 6 ? near_vortex<6, false>(s0, s1, d, rec, x, y)
                      : near_vortex<12, false>(s0, s1, d, rec, x, y);
}

// Laplace kernel: sum of q_j log r over the ranges (global units, logw the
// log of the leaf width), coincident pairs excluded: log r = ln 2 / 2 log2
// rho^2 + logw, the constant taken out of the sum.
__device__ __forceinline__ float near_laplace(const uint32_t (&s0)[9], const uint32_t (&s1)[9],
                                              const float4 *__restrict__ rec, float x, float y,
                                              float logw) {
    const float none = -2.88539008f * logw;  // log2 rho^2 that makes log r zero
    float s = 0.f, qs = 0.f;
#pragma unroll
    for (int o = 0; o < 9; ++o) {
        const float xt = x - float(o % 3 - 1), yt = y - float(o / 3 - 1);
#pragma unroll 4
        for (uint32_t j = s0[o]; j < s1[o]; ++j) {
            const float4 r = __ldg(rec + j);
            const float dx = xt - r.x, dy = yt - r.y;
            const float r2 = fmaf(dx, dx, dy * dy);
            const float l = r2 > 0.f ? lg2_ftz(r2) : none;
            s = fmaf(r.z, l, s);
            qs += r.z;
        }
    }
    return fmaf(0.34657359f, s, logw * qs);
}

}  // namespace petfmm
