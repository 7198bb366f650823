// fmm3d.cu -- the three-dimensional extension and its C ABI (petfmm3d_* in
// include/petfmm.h).  The paper names 3D as its first extension (Sec. 8):
// tree, work model and partition carry over, and the new part is a kernel
// with the 3D series and translation operators.  This file evaluates the
// Laplace potential and field of point charges,
//     phi_i = sum_{j != i} q_j / |x_i - x_j|,    E_i = -grad phi_i,
// by the FMM on a uniform octree: binning with three-coordinate z-order keys
// (Sec. 2.1, Sec. 5.1), the radix sort and gather of the 2D path, then P2M,
// M2M, M2L over the interaction list (at most 189 boxes), L2L, and a final
// per-leaf pass that sums the near field over the leaf and its up to 26
// neighbours and adds L2P (the steps of Sec. 2.2).
//
// Series (the paper gives none for 3D): solid harmonics of the 1/r kernel,
//   R_n^m(v) = r^n P_n^m(z/r) e^{i m phi} / (n + m)!,
//   I_n^m(v) = (n - m)! P_n^m(z/r) e^{i m phi} / r^(n+1),
// P_n^m without the Condon-Shortley phase and X_n^-m = (-1)^m conj(X_n^m),
// from the Legendre recurrences in Cartesian form (rec_r / rec_i below).
// They obey 1/|x - y| = sum conj(R_n^m(y)) I_n^m(x), R(a + b) = sum
// R_k^l(a) R_{n-k}^{m-l}(b) and I_n^m(a + b) = sum (-1)^k conj(R_k^l(b))
// I_{n+k}^{m+l}(a), so that with M_n^m = sum q conj(R_n^m(y - c)) and
// phi = sum L_n^m conj(R_n^m(x - c)) the translations are plain sums:
//   M2M  M'_n^m = sum conj(R_k^l(c - c')) M_{n-k}^{m-l}
//   M2L  L_k^l  = (-1)^k sum M_n^m I_{n+k}^{m+l}(c_t - c_s)
//   L2L  L'_j^s = sum L_{j+k}^{s+l} conj(R_k^l(c' - c)).
// Expansions are rescaled by the box width w (M~ = M / w^n, L~ = L w^(n+1)):
// every operator is then level independent -- M2L one table of
// I_j^s(delta) per integer offset delta between same-level boxes, M2M and
// L2L one table of R_k^l(e) per child octant e = (+-1/4, +-1/4, +-1/4), with
// the level change a power of two -- and FP32 stays in range for p <= 16.
// Only m >= 0 is stored (p (p + 1) / 2 complex per box, index n (n + 1) / 2
// + m); m < 0 follows from the symmetry of a real potential.
//
// HBM layout: uint32 key / value ping-pong pairs of the radix sort (3L-bit
// keys), 8^L + 1 leaf starts, the sorted particles (FP64 path: SoA x, y, z, q
// in double; mixed path: float4 (xi, eta, zeta, q), the position relative to
// the leaf centre in leaf widths), ME and LE of every level (8^l boxes in
// Morton order, level l at box offset (8^l - 1) / 7), the operator tables, and
// the parts of the near field: one entry per charge of the one-sided sums (16
// bytes, FP64 32) and planes of one entry per charge of the pairwise ones (mixed
// 416, FP64 864 bytes a charge; without room for them, or above
// PETFMM3D_OPT_PAIR_BYTES, every leaf pair is summed one-sided).
// Every sum runs in a fixed order: results are bitwise reproducible, as long as
// the planes are had or not had alike.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/petfmm.h"
#include "kernels.cuh"
#include "tcgen05.cuh"

namespace petfmm {
PF_DEFINE_CHECK_READER(fmm3d)
}
using namespace petfmm;

namespace {

constexpr int P3_MAX = PETFMM3D_MAX_P;           // terms
constexpr int L3_MAX = PETFMM3D_MAX_L;           // levels (3L <= 30 key bits)
constexpr int TC3_MAXP = 8;                        // terms of the tensor-core M2L
constexpr int NSLOT3 = 343;                        // offsets in [-3, 3]^3
constexpr int W3 = 8;                              // warps per block

template <typename T> struct C3;
template <> struct C3<float> { using V = float2; };
template <> struct C3<double> { using V = double2; };

template <typename V, typename T>
__host__ __device__ __forceinline__ V mk(T a, T b) { V v; v.x = a; v.y = b; return v; }

// a sorted particle of the FP64 path: x, y, z, q (32 bytes, one load)
struct __align__(32) Dbl4 {
    double x, y, z, w;
};

__host__ __device__ __forceinline__ int nc3(int p) { return p * (p + 1) / 2; }
// I_j^s, j < 2p - 1, s >= 0
__host__ __device__ __forceinline__ int nci3(int p) { return (2 * p - 1) * (2 * p) / 2; }
__host__ __device__ __forceinline__ int64_t lvl_off3(int l) {
    return ((int64_t(1) << (3 * l)) - 1) / 7;
}

// 3D z-order: bit b of ix, iy, iz to bits 3b, 3b + 1, 3b + 2 (10 bits each)
__host__ __device__ __forceinline__ uint32_t spread3(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
__host__ __device__ __forceinline__ uint32_t compact3(uint32_t v) {
    v &= 0x09249249u;
    v = (v ^ (v >> 2)) & 0x030c30c3u;
    v = (v ^ (v >> 4)) & 0x0300f00fu;
    v = (v ^ (v >> 8)) & 0x030000ffu;
    v = (v ^ (v >> 16)) & 0x000003ffu;
    return v;
}
__host__ __device__ __forceinline__ uint32_t morton3(uint32_t ix, uint32_t iy, uint32_t iz) {
    return spread3(ix) | (spread3(iy) << 1) | (spread3(iz) << 2);
}

// particles in box b of level l (from the leaf starts)
__device__ __forceinline__ uint32_t box_count3(const uint32_t *start, int L, int l, uint32_t b) {
    const int sh = 3 * (L - l);
    return start[(uint64_t(b) + 1) << sh] - start[uint64_t(b) << sh];
}

// ---------------------------------------------------------------------------
// Binning (Sec. 2.1 in 3D): t = x - x0; s = t 2^L / W; floor, clamped; FP64
// with round-to-nearest intrinsics (no contraction), through an FP32
// shortcut with the same result.  recu (mixed path): the record (xi, eta,
// zeta, q) in input order, each coordinate rounded to FP32 and held below
// 0.5 - 2^-24.  The cap moves a point by at most one FP32
// rounding and keeps two particles of adjacent leaves apart by at least
// 2^-24 leaf widths along the axis they differ in, so |d| = 0 in the near
// field can only come from the target's own leaf.
// ---------------------------------------------------------------------------
constexpr float REC_MAX = 0.5f - 0x1p-24f;

struct Dom3 {
    double x0, y0, z0, width, scale;  // scale = 2^L / width
    // float-float copies (x0 = x0h + x0l, ..., scale = sh + sl) for the FP32
    // binning shortcut and the records
    float x0h, x0l, y0h, y0l, z0h, z0l, sh, sl;
};

__device__ __forceinline__ uint32_t bin3(double v, double v0, double scale, uint32_t nb) {
    const double f = floor(__dmul_rn(__dsub_rn(v, v0), scale));
    if (!(f >= 0.0)) return 0u;
    if (f > double(nb - 1)) return nb - 1;
    return uint32_t(f);
}

// FP32 shortcut of bin3 (FP64 arithmetic is slow here), bit-identical: with
// xf, x0f, scalef the FP32 roundings of v, v0, scale, s32 = fl(fl(xf - x0f)
// scalef) is within 4 u scale (|v| + |v0|) (u = 2^-24, plus O(u^2)) of the
// FP64 s, and m = 2^-21 scale (|v| + |v0|) covers that and the roundings of
// s32 -/+ m.  Both ends of [s32 - m, s32 + m] in one bin inside
// (0, nb (1 - 2^-20)) put s in that bin, unclamped, and v inside the domain
// (s > 0: v > v0; s < nb (1 - 2^-20): v <= fl(v0 + W) while |v0 + W| <=
// 2^32 W, and a domain farther out makes m > nb, failing the test);
// otherwise (a bin edge, the boundary, NaN, Inf) false: the FP64 path.
__device__ __forceinline__ bool bin3_fast(float xf, float x0f, float scalef, uint32_t nb,
                                          uint32_t *bin) {
    const float sv = __fmul_rn(__fsub_rn(xf, x0f), scalef);
    const float m = __fmul_rn(__fmul_rn(__fadd_rn(fabsf(xf), fabsf(x0f)), scalef), 0x1p-21f);
    const float lo = __fsub_rn(sv, m), hi = __fadd_rn(sv, m);
    if (!(lo > 0.0f && hi < float(nb) * (1.0f - 0x1p-20f))) return false;
    const float f = floorf(lo);
    if (f != floorf(hi)) return false;
    *bin = uint32_t(f);
    return true;
}

// The record coordinate (v - v0) scale - (i + 1/2) in float-float
// arithmetic (two-sum for the difference, FMA for the product's error
// terms): before its final rounding within about 2^-44 of the exact value,
// relative to (v - v0) scale.
__device__ __forceinline__ void ff_split(float v, float *h, float *l) { *h = v; *l = 0.f; }
__device__ __forceinline__ void ff_split(double v, float *h, float *l) {
    *h = float(v);
    *l = float(v - double(*h));
}
template <typename TIn>
__device__ __forceinline__ float rec3_coord(TIn v, float v0h, float v0l, float sh, float sl,
                                            uint32_t i) {
    float vh, vl;
    ff_split(v, &vh, &vl);
    const float th = __fsub_rn(vh, v0h);
    const float bv = __fsub_rn(th, vh);
    float tl = __fadd_rn(__fsub_rn(vh, __fsub_rn(th, bv)), __fsub_rn(-v0h, bv));
    tl = __fadd_rn(tl, __fsub_rn(vl, v0l));
    const float ph = __fmul_rn(th, sh);
    float pe = __fmaf_rn(th, sh, -ph);
    pe = __fmaf_rn(th, sl, __fmaf_rn(tl, sh, pe));
    return __fadd_rn(__fsub_rn(ph, __fadd_rn(float(i), 0.5f)), pe);
}

template <typename TIn>
__global__ void __launch_bounds__(256) k3_bin(int64_t n, const TIn *__restrict__ x,
                                              const TIn *__restrict__ y, const TIn *__restrict__ z,
                                              const TIn *__restrict__ q, Dom3 d, int L,
                                              uint32_t *__restrict__ keys,
                                              float4 *__restrict__ recu, int *status) {
    const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const TIn xv = x[j], yv = y[j], zv = z[j];
    const uint32_t nb = 1u << L;
    uint32_t ix, iy, iz;
    if (!(bin3_fast(float(xv), d.x0h, d.sh, nb, &ix) && bin3_fast(float(yv), d.y0h, d.sh, nb, &iy) &&
          bin3_fast(float(zv), d.z0h, d.sh, nb, &iz))) {
        const double X = double(xv), Y = double(yv), Z = double(zv);
        const double x1 = __dadd_rn(d.x0, d.width), y1 = __dadd_rn(d.y0, d.width),
                     z1 = __dadd_rn(d.z0, d.width);
        if (!(X >= d.x0 && X <= x1 && Y >= d.y0 && Y <= y1 && Z >= d.z0 && Z <= z1))
            set_status(status, ST_EDOMAIN);
        ix = bin3(X, d.x0, d.scale, nb);
        iy = bin3(Y, d.y0, d.scale, nb);
        iz = bin3(Z, d.z0, d.scale, nb);
    }
    keys[j] = morton3(ix, iy, iz);
    if (recu) {
        float4 r;
        r.x = fminf(rec3_coord(xv, d.x0h, d.x0l, d.sh, d.sl, ix), REC_MAX);
        r.y = fminf(rec3_coord(yv, d.y0h, d.y0l, d.sh, d.sl, iy), REC_MAX);
        r.z = fminf(rec3_coord(zv, d.z0h, d.z0l, d.sh, d.sl, iz), REC_MAX);
        r.w = float(q[j]);
        recu[j] = r;
    }
}

// start[b] = first sorted rank with key >= b, b = 0..8^L
__global__ void __launch_bounds__(256) k3_leaf_start(const uint32_t *__restrict__ skeys, int64_t n,
                                                     int64_t nleaf, uint32_t *__restrict__ start) {
    const int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (b > nleaf) return;
    int64_t lo = 0, hi = n;
    if (b == nleaf) {
        lo = n;
    } else {
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (int64_t(skeys[mid]) < b) lo = mid + 1; else hi = mid;
        }
    }
    start[b] = uint32_t(lo);
}

template <typename TIn>
__global__ void __launch_bounds__(256) k3_gather_f64(int64_t n, const uint32_t *__restrict__ perm,
                                                     const TIn *__restrict__ x,
                                                     const TIn *__restrict__ y,
                                                     const TIn *__restrict__ z,
                                                     const TIn *__restrict__ q,
                                                     Dbl4 *__restrict__ out) {
    const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const uint32_t i = perm[r];
    if (!PF_IN(i, n)) return;
    out[r] = Dbl4{double(x[i]), double(y[i]), double(z[i]), double(q[i])};
}

// A particle of the leaf as (position relative to the leaf centre in leaf
// widths, charge).
template <typename T> struct Part3 { T x, y, z, q; };
__device__ __forceinline__ Part3<float> leaf_part(const float4 *rec, int64_t j, double, double,
                                                  double, double) {
    const float4 r = rec[j];
    return {r.x, r.y, r.z, r.w};
}
__device__ __forceinline__ Part3<double> leaf_part(const Dbl4 *xs, int64_t j, double cx,
                                                   double cy, double cz, double inv_w) {
    const Dbl4 r = xs[j];
    return {(r.x - cx) * inv_w, (r.y - cy) * inv_w, (r.z - cz) * inv_w, r.w};
}

// ---------------------------------------------------------------------------
// P2M (leaves): M~_n^m = sum_j q_j conj(R_n^m(xi_j)).  A warp per leaf split
// into 32 / p lane groups; lane m of a group owns column m: R_m^m = (xi + i
// eta)^m / (2^m m!), then the recurrence in n (its reciprocals computed once
// per lane), for every G-th particle of the leaf; the groups' sums are added
// in group order.
// ---------------------------------------------------------------------------
template <typename T, typename P>
__global__ void __launch_bounds__(W3 * 32) k3_p2m(int L, int p, Dom3 d, const uint32_t *__restrict__ start,
                                                  const P *__restrict__ part,
                                                  typename C3<T>::V *__restrict__ me) {
    using V = typename C3<T>::V;
    const int lane = threadIdx.x & 31;
    const int64_t b = int64_t(blockIdx.x) * W3 + (threadIdx.x >> 5);
    if (b >= (int64_t(1) << (3 * L))) return;
    const uint32_t s0 = start[b], s1 = start[b + 1];
    if (s0 == s1) return;
    // G = 32 / p lane groups, group g summing particles g, g + G, ...; lane
    // m of a group owns column m
    const int G = 32 / p, g = lane / p, m = lane - g * p;
    const double w = d.width / double(1u << L);
    const double cx = d.x0 + (double(compact3(uint32_t(b))) + 0.5) * w;
    const double cy = d.y0 + (double(compact3(uint32_t(b) >> 1)) + 0.5) * w;
    const double cz = d.z0 + (double(compact3(uint32_t(b) >> 2)) + 0.5) * w;
    V acc[P3_MAX];
    // the lane's constants, out of the particle loop: 1 / (2^m m!) and
    // 1 / (n^2 - m^2) of the recurrence
    T cm = T(1), inv[P3_MAX];
    for (int t = 1; t <= m; ++t) cm /= T(2 * t);
#pragma unroll
    for (int n = 0; n < P3_MAX; ++n) {
        acc[n] = mk<V>(T(0), T(0));
        inv[n] = n > m && n < p ? T(1) / T(n * n - m * m) : T(0);
    }
    // the leaf's records staged 64 at a time in shared memory by coalesced
    // loads, so that no particle's load waits in the groups' loops
    __shared__ P stage[W3][64];
    const int wid = threadIdx.x >> 5;
    for (uint32_t c0 = s0; c0 < s1; c0 += 64u) {
        const uint32_t cn = min(64u, s1 - c0);
        __syncwarp();
        for (uint32_t i = uint32_t(lane); i < cn; i += 32u) stage[wid][i] = part[c0 + i];
        __syncwarp();
        if (g >= G) continue;
        for (uint32_t j = uint32_t(g); j < cn; j += uint32_t(G)) {
            const Part3<T> a = leaf_part(stage[wid], j, cx, cy, cz, 1.0 / w);
            const T r2 = a.x * a.x + a.y * a.y + a.z * a.z;
            V zm = mk<V>(T(1), T(0));  // (xi + i eta)^m
            for (int t = 1; t <= m; ++t) zm = mk<V>(zm.x * a.x - zm.y * a.y, zm.x * a.y + zm.y * a.x);
            const T qc = a.q * cm;
            V r1 = mk<V>(zm.x * qc, zm.y * qc), r2v = mk<V>(T(0), T(0));  // q R_m^m
#pragma unroll
            for (int n = 0; n < P3_MAX; ++n) {
                if (n < m || n >= p) continue;
                V rn = r1;
                if (n > m) {
                    const T c1 = T(2 * n - 1) * a.z;
                    rn = mk<V>((c1 * r1.x - r2 * r2v.x) * inv[n], (c1 * r1.y - r2 * r2v.y) * inv[n]);
                    r2v = r1;
                    r1 = rn;
                }
                acc[n].x += rn.x;  // q conj(R) summed: conj taken at the end
                acc[n].y += rn.y;
            }
        }
    }
    // the groups' partial sums added into group 0 in group order (every lane
    // takes part in the shuffles)
#pragma unroll
    for (int n = 0; n < P3_MAX; ++n) {
        for (int gg = 1; gg < G; ++gg) {
            const int src = m + gg * p;
            const T ox = __shfl_sync(0xffffffffu, acc[n].x, src);
            const T oy = __shfl_sync(0xffffffffu, acc[n].y, src);
            if (g == 0) {
                acc[n].x += ox;
                acc[n].y += oy;
            }
        }
    }
    if (g == 0) {
        V *dst = me + (lvl_off3(L) + b) * nc3(p);
#pragma unroll
        for (int n = 0; n < P3_MAX; ++n)
            if (n >= m && n < p) dst[n * (n + 1) / 2 + m] = mk<V>(acc[n].x, -acc[n].y);
    }
}

// P2M for p <= 8: a warp per leaf with a lane per charge
// (charges j, j + 32, ... of the leaf), each lane computing all p (p + 1) / 2
// terms q R_n^m column by column with compile-time constants and summing
// them over its charges; then a reduce-scatter across the warp (three
// halving exchanges, offsets 16, 8, 4, then a butterfly over offsets 2 and
// 1) leaves each group of four lanes the full sums of a ninth of the 2 NC
// values, which one lane of the group writes.
// FP64: bound by its pipe; 262,144 charges, 64 a leaf, p = 8: 622 us by columns
// (k3_p2m, few lanes of a group busy in the short columns) -> 235 us.
template <int P, typename T, typename Rec>
__global__ void __launch_bounds__(W3 * 32) k3_p2m_lanes(int L, Dom3 d,
                                                        const uint32_t *__restrict__ start,
                                                        const Rec *__restrict__ rec,
                                                        typename C3<T>::V *__restrict__ me) {
    constexpr int NC = P * (P + 1) / 2, NV = 2 * NC;  // values: Re of all, then Im of all
    constexpr int NV8 = (NV + 7) / 8, NVP = 8 * NV8;  // padded to eight equal parts
    const int lane = threadIdx.x & 31;
    const int64_t b = int64_t(blockIdx.x) * W3 + (threadIdx.x >> 5);
    if (b >= (int64_t(1) << (3 * L))) return;
    const uint32_t s0 = start[b], s1 = start[b + 1];
    if (s0 == s1) return;
    const double w = d.width / double(1u << L), inv_w = 1.0 / w;
    const double cx = d.x0 + (double(compact3(uint32_t(b))) + 0.5) * w;
    const double cy = d.y0 + (double(compact3(uint32_t(b) >> 1)) + 0.5) * w;
    const double cz = d.z0 + (double(compact3(uint32_t(b) >> 2)) + 0.5) * w;
    T v[NVP];
#pragma unroll
    for (int k = 0; k < NVP; ++k) v[k] = T(0);
    for (uint32_t j = s0 + uint32_t(lane); j < s1; j += 32u) {
        const Part3<T> a = leaf_part(rec, j, cx, cy, cz, inv_w);
        const T r2 = a.x * a.x + a.y * a.y + a.z * a.z;
        T pr = a.q, pi = T(0);  // q R_m^m
#pragma unroll
        for (int m = 0; m < P; ++m) {
            if (m > 0) {
                const T sc = T(1) / T(2 * m);
                const T tr = (pr * a.x - pi * a.y) * sc, ti = (pr * a.y + pi * a.x) * sc;
                pr = tr;
                pi = ti;
            }
            T r1r = pr, r1i = pi, r0r = T(0), r0i = T(0);
            v[m * (m + 1) / 2 + m] += r1r;
            v[NC + m * (m + 1) / 2 + m] += r1i;
#pragma unroll
            for (int n = m + 1; n < P; ++n) {
                const T c1 = T(2 * n - 1) * a.z;
                const T inv = T(1) / T(n * n - m * m);
                const T rr = (c1 * r1r - r2 * r0r) * inv, ri = (c1 * r1i - r2 * r0i) * inv;
                r0r = r1r;
                r0i = r1i;
                r1r = rr;
                r1i = ri;
                v[n * (n + 1) / 2 + m] += rr;
                v[NC + n * (n + 1) / 2 + m] += ri;
            }
        }
    }
    // halving exchanges: at offset o the lane keeps the lower half of its
    // values if (lane & o) == 0, else the upper half, adding the partner's
    // copy of the half it keeps
#pragma unroll
    for (int k = 0; k < NVP / 2; ++k) {
        const bool up = lane & 16;
        const T send = up ? v[k] : v[k + NVP / 2];
        const T keep = up ? v[k + NVP / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int k = 0; k < NVP / 4; ++k) {
        const bool up = lane & 8;
        const T send = up ? v[k] : v[k + NVP / 4];
        const T keep = up ? v[k + NVP / 4] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int k = 0; k < NV8; ++k) {
        const bool up = lane & 4;
        const T send = up ? v[k] : v[k + NV8];
        const T keep = up ? v[k + NV8] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
#pragma unroll
    for (int k = 0; k < NV8; ++k) {
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 2);
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1);
    }
    // this group's values: index 4 NVP/8 bit4 + 2 NVP/8 bit3 + NVP/8 bit2 + k
    if ((lane & 3) == 0) {
        const int base = NV8 * (4 * ((lane >> 4) & 1) + 2 * ((lane >> 3) & 1) + ((lane >> 2) & 1));
        T *dst = reinterpret_cast<T *>(me + (lvl_off3(L) + b) * NC);
#pragma unroll
        for (int k = 0; k < NV8; ++k) {
            const int vi = base + k;
            if (vi < NC)
                dst[2 * vi] = v[k];
            else if (vi < NV)
                dst[2 * (vi - NC) + 1] = -v[k];  // conj
        }
    }
}

template <typename T, typename Rec>
cudaError_t launch_p2m_lanes(int p, int L, const Dom3 &d, const uint32_t *start, const Rec *rec,
                             typename C3<T>::V *me, cudaStream_t st) {
    const unsigned grid = unsigned(((int64_t(1) << (3 * L)) + W3 - 1) / W3);
    switch (p) {
#define PL_CASE(P) \
    case P: k3_p2m_lanes<P, T><<<grid, W3 * 32, 0, st>>>(L, d, start, rec, me); break;
        PL_CASE(1) PL_CASE(2) PL_CASE(3) PL_CASE(4) PL_CASE(5) PL_CASE(6) PL_CASE(7) PL_CASE(8)
#undef PL_CASE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// M2L by reflection orbits (all levels in one launch): the FP64 path, and the
// mixed path's small trees.  The coefficients of a
// real potential with degrees < p are p^2 real numbers (host_m2l_real); in
// that basis a reflection of an axis is a diagonal of signs, so the operator
// of delta = (+-a, +-b, +-c) is S T S with the one of (a, b, c) and S the
// signs of the reflected axes.  The up to eight sources of an orbit are
// therefore added first, with signs, and translated by one product:
//   c_r += sum_k T[k][r] H[q(r) ^ q(k)][k],
//   H[q][k] = sum_s (-1)^popc(q & s) a_s[k]
// (q: a coefficient's parity along x, y, z; s: the reflected axes), 56 real
// p^2 x p^2 products for the up to 189 boxes of the interaction list and
// three butterfly stages for H.  FP64 is bound by its pipe (two lanes a cycle
// and SM on this part), so the work is laid out to leave no lane idle: a
// group of threads takes (target box, coefficient) pairs flat, NI each, and
// GROUPS groups of a block every GROUPS-th orbit, their sums added at the end
// in group order; operators come through L1, H from shared memory.
// Measured (one GB300, 262,144 uniform charges, L = 4, p = 8, FP64): 76.6 ms
// with a warp per target box and the complex sums of every source -> 2.3 ms;
// the FP32 sides are at use_orbits3 and launch_m2l_orbits.
// ---------------------------------------------------------------------------
constexpr int ORB_THREADS = 256;

// the offsets (|dx| + 4 |dy| + 16 |dz|) of the interaction list
struct Orbits3 {
    uint8_t o[56];
};
constexpr Orbits3 orbits3() {
    Orbits3 r{};
    for (int o = 1, n = 0; o < 64; ++o)
        if ((o & 3) >= 2 || ((o >> 2) & 3) >= 2 || (o >> 4) >= 2) r.o[n++] = uint8_t(o);
    return r;
}
__constant__ Orbits3 c_orbits = orbits3();

// targets of a block, from the (target, coefficient) pairs of a group
__host__ __device__ constexpr int orb_items(int ni, int groups) { return ORB_THREADS / groups * ni; }
__host__ __device__ constexpr int orb_rows(int items, int p) { return items / (p * p); }
// blocks of level l: ceil(8^(l-1) / rows) x 8 child classes
__host__ __device__ __forceinline__ int64_t orb_blocks(int l, int rows) {
    return ((int64_t(1) << (3 * (l - 1))) + rows - 1) / rows * 8;
}
// values between the H of two parity classes (two of padding keep the eight
// classes on different banks)
__host__ __device__ constexpr int orb_stride(int rows, int p) { return rows * p * p + 2; }

template <typename T, int NI, int GROUPS>
__global__ void __launch_bounds__(ORB_THREADS) k3_m2l_orbits(
    int L, int p, const uint32_t *__restrict__ start, const T *__restrict__ atab,
    const short2 *__restrict__ rmap, const uint8_t *__restrict__ parity,
    const typename C3<T>::V *__restrict__ me, typename C3<T>::V *__restrict__ le) {
    constexpr int GT = ORB_THREADS / GROUPS;  // threads of a group
    extern __shared__ __align__(16) unsigned char orb_smem[];
    __shared__ uint8_t sq[P3_MAX * P3_MAX];    // parity class of each real index
    __shared__ uint16_t soff[P3_MAX * P3_MAX]; // its place in a box's stored doubles
    const int g = int(threadIdx.x) / GT, tid = int(threadIdx.x) % GT;
    const int nr = p * p, nc = nc3(p);
    const int rows = orb_rows(orb_items(NI, GROUPS), p), qs = orb_stride(rows, p);
    T *const hall = reinterpret_cast<T *>(orb_smem), *const hs = hall + g * 8 * qs;
    // source box of (target, member), -1: none
    int *const srow = reinterpret_cast<int *>(hall + GROUPS * 8 * qs) + g * 8 * rows;
    int l = 2;
    int64_t bid = blockIdx.x;
    while (l < L && bid >= orb_blocks(l, rows)) bid -= orb_blocks(l++, rows);
    const int c = int(bid & 7);
    const int64_t np = int64_t(1) << (3 * (l - 1)), p0 = (bid >> 3) * rows;
    const int side = 1 << l;
    bool mine = false;
    for (int t = tid; t < rows; t += GT)
        if (p0 + t < np) mine |= box_count3(start, L, l, uint32_t((p0 + t) * 8 + c)) != 0;
    if (!__syncthreads_or(mine)) return;  // no target holds particles
    for (int r = threadIdx.x; r < nr; r += ORB_THREADS) {
        sq[r] = parity[r];
        const short2 mp = rmap[r];
        soff[r] = uint16_t(2 * mp.x + (mp.y == 1));
    }
    // this thread's (target, coefficient) pairs
    int it_r[NI], it_t[NI], it_q[NI];
    T acc[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int e = tid + i * GT;
        const bool in = e < rows * nr;
        it_t[i] = in ? e / nr : 0;
        it_r[i] = in ? e % nr : 0;
        it_q[i] = parity[it_r[i]];
        acc[i] = T(0);
    }
    const T *lev = reinterpret_cast<const T *>(me + lvl_off3(l) * nc);
    static_assert(56 % GROUPS == 0, "orbits per group");
    for (int step = g; step < 56; step += GROUPS) {
        const int o = c_orbits.o[step];
        const int a[3] = {o & 3, (o >> 2) & 3, o >> 4};
        // axis d: both signs of the offset, or one (0; 3 reaches out of the
        // parent's neighbours on one side); delta = target - source
        bool both[3], neg[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            both[d] = a[d] == 1 || a[d] == 2;
            neg[d] = a[d] == 3 && !((c >> d) & 1);
        }
        __syncthreads();  // the previous orbit's products are done
        bool have = false;
        for (int e = tid; e < 8 * rows; e += GT) {
            const int s = e & 7, t = e >> 3;
            int src = -1;
            bool member = p0 + t < np;
            int x[3];
            const uint32_t tb = uint32_t((p0 + t) * 8 + c);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const bool up = (s >> d) & 1;  // reflected
                member = member && (both[d] || !up);
                x[d] = int(compact3(tb >> d)) + (up || neg[d] ? a[d] : -a[d]);
                member = member && x[d] >= 0 && x[d] < side;
            }
            if (member) {
                const uint32_t sb = morton3(uint32_t(x[0]), uint32_t(x[1]), uint32_t(x[2]));
                if (box_count3(start, L, l, sb)) src = int(sb);
            }
            srow[e] = src;
            have |= src >= 0;
        }
        if (!__syncthreads_or(have)) continue;
        for (int e = tid; e < rows * nr; e += GT) {
            const int t = e / nr, k = e - t * nr;
            T v[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const int sb = srow[8 * t + s];
                v[s] = sb >= 0 && PF_IN(sb, int64_t(1) << (3 * l)) ? lev[int64_t(sb) * (2 * nc) + soff[k]]
                                                                    : T(0);
            }
            // butterflies along the axes with both signs (entries reflected
            // along another axis are not there yet), then copies
#pragma unroll
            for (int d = 0; d < 3; ++d)
                if (both[d])
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        if ((s >> d) & 1) continue;
                        bool there = true;
#pragma unroll
                        for (int f = 0; f < 3; ++f) there = there && (both[f] || !((s >> f) & 1));
                        if (!there) continue;
                        const T x = v[s], y = v[s | (1 << d)];
                        v[s] = x + y;
                        v[s | (1 << d)] = x - y;
                    }
#pragma unroll
            for (int d = 0; d < 3; ++d)
                if (!both[d])
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (!((s >> d) & 1)) v[s | (1 << d)] = neg[d] ? -v[s] : v[s];
#pragma unroll
            for (int s = 0; s < 8; ++s) hs[s * qs + e] = v[s];
        }
        __syncthreads();
        const T *at = atab + size_t(o) * nr * nr;
#pragma unroll 4
        for (int k = 0; k < nr; ++k) {
            const int qk = sq[k];
#pragma unroll
            for (int i = 0; i < NI; ++i)
                acc[i] = fma(__ldg(at + size_t(k) * nr + it_r[i]),
                             hs[(it_q[i] ^ qk) * qs + it_t[i] * nr + k], acc[i]);
        }
    }
    if (GROUPS > 1) {
        __syncthreads();
        if (g)
#pragma unroll
            for (int i = 0; i < NI; ++i) hall[((g - 1) * NI + i) * GT + tid] = acc[i];
        __syncthreads();
        if (g) return;
        for (int k = 0; k + 1 < GROUPS; ++k)
#pragma unroll
            for (int i = 0; i < NI; ++i) acc[i] += hall[(k * NI + i) * GT + tid];
    }
    T *lef = reinterpret_cast<T *>(le + lvl_off3(l) * nc);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        if (tid + i * GT >= rows * nr || p0 + it_t[i] >= np) continue;
        const short2 mp = rmap[it_r[i]];
        T *dst = lef + ((p0 + it_t[i]) * 8 + c) * (2 * nc) + 2 * mp.x;
        dst[mp.y == 1] = acc[i];
        if (mp.y == 2) dst[1] = T(0);  // Im of m = 0
    }
}

template <typename T, int NI, int GROUPS>
cudaError_t launch_orbits3(int L, int p, const uint32_t *start, const T *atab, const short2 *rmap,
                           const uint8_t *parity, const typename C3<T>::V *me,
                           typename C3<T>::V *le, cudaStream_t st) {
    const int rows = orb_rows(orb_items(NI, GROUPS), p);
    const size_t smem = GROUPS * (size_t(8) * orb_stride(rows, p) * sizeof(T) +
                                  size_t(8) * rows * sizeof(int));
    cudaError_t e = cudaFuncSetAttribute(k3_m2l_orbits<T, NI, GROUPS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    int64_t grid = 0;
    for (int k = 2; k <= L; ++k) grid += orb_blocks(k, rows);
    k3_m2l_orbits<T, NI, GROUPS><<<unsigned(grid), ORB_THREADS, smem, st>>>(L, p, start, atab, rmap,
                                                                            parity, me, le);
    return cudaGetLastError();
}

// NI and GROUPS by size: four groups of orbits shorten the serial chain, small
// runs of targets make more blocks; runs of 1,024 pairs (one group) reuse the
// operators best.  M2L of one GB300, us, <4,1> / <2,4> / <1,4>:
//   FP64  L = 2, p = 6   954 / 131 / 84      FP32  443 / 55 / 45
//         L = 3, p = 8   1421 / 320 / 324          713 / 90 / 94
//         L = 4, p = 8   2459 / 2305 / 2241        899 / 549 / 545
// and above the 128 pairs that <2,4> holds, <4,1> / <4,4>: FP64 L = 4, p = 11
// 8258 / 7618, FP32 L = 4, p = 12 2845 / 4434.
template <typename T>
cudaError_t launch_m2l_orbits(int L, int p, const uint32_t *start, const T *atab,
                              const short2 *rmap, const uint8_t *parity,
                              const typename C3<T>::V *me, typename C3<T>::V *le,
                              cudaStream_t st) {
    const int64_t sms = device_sm_count();
    auto blocks = [&](int ni, int groups) {
        int64_t n = 0;
        for (int k = 2; k <= L; ++k) n += orb_blocks(k, orb_rows(orb_items(ni, groups), p));
        return n;
    };
    if (p <= 8 && blocks(2, 4) < sms)
        return launch_orbits3<T, 1, 4>(L, p, start, atab, rmap, parity, me, le, st);
    if (p <= 11 && (sizeof(T) == 8 || p <= 8))
        return launch_orbits3<T, 2, 4>(L, p, start, atab, rmap, parity, me, le, st);
    if (sizeof(T) == 8 || blocks(4, 1) < 2 * sms)
        return launch_orbits3<T, 4, 4>(L, p, start, atab, rmap, parity, me, le, st);
    return launch_orbits3<T, 4, 1>(L, p, start, atab, rmap, parity, me, le, st);
}

// ---------------------------------------------------------------------------
// M2L of the mixed path as GEMMs.  The coefficients of a real potential with
// degrees < p are p^2 real numbers: Re of every stored (n, m), then Im of
// those with m > 0 (Im of m = 0 is zero).  In that basis each offset's
// translation is a fixed real p^2 x p^2 matrix A_delta (built on the host in
// FP64 from the M2L sum, rounded to FP32; stored transposed, k-major, padded
// to NRP = p^2 rounded up to 32); rmap[r] = (coefficient, part) of real index
// r, part 0 = Re, 1 = Im, 2 = Re of an m = 0 coefficient (its Im is zero).
// (p <= 8: above, and on small trees, M2L goes by orbits.)
// ---------------------------------------------------------------------------
constexpr int MG_THREADS = 128;
#ifndef MG_PIPE_ROWS
#define MG_PIPE_ROWS 128  // target rows per block of the pipelined M2L (64 or 128)
#endif

__host__ __device__ constexpr int mg_nrp(int p) { return (p * p + 31) / 32 * 32; }
// The same GEMMs with the operands of the next offset in flight: for p <= 8
// (a whole operator is one K chunk) the operator and the source rows of
// offset i + 1 are copied with cp.async (16-byte chunks; 8 when a box's
// coefficients are an odd number of float2; rows of empty or outside boxes
// zero-filled without a read) into the second operator buffer and a raw row
// buffer while offset i multiplies; then the raw rows are split into the
// k-major real layout.  Offsets whose 64 source rows are all empty skip
// their multiply.
__device__ __forceinline__ void cp_async_z(void *dst, const void *src, int bytes, bool pred) {
    const unsigned d = unsigned(__cvta_generic_to_shared(dst));
    const int n = pred ? bytes : 0;
    if (bytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n));
}

template <int P, int R>
constexpr size_t mgp_smem_bytes() {
    return size_t(mg_nrp(P) * (R + 4) + 2 * mg_nrp(P) * mg_nrp(P)) * sizeof(float) +
           size_t(R) * (P * (P + 1) / 2) * sizeof(float2);
}

// blocks of level l in an all-levels M2L launch of R-row blocks:
// ceil(8^(l-1) / R) x 8
__host__ __device__ __forceinline__ int64_t mg_blocks(int l, int R) {
    return ((int64_t(1) << (3 * (l - 1))) + R - 1) / R * 8;
}

// R target rows per block (R Morton-consecutive parent cells: 4 x 4 x 4 for
// 64, 8 x 4 x 4 for 128), R / 16 rows per thread.
template <int P, int R>
__global__ void __launch_bounds__(MG_THREADS) k3_m2l_pipe(int L, const uint32_t *__restrict__ start,
                                                        const float *__restrict__ atab,
                                                        const float2 *__restrict__ me,
                                                        float2 *__restrict__ le) {
    // this block's level: levels 2..L one after another in the grid
    int l = 2;
    int64_t bid = blockIdx.x;
    while (l < L && bid >= mg_blocks(l, R)) bid -= mg_blocks(l++, R);
    constexpr int NC = P * (P + 1) / 2, NR = P * P, NRP = mg_nrp(P), CG = NRP / 8;
    static_assert(NRP <= 64, "one K chunk per operator");
    constexpr int XS = R + 4, RT = R / 16;
    constexpr int BITS = R == 128 ? 7 : 6;              // Morton bits of the block's parents
    constexpr int NX = 1 << ((BITS + 2) / 3), NY = 1 << ((BITS + 1) / 3), NZ = 1 << (BITS / 3);
    constexpr int HX = NX + 2, HY = NY + 2, HZ = NZ + 2;
    static_assert(R == 64 || R == 128, "rows per block");
    constexpr int CB = (NC % 2 == 0) ? 16 : 8;          // copy chunk bytes of a row
    constexpr int RCH = NC * 8 / CB;                     // chunks per row
    extern __shared__ __align__(16) float mg_smem[];
    float *xs = mg_smem;                                 // [NRP][XS]
    float *as0 = xs + NRP * XS;                          // 2 x [NRP][NRP]
    float2 *raw = reinterpret_cast<float2 *>(as0 + 2 * NRP * NRP);  // [R][NC]
    __shared__ int srow[2][R];
    __shared__ short imr[NC];
    __shared__ unsigned char offs[216];                  // the class's offsets (cs, d)
    __shared__ int noff;
    // occupied boxes of the parent cells around the block's (one cell of
    // halo), 8 classes each: one bit per class
    __shared__ unsigned char hocc[HX * HY * HZ];
    const int tid = threadIdx.x, rg = tid >> 3, g = tid & 7;
    const int c = int(bid & 7);
    const int64_t np = int64_t(1) << (3 * (l - 1));
    const int64_t p0 = (bid >> 3) * R;
    const int pside = 1 << (l - 1);
    const int hx0 = int(compact3(uint32_t(p0))) - 1, hy0 = int(compact3(uint32_t(p0) >> 1)) - 1,
              hz0 = int(compact3(uint32_t(p0) >> 2)) - 1;
    for (int h = tid; h < HX * HY * HZ; h += MG_THREADS) {
        const int qx = hx0 + h % HX, qy = hy0 + (h / HX) % HY, qz = hz0 + h / (HX * HY);
        unsigned bits = 0;
        if (qx >= 0 && qy >= 0 && qz >= 0 && qx < pside && qy < pside && qz < pside) {
            const uint32_t pb = morton3(uint32_t(qx), uint32_t(qy), uint32_t(qz));
            for (int cs = 0; cs < 8; ++cs)
                if (box_count3(start, L, l, pb * 8u + uint32_t(cs))) bits |= 1u << cs;
        }
        hocc[h] = (unsigned char)bits;
    }
    __syncthreads();
    // a block whose target boxes (class c of its own parent cells) are all
    // empty writes nothing: an empty box's local expansion is never read
    {
        bool mine = false;
        for (int r = tid; r < R; r += MG_THREADS) {
            const int64_t pc = p0 + r;
            if (pc >= np) continue;
            const int qx = int(compact3(uint32_t(pc))), qy = int(compact3(uint32_t(pc) >> 1)),
                      qz = int(compact3(uint32_t(pc) >> 2));
            mine |= (hocc[(qx - hx0) + HX * ((qy - hy0) + HY * (qz - hz0))] >> c) & 1u;
        }
        if (!__syncthreads_or(mine)) return;
    }
    for (int i = tid; i < (NRP - NR) * XS; i += MG_THREADS) xs[NR * XS + i] = 0.f;
    for (int j = tid; j < NC; j += MG_THREADS) {
        int n = 0;
        while ((n + 1) * (n + 2) / 2 <= j) ++n;
        imr[j] = short(j == n * (n + 1) / 2 ? -1 : NC + j - n - 1);
    }
    if (tid == 0) {
        int k = 0;
        for (int o = 0; o < 216; ++o) {
            const int cs = o / 27, d = o % 27;
            const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
            const int ex = (c & 1) - (cs & 1) - 2 * dx, ey = ((c >> 1) & 1) - ((cs >> 1) & 1) - 2 * dy,
                      ez = (c >> 2) - (cs >> 2) - 2 * dz;
            if (ex >= -1 && ex <= 1 && ey >= -1 && ey <= 1 && ez >= -1 && ez <= 1) continue;
            offs[k++] = (unsigned char)o;
        }
        noff = k;
    }
    __syncthreads();
    const float2 *lev = me + lvl_off3(l) * NC;
    // source box of target row `row` for offset entry o (-1: none), from the
    // halo occupancy (no global load)
    auto source = [&](int o, int row) {
        const int cs = o / 27, d = o % 27;
        const int64_t pc = p0 + row;
        if (pc >= np) return -1;
        const int qx = int(compact3(uint32_t(pc))) + d % 3 - 1,
                  qy = int(compact3(uint32_t(pc) >> 1)) + (d / 3) % 3 - 1,
                  qz = int(compact3(uint32_t(pc) >> 2)) + d / 9 - 1;
        if (qx < 0 || qy < 0 || qz < 0 || qx >= pside || qy >= pside || qz >= pside) return -1;
        if (!((hocc[(qx - hx0) + HX * ((qy - hy0) + HY * (qz - hz0))] >> cs) & 1u)) return -1;
        return int(morton3(uint32_t(qx), uint32_t(qy), uint32_t(qz)) * 8u + uint32_t(cs));
    };
    auto slot_of = [&](int o) {
        const int cs = o / 27, d = o % 27;
        const int ex = (c & 1) - (cs & 1) - 2 * (d % 3 - 1),
                  ey = ((c >> 1) & 1) - ((cs >> 1) & 1) - 2 * ((d / 3) % 3 - 1),
                  ez = (c >> 2) - (cs >> 2) - 2 * (d / 9 - 1);
        return (ex + 3) + 7 * (ey + 3) + 49 * (ez + 3);
    };
    auto issue = [&](int i) {  // copies of offset i (srow[i & 1] ready)
        const int o = offs[i];
        const float *at = atab + size_t(slot_of(o)) * NRP * NRP;
        float *asb = as0 + (i & 1) * NRP * NRP;
        for (int q = tid; q < NRP * NRP / 4; q += MG_THREADS)
            cp_async_z(asb + 4 * q, at + 4 * q, 16, true);
        for (int q = tid; q < R * RCH; q += MG_THREADS) {
            const int row = q / RCH, ch = q - row * RCH;
            const int sb = srow[i & 1][row];
            const char *src = reinterpret_cast<const char *>(sb >= 0 ? lev + int64_t(sb) * NC : lev);
            cp_async_z(reinterpret_cast<char *>(raw + row * NC) + ch * CB, src + ch * CB, CB, sb >= 0);
        }
        cp_async_commit();
    };
    float acc[RT][CG];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < CG; ++j) acc[i][j] = 0.f;
    const int nof = noff;
    bool have = false;
    if (tid < R) {
        srow[0][tid] = source(offs[0], tid);
        have = srow[0][tid] >= 0;
    }
    bool cur_any = __syncthreads_or(have);
    issue(0);
    for (int i = 0; i < nof; ++i) {
        cp_async_wait_all();
        __syncthreads();
        // split the raw rows of offset i into the k-major real layout, and
        // find the source rows of offset i + 1
        for (int q = tid; q < R * NC; q += MG_THREADS) {
            const int row = q % R, j = q / R;
            const float2 v = raw[row * NC + j];
            xs[j * XS + row] = v.x;
            if (imr[j] >= 0) xs[imr[j] * XS + row] = v.y;
        }
        have = false;
        if (tid < R && i + 1 < nof) {
            srow[(i + 1) & 1][tid] = source(offs[i + 1], tid);
            have = srow[(i + 1) & 1][tid] >= 0;
        }
        const bool next_any = __syncthreads_or(have);
        if (i + 1 < nof) issue(i + 1);
        if (cur_any) {
            const float *asb = as0 + (i & 1) * NRP * NRP;
#pragma unroll 4
            for (int k = 0; k < NRP; ++k) {
                float xv[RT];
#pragma unroll
                for (int i4 = 0; i4 < RT; i4 += 4) {
                    const float4 x4 = *reinterpret_cast<const float4 *>(xs + k * XS + RT * rg + i4);
                    xv[i4] = x4.x;
                    xv[i4 + 1] = x4.y;
                    xv[i4 + 2] = x4.z;
                    xv[i4 + 3] = x4.w;
                }
                const float *ar = asb + k * NRP + g * CG;
#pragma unroll
                for (int j4 = 0; j4 < CG; j4 += 4) {
                    const float4 a4 = *reinterpret_cast<const float4 *>(ar + j4);
                    const float av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t)
#pragma unroll
                        for (int i = 0; i < RT; ++i)
                            acc[i][j4 + t] = fmaf(xv[i], av[t], acc[i][j4 + t]);
                }
            }
        }
        cur_any = next_any;
    }
    cp_async_wait_all();
    float *lef = reinterpret_cast<float *>(le + lvl_off3(l) * NC);
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const int64_t pc = p0 + RT * rg + i;
        if (pc >= np) continue;
        const int64_t box = pc * 8 + c;
#pragma unroll
        for (int j = 0; j < CG; ++j) {
            const int r = g * CG + j;
            if (r >= NR) continue;
            // real index r: Re of coefficient r (r < NC), else Im of the
            // (r - NC)-th coefficient with m > 0
            if (r < NC) {
                lef[(box * NC + r) * 2] = acc[i][j];
                int n = 0;
                while ((n + 1) * (n + 2) / 2 <= r) ++n;
                if (r == n * (n + 1) / 2) lef[(box * NC + r) * 2 + 1] = 0.f;
            }
        }
    }
    // Im parts: thread columns r >= NC map back through imr (search)
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const int64_t pc = p0 + RT * rg + i;
        if (pc >= np) continue;
        const int64_t box = pc * 8 + c;
#pragma unroll
        for (int j = 0; j < CG; ++j) {
            const int r = g * CG + j;
            if (r < NC || r >= NR) continue;
            for (int jj = 0; jj < NC; ++jj)
                if (imr[jj] == r) lef[(box * NC + jj) * 2 + 1] = acc[i][j];
        }
    }
}

// ---------------------------------------------------------------------------
// M2L of the mixed path on the 5th-generation tensor cores (p <= 8): the
// same real GEMMs as k3_m2l_pipe with TF32 inputs split into hi and lo
// parts, each rounded to TF32 (a_hi = a to nearest, a_lo = a - a_hi to
// nearest: a - a_hi - a_lo is within about 2^-23 |a|, near an FP32
// rounding; the products a_hi b_hi + a_lo b_hi + a_hi b_lo leave out
// a_lo b_lo, about 2^-24) and FP32 accumulation in tensor memory, spread
// over TC3_SETS accumulator sets that consecutive pairs take in turn, read
// out every TC3_FLUSH pairs and added in registers (round to nearest): a
// chain of MMA additions into one accumulator spans two pairs, 48 steps.  (With one set the potential of a 20k-charge test
// drifted 1.2e-5 from the FP64 path, past the mixed path's 1e-5 budget,
// whether the split truncated or rounded: the error grows with the length
// of the accumulation chain, some 4,500 MMA steps per output here.)  A CTA takes the 128
// Morton-consecutive parent cells of a pipelined-M2L block and two target
// classes c0, c0 + 1: M = 128 rows (TMEM lanes), 2 x NRP accumulator
// columns.  For each (source class cs, parent offset d) pair in a fixed
// order whose operator is not near for one of the two classes and whose
// sources are not all empty, the 128 source rows (the expansion of box
// (P + d) 8 + cs in the real basis, zero for an empty or outside box) are
// split into hi and lo images in shared memory, K-major without swizzle
// (core matrices of 8 rows x 16 bytes: element (m, k) at
// ((k / 4) 128 + m) 16 + (k mod 4) 4 bytes), the two classes' operator
// images (host-built in the same layout, B(n, k) = A_delta[k][n]) are copied
// beside them, and one thread issues the MMAs and commits them to an
// mbarrier that the next pair waits on (bounded) before it overwrites the
// images.  A wait that gives up sets PETFMM_ETIMEOUT and the CTA writes
// nothing.
// ---------------------------------------------------------------------------
constexpr int TC3_STAGERS = 256;  // two threads per row (and per TMEM lane)
constexpr int TC3_THREADS = TC3_STAGERS + 32;  // and a warp that copies and issues
constexpr int TC3_ROWS = 128;
constexpr int TC3_SETS = 4;       // accumulator sets
constexpr int TC3_FLUSH = 8;      // pairs between read-outs of the sets into registers

// coefficient index n (n + 1) / 2 + m of the t-th coefficient with m > 0
template <int P> __host__ __device__ constexpr int tc3_imcoef(int t) {
    int r = 0;
    for (int n = 1; n < P; ++n)
        for (int m = 1; m <= n; ++m) {
            if (r == t) return n * (n + 1) / 2 + m;
            ++r;
        }
    return 0;
}

// v rounded to TF32 (nearest, ties away), in FP32 format
__device__ __forceinline__ float tf32_rna(float v) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
    return __uint_as_float(r);
}

// The tensor-core M2L's input (K) basis, coefficient by coefficient: Re of
// coefficient j, then Im of j if its m > 0 (zero padding to NRP), so that
// each half of K covers about half of a row's coefficients and each of the
// two threads staging a row loads about half of it.  The output (N) basis
// stays the one of the M2L matrices (Re of all, then Im of m > 0).
template <int P> struct Tc3Basis {
    int j[mg_nrp(P)];     // coefficient, -1 for padding
    int part[mg_nrp(P)];  // 0 Re, 1 Im
    __host__ __device__ constexpr Tc3Basis() : j(), part() {
        int k = 0;
        for (int n = 0; n < P; ++n)
            for (int m = 0; m <= n; ++m) {
                const int jj = n * (n + 1) / 2 + m;
                j[k] = jj;
                part[k++] = 0;
                if (m > 0) {
                    j[k] = jj;
                    part[k++] = 1;
                }
            }
        for (; k < mg_nrp(P); ++k) {
            j[k] = -1;
            part[k] = 0;
        }
    }
    // the coefficients K half h reads: [lo, hi]
    __host__ __device__ constexpr int jlo(int h) const {
        int r = 1 << 30;
        for (int k = h * (mg_nrp(P) / 2); k < (h + 1) * (mg_nrp(P) / 2); ++k)
            if (j[k] >= 0 && j[k] < r) r = j[k];
        return r == (1 << 30) ? 0 : r;
    }
    __host__ __device__ constexpr int jhi(int h) const {
        int r = -1;
        for (int k = h * (mg_nrp(P) / 2); k < (h + 1) * (mg_nrp(P) / 2); ++k)
            if (j[k] > r) r = j[k];
        return r;
    }
};

// Coefficients a K half reads, and the most either half reads.
template <int P> __host__ __device__ constexpr int tc3_half_j0(int h) { return Tc3Basis<P>{}.jlo(h); }
template <int P> __host__ __device__ constexpr int tc3_half_nw(int h) {
    return Tc3Basis<P>{}.jhi(h) - Tc3Basis<P>{}.jlo(h) + 1;
}
template <int P> __host__ __device__ constexpr int tc3_nw() {
    return tc3_half_nw<P>(0) > tc3_half_nw<P>(1) ? tc3_half_nw<P>(0) : tc3_half_nw<P>(1);
}

// Registers for a half row: from coefficient j0 rounded down to even (so
// that rows with an even coefficient count load 16-byte pieces), one spare.
template <int P> __host__ __device__ constexpr int tc3_nwr() { return tc3_nw<P>() + 2; }

// One K half H of a row of A in the input basis, hi and lo, into the K-major
// images, from the coefficients (j0(H) rounded down to even) .. of the row
// held in w.
template <int P, int H>
__device__ __forceinline__ void tc3_write_half(const float2 (&w)[tc3_nwr<P>()], float *ahi, float *alo,
                                               int row) {
    constexpr int NRP = mg_nrp(P), KH = NRP / 2;
    constexpr Tc3Basis<P> bas{};
    constexpr int J0 = tc3_half_j0<P>(H) & ~1;
#pragma unroll
    for (int g = 0; g < KH / 4; ++g) {
        float v4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = H * KH + 4 * g + e;
            const int jj = bas.j[k];
            v4[e] = jj < 0 ? 0.f : (bas.part[k] ? w[jj - J0].y : w[jj - J0].x);
        }
        float4 h4, l4;
        h4.x = tf32_rna(v4[0]);
        h4.y = tf32_rna(v4[1]);
        h4.z = tf32_rna(v4[2]);
        h4.w = tf32_rna(v4[3]);
        l4 = make_float4(tf32_rna(v4[0] - h4.x), tf32_rna(v4[1] - h4.y), tf32_rna(v4[2] - h4.z),
                         tf32_rna(v4[3] - h4.w));
        const int kg = H * (KH / 4) + g;
        reinterpret_cast<float4 *>(ahi)[kg * TC3_ROWS + row] = h4;
        reinterpret_cast<float4 *>(alo)[kg * TC3_ROWS + row] = l4;
    }
}

template <int P> constexpr size_t tc3_smem_bytes() {
    // one A buffer of hi and lo (128 x NRP each), then four slots of a
    // class's B hi and lo (NRP x NRP each)
    return size_t(2 * TC3_ROWS * mg_nrp(P) + 8 * mg_nrp(P) * mg_nrp(P)) * sizeof(float);
}

// blocks of level l in the all-levels launch: 128 parent cells x 4 class pairs
__host__ __device__ __forceinline__ int64_t tc3_blocks(int l) {
    return ((int64_t(1) << (3 * (l - 1))) + TC3_ROWS - 1) / TC3_ROWS * 4;
}

template <int P>
__global__ void __launch_bounds__(TC3_THREADS, 1) k3_m2l_tc(int L, const uint32_t *__restrict__ start,
                                                          const float *__restrict__ bimg,
                                                          const float2 *__restrict__ me,
                                                          float2 *__restrict__ le,
                                                          long long spin_limit, int *status) {
    constexpr int NC = P * (P + 1) / 2, NR = P * P, NRP = mg_nrp(P), KG = NRP / 4;
    static_assert(NRP <= 64 && NRP % 16 == 0, "tensor-core M2L orders");
    constexpr int HX = 10, HY = 6, HZ = 6;  // the block's 8 x 4 x 4 parent cells and one of halo
    constexpr int AIMG = TC3_ROWS * NRP;    // floats of one A image (hi or lo)
    constexpr int BIMG = 2 * NRP * NRP;     // floats of one class's B images (hi, lo)
    constexpr int NSLOT = 4;                // B slots: step s = 2 pair + class uses slot s mod 4
    extern __shared__ __align__(1024) float tsm[];
    float *ahi = tsm, *alo = ahi + AIMG;    // [KG][128][4] each
    float *bsm = alo + AIMG;                // NSLOT x [hi, lo][KG][NRP][4]
    __shared__ unsigned char hocc[HX * HY * HZ];
    __shared__ unsigned char plist[216];    // the pairs that run: offset entries o
    __shared__ uint32_t pmask[7];           // offsets o with an occupied source row
    __shared__ int npl;
    __shared__ __align__(8) uint64_t mbar[NSLOT], bbar[NSLOT];  // per slot: MMAs done, B landed
    __shared__ uint32_t tslot;
    __shared__ uint32_t set_used;  // bit 2 set + class: that accumulator was written
    int l = 2;
    int64_t bid = blockIdx.x;
    while (l < L && bid >= tc3_blocks(l)) bid -= tc3_blocks(l++);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int row = tid & (TC3_ROWS - 1), half = (tid / TC3_ROWS) & 1;  // two stagers per row
    const bool stager = tid < TC3_STAGERS;
    const int c0 = 2 * int(bid & 3);
    const int64_t np = int64_t(1) << (3 * (l - 1));
    const int64_t p0 = (bid >> 2) * TC3_ROWS;
    const int pside = 1 << (l - 1);
    const int hx0 = int(compact3(uint32_t(p0))) - 1, hy0 = int(compact3(uint32_t(p0) >> 1)) - 1,
              hz0 = int(compact3(uint32_t(p0) >> 2)) - 1;
    if (tid < 7) pmask[tid] = 0;
    for (int h = tid; h < HX * HY * HZ; h += TC3_THREADS) {
        const int qx = hx0 + h % HX, qy = hy0 + (h / HX) % HY, qz = hz0 + h / (HX * HY);
        unsigned bits = 0;
        if (qx >= 0 && qy >= 0 && qz >= 0 && qx < pside && qy < pside && qz < pside) {
            const uint32_t pb = morton3(uint32_t(qx), uint32_t(qy), uint32_t(qz));
            for (int cs = 0; cs < 8; ++cs)
                if (box_count3(start, L, l, pb * 8u + uint32_t(cs))) bits |= 1u << cs;
        }
        hocc[h] = (unsigned char)bits;
    }
    __syncthreads();
    // this thread's row: parent cell p0 + row, its halo position
    const int64_t pc = p0 + row;
    const bool row_ok = pc < np;
    const int rx = int(compact3(uint32_t(pc))), ry = int(compact3(uint32_t(pc) >> 1)),
              rz = int(compact3(uint32_t(pc) >> 2));
    const unsigned own = row_ok ? hocc[(rx - hx0) + HX * ((ry - hy0) + HY * (rz - hz0))] : 0u;
    // nothing to do if the block's targets of both classes are empty
    if (!__syncthreads_or(int((own >> c0) & 3u))) return;
    // the row's source box for offset entry o (-1: empty or outside)
    auto source = [&](int o) {
        if (!row_ok) return -1;
        const int cs = o / 27, dd = o % 27;
        const int qx = rx + dd % 3 - 1, qy = ry + (dd / 3) % 3 - 1, qz = rz + dd / 9 - 1;
        if (qx < 0 || qy < 0 || qz < 0 || qx >= pside || qy >= pside || qz >= pside) return -1;
        if (!((hocc[(qx - hx0) + HX * ((qy - hy0) + HY * (qz - hz0))] >> cs) & 1u)) return -1;
        return int(morton3(uint32_t(qx), uint32_t(qy), uint32_t(qz)) * 8u + uint32_t(cs));
    };
    // class cc's operator slot for offset entry o, or -1 where it is near
    auto op_slot = [&](int o, int cc) {
        const int c = c0 + cc, cs = o / 27, dd = o % 27;
        const int ex = (c & 1) - (cs & 1) - 2 * (dd % 3 - 1),
                  ey = ((c >> 1) & 1) - ((cs >> 1) & 1) - 2 * ((dd / 3) % 3 - 1),
                  ez = (c >> 2) - (cs >> 2) - 2 * (dd / 9 - 1);
        if (ex >= -1 && ex <= 1 && ey >= -1 && ey <= 1 && ez >= -1 && ez <= 1) return -1;
        return (ex + 3) + 7 * (ey + 3) + 49 * (ez + 3);
    };
    // the pairs that run: an operator for one of the two classes, a source row
    if (stager && half == 0)
        for (int o = 0; o < 216; ++o)
            if (source(o) >= 0) atomicOr(&pmask[o >> 5], 1u << (o & 31));
    __syncthreads();
    if (tid == 0) {
        int k = 0;
        for (int o = 0; o < 216; ++o)
            if (((pmask[o >> 5] >> (o & 31)) & 1u) && (op_slot(o, 0) >= 0 || op_slot(o, 1) >= 0))
                plist[k++] = (unsigned char)o;
        npl = k;
        for (int b = 0; b < NSLOT; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar[b])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bbar[b])));
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
        set_used = 0;
    }
    constexpr uint32_t NCOLS = TC3_SETS * 2 * NRP;  // 256 or 512: a power of two
    static_assert(NCOLS <= 512, "TMEM columns");
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&tslot)),
                     "r"(NCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tslot;
    const int n_pairs = npl;
    // kind::tf32: D F32 (bit 4), A and B TF32 (bits 7, 10), both K-major,
    // N / 8 at bit 17, M / 16 at bit 24
    constexpr uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(NRP >> 3) << 17) |
                               (uint32_t(TC3_ROWS >> 4) << 24);
    constexpr uint32_t LBO_A = TC3_ROWS * 16, SBO_A = 128, LBO_B = NRP * 16, SBO_B = 128;
    const float2 *lev = me + lvl_off3(l) * NC;
    // Pipeline over the pairs i = 0 .. n_pairs - 1, each two steps s = 2 i +
    // class: ORCH (warp 8, one thread) copies the operator images of pair
    // i + 1 into slots (2 i + 2 + class) mod 4 while pair i multiplies; the
    // stagers hold pair i + 1's source rows in registers, loaded while pair
    // i multiplies, and write them into the single A buffer once ORCH has
    // seen pair i's MMAs done (barrier 1), then ORCH issues pair i + 1's
    // MMAs (barrier 2).  Every step commits once to its slot's mbar (also a
    // near class with no MMA), so mbar[s mod 4] phase s / 4 is "step s done".
    constexpr int ORCH = TC3_STAGERS;
    bool ok = true;
    uint32_t used = 0;        // ORCH: accumulators written
    int ncopy[NSLOT] = {0, 0, 0, 0};  // ORCH: copies into each slot
    int committed = 0;                // ORCH: steps committed
    auto wait_step = [&](int st) {  // ORCH: step st's MMAs done
        if (ok && st >= 0)
            ok = mbar_wait(smem_addr(&mbar[st % NSLOT]), uint32_t(st / NSLOT) & 1u, spin_limit);
    };
    auto copy_pair = [&](int i) {  // ORCH: pair i's images into slots (2 i + class) mod 4
        const int o = plist[i];
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            const int os = op_slot(o, cc);
            const int sl = (2 * i + cc) % NSLOT;
            if (os < 0 || !ok) continue;
            const uint32_t bb = smem_addr(&bbar[sl]);
            mbar_arrive_expect_tx(bb, uint32_t(BIMG * 4));
            bulk_g2s(smem_addr(bsm + sl * BIMG), bimg + size_t(os) * BIMG, uint32_t(BIMG * 4), bb);
            ++ncopy[sl];
        }
    };
    // rows of pair 0 in registers; the images of pair 0 on their way
    // this stager's half of the next pair's row, in registers, from its
    // first coefficient rounded down to even
    constexpr int NWR = tc3_nwr<P>();
    const int j0 = (half ? tc3_half_j0<P>(1) : tc3_half_j0<P>(0)) & ~1;
    const int jend = (half ? tc3_half_j0<P>(1) + tc3_half_nw<P>(1) : tc3_half_j0<P>(0) + tc3_half_nw<P>(0));
    const int nw = jend - j0;  // coefficients wanted, <= NWR
    float2 w[NWR];
    auto load_row = [&](int i) {
        const int sb = (stager && i < n_pairs) ? source(plist[i]) : -1;
        const float2 *src = lev + int64_t(sb < 0 ? 0 : sb) * NC + j0;
        if constexpr (NC % 2 == 0) {
            // 16-byte pieces: the row starts 16-byte aligned and j0 is even
#pragma unroll
            for (int t = 0; t < NWR / 2; ++t) {
                float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (sb >= 0 && 2 * t < nw && j0 + 2 * t + 1 < NC)
                    q4 = reinterpret_cast<const float4 *>(src)[t];
                else if (sb >= 0 && 2 * t < nw)
                    q4 = make_float4(src[2 * t].x, src[2 * t].y, 0.f, 0.f);
                w[2 * t] = make_float2(q4.x, q4.y);
                w[2 * t + 1] = make_float2(q4.z, q4.w);
            }
        } else {
#pragma unroll
            for (int t = 0; t < NWR; ++t) w[t] = (sb >= 0 && t < nw) ? src[t] : make_float2(0.f, 0.f);
        }
    };
    // the stager's class, its row's sums so far (registers, FP32 round to
    // nearest): every TC3_FLUSH pairs the accumulator sets are read out of
    // TMEM, added here, and the next pairs start the sets afresh
    const int my_cc = half;
    float acc[NRP];
#pragma unroll
    for (int k = 0; k < NRP; ++k) acc[k] = 0.f;
    load_row(0);
    if (tid == ORCH && n_pairs > 0) copy_pair(0);
    for (int i = 0; i < n_pairs && ok; ++i) {
        // barrier 1: the A buffer is free (pair i - 1's MMAs done)
        if (tid == ORCH) wait_step(2 * i - 1);
        ok = __syncthreads_and(int(tid != ORCH || ok)) != 0;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (stager) {
            // A: the row in the input basis, each of the two stagers of a row
            // writing its half of the K groups
            if (half == 0)
                tc3_write_half<P, 0>(w, ahi, alo, row);
            else
                tc3_write_half<P, 1>(w, ahi, alo, row);
            asm volatile("fence.proxy.async.shared::cta;");
        } else if (tid == ORCH && i + 1 < n_pairs) {
            // pair i + 1's images: its slots last held steps 2 i - 2 and
            // 2 i - 1, done (waited above)
            copy_pair(i + 1);
        }
        // barrier 2: A(i) written
        __syncthreads();
        if (tid == ORCH && ok) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t dah = mma_desc(smem_addr(ahi), LBO_A, SBO_A);
            const uint64_t dal = mma_desc(smem_addr(alo), LBO_A, SBO_A);
            constexpr uint64_t sa = (2 * LBO_A) >> 4, sbk = (2 * LBO_B) >> 4;
            const int set = i % TC3_SETS;
            const int o = plist[i];
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                const int sl = (2 * i + cc) % NSLOT;
                if (op_slot(o, cc) >= 0 && ok) {
                    ok = mbar_wait(smem_addr(&bbar[sl]), uint32_t(ncopy[sl] - 1) & 1u, spin_limit);
                    if (ok) {
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        const uint32_t bh = smem_addr(bsm + sl * BIMG);
                        const uint64_t dbh = mma_desc(bh, LBO_B, SBO_B);
                        const uint64_t dbl = mma_desc(bh + uint32_t(NRP * NRP * 4), LBO_B, SBO_B);
                        const uint32_t dt = tbase + uint32_t((2 * set + cc) * NRP);
                        const uint32_t bit = 1u << (2 * set + cc);
                        const bool was = (used & bit) != 0;
#pragma unroll
                        for (int ks = 0; ks < NRP / 8; ++ks) {
                            mma_tf32(dt, dah + ks * sa, dbh + ks * sbk, idesc,
                                     (was || ks > 0) ? 1u : 0u);
                            mma_tf32(dt, dal + ks * sa, dbh + ks * sbk, idesc, 1u);
                            mma_tf32(dt, dah + ks * sa, dbl + ks * sbk, idesc, 1u);
                        }
                        used |= bit;
                    }
                }
                // one commit per step (also with no MMA)
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        smem_addr(&mbar[sl])));
                ++committed;
            }
        }
        // the stagers load pair i + 1's rows while pair i multiplies
        load_row(i + 1);
        if ((i + 1) % TC3_FLUSH == 0 || i + 1 == n_pairs) {
            // flush: every MMA so far done, the sets added into registers
            if (tid == ORCH) {
                wait_step(2 * i + 1);
                set_used = used;
            }
            ok = __syncthreads_and(int(tid != ORCH || ok)) != 0;
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            if (stager) {
                const uint32_t su = set_used;
                for (int set = 0; set < TC3_SETS; ++set) {  // the sets in order
                    if (!((su >> (2 * set + my_cc)) & 1u)) continue;  // uniform in the warp
                    const uint32_t taddr = tbase + (uint32_t((warp & 3) * 32) << 16) +
                                           uint32_t((2 * set + my_cc) * NRP);
#pragma unroll
                    for (int q = 0; q < NRP / 16; ++q) {
                        float t16[16];
                        tmem_ld16(taddr + uint32_t(16 * q), t16);
#pragma unroll
                        for (int k = 0; k < 16; ++k) acc[16 * q + k] += t16[k];
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();
            if (tid == ORCH) used = 0;  // the next MMAs overwrite the sets
        }
    }
    if (tid == ORCH) {
        wait_step(2 * n_pairs - 1);
        if (!ok) {
            set_status(status, ST_ETIMEOUT);
            // the copies and MMAs in flight finish before the memory goes
            // (bounded)
            for (int sl = 0; sl < NSLOT; ++sl)
                if (ncopy[sl] > 0) mbar_wait(smem_addr(&bbar[sl]), uint32_t(ncopy[sl] - 1) & 1u, 1LL << 26);
            if (committed > 0) {  // the last commit covers every earlier MMA
                const int st = committed - 1;
                mbar_wait(smem_addr(&mbar[st % NSLOT]), uint32_t(st / NSLOT) & 1u, 1LL << 26);
            }
        }
    }
    ok = __syncthreads_and(int(tid != ORCH || ok)) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok && stager) {
        // warps 0-3 take class c0 (TMEM lanes 32 w ..), warps 4-7 class c0 + 1
        float *lef = reinterpret_cast<float *>(le + lvl_off3(l) * NC);
        const int c = c0 + my_cc;
        const float *v = acc;
        if (row_ok && ((own >> c) & 1u)) {
            float *dst = lef + (pc * 8 + c) * NC * 2;
#pragma unroll
            for (int j = 0; j < NC; ++j) dst[2 * j] = v[j];
            int t = 0;
#pragma unroll
            for (int n = 0; n < P; ++n)
#pragma unroll
                for (int m = 0; m <= n; ++m) {
                    const int j = n * (n + 1) / 2 + m;
                    dst[2 * j + 1] = m == 0 ? 0.f : v[NC + t];
                    t += m > 0 ? 1 : 0;
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(NCOLS));
}

// ---------------------------------------------------------------------------
// M2M and L2L by reflections.  In the real basis of the M2L matrices the
// operator of child octant c is S_c A S_c with the one of octant 0 and S_c the
// signs of the coefficients under the reflections c (bits of c against a
// coefficient's parities q).  So all eight children of a box share one real
// p^2 x p^2 product:
//   M2M  M'_r = sum_k A[k][r] H[q(r) ^ q(k)][k],
//        H[g][k] = sum_c (-1)^popc(g & c) M_c[k]  (three butterfly stages)
//   L2L  L_c[r] = sum_f (-1)^popc((f ^ q(r)) & c) Z_f[r],
//        Z_f[r] = sum over the k of parity class f of B[k][r] L[k]
// (the rows of B and L sorted by class).  A thread per (box, coefficient),
// about 256 a block; operators come through L1.  Bound by launches and load
// latency: one GB300, M2M / L2L together, all levels:
//   262,144 charges, L = 4, p = 8, FP64    1.22 / 0.08 ms
//   2 M uniform charges, L = 5, p = 8, FP32    0.135 / 0.088 ms
// (a warp per box over the complex sums, in FP32 eight real matrices).
// ---------------------------------------------------------------------------
struct Shift3 {
    int p, nr, boxes;           // terms, p^2, boxes per block
    int cls[9];                 // rows of class f: cls[f] .. cls[f + 1]
};

// Boxes of level l (M2M: from level l + 1; L2L: to level l + 1).
template <typename T, bool L2L>
__global__ void __launch_bounds__(256) k3_shift(int l, int L, const Shift3 s,
                                                const uint32_t *__restrict__ start,
                                                const T *__restrict__ op,
                                                const short2 *__restrict__ rmap,
                                                const uint8_t *__restrict__ par,
                                                const uint16_t *__restrict__ order,
                                                typename C3<T>::V *__restrict__ ex) {
    __shared__ T sh[L2L ? 256 : 256 * 8];
    __shared__ uint8_t spar[256];
    const int nr = s.nr, nc = nc3(s.p);
    const int w = int(threadIdx.x) / nr, r = int(threadIdx.x) - w * nr;
    const int64_t b = int64_t(blockIdx.x) * s.boxes + w;
    const bool act = w < s.boxes && b < (int64_t(1) << (3 * l)) &&
                     box_count3(start, L, l, uint32_t(b)) != 0;
    const short2 rm = w < s.boxes ? rmap[r] : make_short2(0, 0);
    const int q = w < s.boxes ? par[r] : 0;
    // real element rm of a series: component 2 coefficient + (Im: 1)
    const int at = 2 * rm.x + (rm.y == 1 ? 1 : 0);
    if (w == 0) spar[r] = uint8_t(q);
    T v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = T(0);
    if (!L2L) {
        if (act) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t cb = uint32_t(b) * 8u + uint32_t(c);
                if (box_count3(start, L, l + 1, cb) != 0)
                    v[c] = reinterpret_cast<const T *>(ex + (lvl_off3(l + 1) + cb) * nc)[at];
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (!(c & o)) {
                        const T a = v[c], d = v[c | o];
                        v[c] = a + d;
                        v[c | o] = a - d;
                    }
        }
        if (w < s.boxes)
#pragma unroll
            for (int c = 0; c < 8; ++c) sh[threadIdx.x * 8 + c] = v[c];
        __syncthreads();
        if (!act) return;
        const T *h = sh + w * nr * 8;
        T acc = T(0);
#pragma unroll 8
        for (int k = 0; k < nr; ++k) acc = fma(op[k * nr + r], h[k * 8 + (q ^ spar[k])], acc);
        T *dst = reinterpret_cast<T *>(ex + (lvl_off3(l) + b) * nc);
        dst[at] = acc;
        if (rm.y == 2) dst[at + 1] = T(0);  // Im of m = 0
    } else {
        if (act) {  // row r of the sorted order
            const short2 o = rmap[order[r]];
            sh[threadIdx.x] = reinterpret_cast<const T *>(
                ex + (lvl_off3(l) + b) * nc)[2 * o.x + (o.y == 1 ? 1 : 0)];
        }
        __syncthreads();
        if (!act) return;
        const T *y = sh + w * nr;
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            T acc = T(0);
#pragma unroll 8
            for (int k = s.cls[f]; k < s.cls[f + 1]; ++k) acc = fma(op[k * nr + r], y[k], acc);
            v[f] = acc;
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (!(c & o)) {
                    const T a = v[c], d = v[c | o];
                    v[c] = a + d;
                    v[c | o] = a - d;
                }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint32_t cb = uint32_t(b) * 8u + uint32_t(c);
            if (box_count3(start, L, l + 1, cb) == 0) continue;
            T *dst = reinterpret_cast<T *>(ex + (lvl_off3(l + 1) + cb) * nc) + at;
            *dst += __popc(q & c) & 1 ? -v[c] : v[c];
        }
    }
}

template <typename T, bool L2L>
cudaError_t launch_shift3(int l, int L, const Shift3 &s, const uint32_t *start, const T *op,
                          const short2 *rmap, const uint8_t *par, const uint16_t *order,
                          typename C3<T>::V *ex, cudaStream_t st) {
    const int64_t blocks = ((int64_t(1) << (3 * l)) + s.boxes - 1) / s.boxes;
    k3_shift<T, L2L><<<unsigned(blocks), unsigned(s.boxes * s.nr + 31) / 32 * 32, 0, st>>>(
        l, L, s, start, op, rmap, par, order, ex);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// L2P in leaf units: phi = sum L~_n^m conj(R_n^m(xi)) and g = grad_xi of it,
// column by column (m >= 0, weight 2 for m > 0: the m and -m terms of a real
// potential are conjugate), with
//   d/dz:  sum conj(R_n^m) L_{n+1}^m
//   d/dx:  sum conj(R_n^m) (L_{n+1}^{m+1} - L_{n+1}^{m-1}) / 2
//   d/dy:  sum conj(R_n^m) (-i / 2) (L_{n+1}^{m+1} + L_{n+1}^{m-1})
// (from d/dz R_n^m = R_{n-1}^m, (d/dx -+ i d/dy) R_n^m = +-R_{n-1}^{m-+1}).
// ---------------------------------------------------------------------------
template <typename T, typename V>
__device__ __forceinline__ void l2p3(const V *lc, int p, T x, T y, T z, T &phi, T &gx, T &gy,
                                     T &gz) {
    const T r2 = x * x + y * y + z * z;
    V rmm = mk<V>(T(1), T(0));
    for (int mu = 0; mu < p; ++mu) {
        if (mu > 0) {
            const T s = T(1) / T(2 * mu);
            rmm = mk<V>((rmm.x * x - rmm.y * y) * s, (rmm.x * y + rmm.y * x) * s);
        }
        const T wgt = mu == 0 ? T(1) : T(2);
        V r1 = rmm, r2v = mk<V>(T(0), T(0));
        for (int n = mu; n < p; ++n) {
            V rn = r1;
            if (n > mu) {
                const T inv = T(1) / T(n * n - mu * mu);
                const T c1 = T(2 * n - 1) * z;
                rn = mk<V>((c1 * r1.x - r2 * r2v.x) * inv, (c1 * r1.y - r2 * r2v.y) * inv);
                r2v = r1;
                r1 = rn;
            }
            const V a = lc[n * (n + 1) / 2 + mu];
            phi += wgt * (a.x * rn.x + a.y * rn.y);  // Re(a conj(rn))
            if (n + 1 < p) {
                const int o = (n + 1) * (n + 2) / 2;
                const V lz = lc[o + mu], lpv = lc[o + mu + 1];
                V lm;
                if (mu >= 1) {
                    lm = lc[o + mu - 1];
                } else {
                    const V l1 = lc[o + 1];
                    lm = mk<V>(-l1.x, l1.y);  // L^-1 = -conj(L^1)
                }
                // Re(conj(rn) A) = rn.x A.x + rn.y A.y
                const T axr = (lpv.x - lm.x) * T(0.5), axi = (lpv.y - lm.y) * T(0.5);
                const T ayr = (lpv.y + lm.y) * T(0.5), ayi = -(lpv.x + lm.x) * T(0.5);
                gx += wgt * (rn.x * axr + rn.y * axi);
                gy += wgt * (rn.x * ayr + rn.y * ayi);
                gz += wgt * (rn.x * lz.x + rn.y * lz.y);
            }
        }
    }
}

template <typename TOut>
__device__ __forceinline__ void store3(void *o, int64_t i, double v) {
    static_cast<TOut *>(o)[i] = TOut(v);
}

// ---------------------------------------------------------------------------
// Near field of the mixed path.  Leaf pairs of at least P3_PAIR_MIN charges
// each are evaluated pairwise (k3_pairs): 1/r and 1/r^3 of a pair of charges
// serve both, 18 FP32 operations where two one-sided sums take 26 and two
// rsqrt.  The other leaf pairs are summed one-sided (k3_near_directed), and a
// last pass (k3_near_final) adds the parts and L2P.  Every part has one writer
// and the parts are added in a fixed order.
//
// A pair item is (leaf A, group of the 13 forward directions); a heavier leaf
// has more groups.  Parts: fwd[g] of A's charges (from group g's neighbours;
// group 0 also the leaf itself), bwd[d] of a leaf's charges from the leaf behind
// it in direction d, own (one-sided).
//
// One warp evaluates a leaf pair, all of it (its reactions have one writer), so
// few or heavy pairs leave the GPU waiting for single warps; the one-sided sums
// are shared by any number of them.  A pair (a leaf with itself) of na nb pairs
// of charges is therefore summed pairwise up to a limit: the largest, in half
// octaves, of which all pairs up to it together hold 16,384 / P3_SHARE; at least
// up to P3_LEAST (a group of three such pairs is no more than the six of 96
// charges that two groups a leaf give); and none where those up to the limit
// together are fewer than P3_ENOUGH.
// Measured (one GB300, whole evaluations, p = 6, us; every pair pairwise / at this
// limit / every pair one-sided): mixed, clustered charges, 5,000 714 / 356 / 323,
// 150,000 16,800 / 2,030 / 1,950, 600,000 279,000 / 18,900 / 18,800; 100,000 charges
// in eight leaves 342,000 / 6,900 / 6,700; even trees, 8,000 329 / 297 / 277,
// 220,000 (54 a leaf) 629 / 629 / 660, 2 M (64) 2,685 / 2,689 / 3,080; below some 48
// a leaf one-sided is up to 15 % faster.  FP64, clustered, 20,000 39,000 / 9,900 /
// 8,400, 150,000 296,000 / 102,000 / 90,000; even, 262,144 10,890 / 10,890 / 17,600.
// With the limit a fixed part of the sum over all pairs, few middling ones among
// many heavy ones still held the launch up (150,000 clustered 2,450).
// ---------------------------------------------------------------------------
constexpr uint32_t P3_PAIR_MIN = 24;
constexpr uint32_t P3_SHARE = 5, P3_SHARE64 = 40;  // of 16,384
constexpr int P3_LEAST = 27;                       // half octave: below 2^14
constexpr uint32_t P3_ENOUGH = 1u << 24, P3_ENOUGH64 = 0;
constexpr int P3_DIRS = 13;
// planes of one entry per charge, fwd and bwd: mixed (the leaf itself in its
// first group) and FP64 (a group by itself in the heaviest leaves)
constexpr int P3_SLOTS = P3_DIRS + P3_DIRS, P3_GROUPS64 = P3_DIRS + 1;
constexpr int P3_SLOTS64 = P3_GROUPS64 + P3_DIRS;

// forward direction k of 13: (dx, dy, dz) with (dz, dy, dx) above zero
__host__ __device__ __forceinline__ void fwd3(int k, int *dx, int *dy, int *dz) {
    const int o = 14 + k;  // of 27, 13 the leaf itself
    *dx = o % 3 - 1;
    *dy = (o / 3) % 3 - 1;
    *dz = o / 9 - 1;
}
// groups of a leaf of n charges, and group g's directions [first, last)
template <int MAX = P3_DIRS> __host__ __device__ __forceinline__ int groups3(uint32_t n) {
    return n <= 16 && MAX == P3_GROUPS64 ? 1 : n <= 96 ? 2 : n <= 384 ? 4 : MAX;
}
__host__ __device__ __forceinline__ int group_first3(int g, int groups) {
    return groups == P3_GROUPS64 ? (g < P3_DIRS ? g : P3_DIRS) : g * P3_DIRS / groups;
}
// the group that sums the leaf itself
__host__ __device__ __forceinline__ int own_group3(int groups) {
    return groups == P3_GROUPS64 ? P3_DIRS : 0;
}
// leaf flags of the final pass: bit d: bwd[d] holds a part; bit 13: own does;
// bit 14: fwd of the leaf's groups do
constexpr uint32_t LF3_OWN = 1u << 13, LF3_FWD = 1u << 14;
// counters: directed items, pair items, per work class the pair items counted and
// placed, blocks of the counting launch done, the limit of a pairwise leaf pair,
// and the leaf pairs of each half octave of their pairs of charges
constexpr int C3_DIRECTED = 0, C3_PAIRS = 1, C3_COUNT = 2, C3_CLASSES = 64,
              C3_PLACED = C3_COUNT + C3_CLASSES, C3_DONE = C3_PLACED + C3_CLASSES,
              C3_LIMIT = C3_DONE + 1, C3_COST = C3_LIMIT + 1, C3_OCTAVES = 64,
              C3_WORDS = C3_COST + C3_OCTAVES;

constexpr uint32_t NO_GROUP3 = ~0u;  // an item with nothing to sum

struct Near3 {
    float4 *own, *slots;  // slots[P3_SLOTS][n], or no pairs
    uint32_t *flags;      // per leaf
    uint32_t *ctrl;       // C3_WORDS counters
    uint2 *directed;      // (leaf, first charge): up to 32 targets
    uint2 *items;         // (leaf, group)
    int64_t n;
    uint32_t pmin;        // P3_PAIR_MIN, or all ones: no pairs
    uint32_t share, enough;  // P3_SHARE, P3_ENOUGH of the path
};

// Half octave of a leaf pair's na nb = x pairs of charges (2^e .. 1.5 2^e .. 2^(e+1)),
// C3_OCTAVES and more: too many for any limit; the end of half octave h.
__device__ __forceinline__ int octave3(uint64_t x) {
    if (x >> 32) return C3_OCTAVES;
    const int e = 31 - __clz(int(uint32_t(x) | 1u));
    return 2 * e + int(e ? (x >> (e - 1)) & 1u : 0u);
}
__device__ __forceinline__ uint64_t octave_end3(int h) {
    return h & 1 ? uint64_t(2) << (h / 2) : uint64_t(3) << (h / 2) >> 1;
}
// Most charges of a leaf that is summed pairwise with one of n charges (n >= 1;
// na nb <= limit is the same for both leaves), 0: none is.
__device__ __forceinline__ uint32_t most3(const Near3 &w, uint32_t n) {
    return n < w.pmin ? 0u : w.ctrl[C3_LIMIT] / n;
}
// Whether a leaf with most = most3 of its charges and a neighbour of n (or
// itself) are summed pairwise.
__device__ __forceinline__ bool pairwise3(const Near3 &w, uint32_t most, uint32_t n) {
    return n >= w.pmin && n <= most;
}

__device__ __forceinline__ uint32_t leaf_count3(const uint32_t *start, int side, int x, int y,
                                                int z) {
    if (x < 0 || y < 0 || z < 0 || x >= side || y >= side || z >= side) return 0;
    const uint32_t b = morton3(uint32_t(x), uint32_t(y), uint32_t(z));
    return start[b + 1] - start[b];
}

// Work class of group g of a leaf of n charges: log2 of targets x sources in
// half steps, heaviest = class 0.
__device__ __forceinline__ int class3(uint32_t n, uint64_t src) {
    const uint64_t cost = uint64_t(n) * src + 1;
    const int e = 63 - __clzll((long long)cost);
    const int c = 2 * e + int(e ? (cost >> (e - 1)) & 1u : 0u);
    return c >= C3_CLASSES ? 0 : C3_CLASSES - 1 - c;
}

// Calls f(class, group) for the pair items of leaf b (n charges) and pair(na nb)
// for its leaf pairs, as if every one of at least pmin charges each were summed
// pairwise.
template <int MAX, typename F, typename G>
__device__ __forceinline__ void leaf_items3(const uint32_t *__restrict__ start, int L, uint32_t b,
                                            uint32_t n, uint32_t pmin, F &&f, G &&pair) {
    const int side = 1 << L;
    const int ix = int(compact3(b)), iy = int(compact3(b >> 1)), iz = int(compact3(b >> 2));
    const int groups = groups3<MAX>(n);
    for (int g = 0; g < groups; ++g) {
        uint64_t src = 0;
        if (g == own_group3(groups)) {
            src = n;
            pair(uint64_t(n) * n);
        }
        for (int k = group_first3(g, groups); k < group_first3(g + 1, groups); ++k) {
            int dx, dy, dz;
            fwd3(k, &dx, &dy, &dz);
            const uint32_t c = leaf_count3(start, side, ix + dx, iy + dy, iz + dz);
            if (c < pmin) continue;
            src += c;
            pair(uint64_t(n) * c);
        }
        f(class3(n, src), g);
    }
}

// Two launches over the leaves: EMIT = false counts the pair items of each
// class and finds the limit of a pairwise leaf pair (its last block), EMIT = true writes them, heaviest class first, the directed items and
// the leaf flags.  A block counts in shared memory and takes its run of each
// list by one atomic (the order of items changes no result).
template <bool EMIT, int MAX>
__global__ void __launch_bounds__(256) k3_near_items(int L, const uint32_t *__restrict__ start,
                                                     Near3 w) {
    __shared__ uint32_t hist[C3_CLASSES], base[C3_CLASSES], ndir, dbase;
    __shared__ uint32_t cost[EMIT ? 1 : C3_OCTAVES];
    __shared__ uint32_t last;
    const int64_t nleaf = int64_t(1) << (3 * L);
    const int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (threadIdx.x < C3_CLASSES) hist[threadIdx.x] = 0;
    if (!EMIT && threadIdx.x < C3_OCTAVES) cost[threadIdx.x] = 0;
    if (threadIdx.x == 0) ndir = 0;
    __syncthreads();
    const uint32_t s0 = b < nleaf ? start[b] : 0u, n = b < nleaf ? start[b + 1] - s0 : 0u;
    const bool big = n >= w.pmin;
    int run = C3_OCTAVES;  // half octave of the leaf pairs not yet counted: a leaf's
    uint32_t pairs = 0;    // neighbours are mostly alike
    auto flush = [&] {
        if (!EMIT && run < C3_OCTAVES) atomicAdd(&cost[run], pairs);
    };
    if (big)
        leaf_items3<MAX>(
            start, L, uint32_t(b), n, w.pmin, [&](int c, int) { atomicAdd(&hist[c], 1u); },
            [&](uint64_t q) {
                if (EMIT) return;
                const int h = octave3(q);
                if (h != run) {
                    flush();
                    run = h;
                    pairs = 0;
                }
                ++pairs;
            });
    if (!EMIT) {
        flush();
        __syncthreads();
        if (threadIdx.x < C3_OCTAVES && cost[threadIdx.x])
            atomicAdd(w.ctrl + C3_COST + threadIdx.x, cost[threadIdx.x]);
        if (threadIdx.x < C3_CLASSES && hist[threadIdx.x]) {
            atomicAdd(w.ctrl + C3_COUNT + threadIdx.x, hist[threadIdx.x]);
            atomicAdd(w.ctrl + C3_PAIRS, hist[threadIdx.x]);
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(w.ctrl + C3_DONE, 1u) + 1u == gridDim.x;
        __syncthreads();
        if (!last) return;
        if (threadIdx.x < C3_OCTAVES) cost[threadIdx.x] = __ldcg(w.ctrl + C3_COST + threadIdx.x);
        __syncthreads();
        if (threadIdx.x == 0) {
            uint64_t sum = 0, limit = 0;
            for (int h = 0; h < C3_OCTAVES; ++h) {
                // (a leaf pair of the half octave taken for one at its end)
                const uint64_t end = octave_end3(h);
                sum += cost[h] * end;
                if (sum >= w.enough && (h <= P3_LEAST || sum * w.share >= end * 16384)) limit = end - 1;
            }
            w.ctrl[C3_LIMIT] = uint32_t(limit);
        }
        return;
    }
    uint32_t mine = 0, at = 0;  // directed items and their place in the block's run
    bool paired = false;        // some pair of the leaf's items is summed pairwise
    if (n) {
        const int side = 1 << L;
        const int ix = int(compact3(uint32_t(b))), iy = int(compact3(uint32_t(b) >> 1)),
                  iz = int(compact3(uint32_t(b) >> 2));
        uint32_t flags = 0;
        const uint32_t most = most3(w, n);
        paired = pairwise3(w, most, n);
        bool directed = !paired;
        for (int k = 0; big && k < P3_DIRS; ++k) {
            int dx, dy, dz;
            fwd3(k, &dx, &dy, &dz);
            const uint32_t f = leaf_count3(start, side, ix + dx, iy + dy, iz + dz);
            const uint32_t r = leaf_count3(start, side, ix - dx, iy - dy, iz - dz);
            const bool fp = pairwise3(w, most, f), rp = pairwise3(w, most, r);
            if (rp) flags |= 1u << k;
            paired |= fp;
            directed |= (f && !fp) || (r && !rp);
        }
        if (paired) flags |= LF3_FWD;
        if (directed) {
            flags |= LF3_OWN;
            mine = (n + 31) / 32;
            at = atomicAdd(&ndir, mine);
        }
        w.flags[b] = flags;
    }
    __syncthreads();
    if (threadIdx.x < C3_CLASSES) {
        uint32_t first = 0;
        for (int i = 0; i < int(threadIdx.x); ++i) first += w.ctrl[C3_COUNT + i];
        const uint32_t h = hist[threadIdx.x];
        base[threadIdx.x] = first + (h ? atomicAdd(w.ctrl + C3_PLACED + threadIdx.x, h) : 0u);
        hist[threadIdx.x] = 0;
    } else if (threadIdx.x == C3_CLASSES && ndir) {
        dbase = atomicAdd(w.ctrl + C3_DIRECTED, ndir);
    }
    __syncthreads();
    for (uint32_t i = 0; i < mine; ++i)
        w.directed[dbase + at + i] = make_uint2(uint32_t(b), s0 + 32 * i);
    if (big)
        leaf_items3<MAX>(
            start, L, uint32_t(b), n, w.pmin,
            [&](int c, int g) {
                w.items[base[c] + atomicAdd(&hist[c], 1u)] =
                    make_uint2(uint32_t(b), paired ? uint32_t(g) : NO_GROUP3);
            },
            [](uint64_t) {});
}

// 1/sqrt(x) for a normal x > 0: the PTX approximate reciprocal square root
// with denormal inputs flushed (none reach it: the pairs of two adjacent
// leaves have |d|^2 >= 2^-48).
__device__ __forceinline__ float rsqrt_normal(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A lane's 2 TP targets, two to a float2 (packed FP32 instructions).
template <int TP> struct Tgt3 {
    float2 x[TP], y[TP], z[TP], q[TP];      // places, charges
    float2 f[TP], gx[TP], gy[TP], gz[TP];   // sums
};
struct Src3 {
    float nx, ny, nz, q;      // minus the place (in the targets' frame), charge
    float f, gx, gy, gz;      // sums of the reactions (field: of its negative)
};

template <int TP> __device__ __forceinline__ void clear3(Tgt3<TP> &t) {
#pragma unroll
    for (int i = 0; i < TP; ++i) t.f[i] = t.gx[i] = t.gy[i] = t.gz[i] = make_float2(0.f, 0.f);
}

// One source against the lane's targets, both ways.  The differences are
// scalar: packed ones would need the source's coordinates twice in a register
// pair each, as many instructions again.
template <int TP> __device__ __forceinline__ void pair3(Tgt3<TP> &t, Src3 &s) {
    const float2 q = make_float2(s.q, s.q);
#pragma unroll
    for (int i = 0; i < TP; ++i) {
        const float2 dx = make_float2(t.x[i].x + s.nx, t.x[i].y + s.nx);
        const float2 dy = make_float2(t.y[i].x + s.ny, t.y[i].y + s.ny);
        const float2 dz = make_float2(t.z[i].x + s.nz, t.z[i].y + s.nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 ri = make_float2(rsqrt_normal(r2.x), rsqrt_normal(r2.y));
        const float2 r3 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
        t.f[i] = __ffma2_rn(q, ri, t.f[i]);
        s.f = fmaf(t.q[i].x, ri.x, s.f);
        s.f = fmaf(t.q[i].y, ri.y, s.f);
        const float2 a = __fmul2_rn(q, r3), c = __fmul2_rn(t.q[i], r3);
        t.gx[i] = __ffma2_rn(a, dx, t.gx[i]);
        t.gy[i] = __ffma2_rn(a, dy, t.gy[i]);
        t.gz[i] = __ffma2_rn(a, dz, t.gz[i]);
        s.gx = fmaf(c.x, dx.x, s.gx);
        s.gx = fmaf(c.y, dx.y, s.gx);
        s.gy = fmaf(c.x, dy.x, s.gy);
        s.gy = fmaf(c.y, dy.y, s.gy);
        s.gz = fmaf(c.x, dz.x, s.gz);
        s.gz = fmaf(c.y, dz.y, s.gz);
    }
}

// One source of the targets' own leaf, one way; self and coincident charges
// (|d| = 0) add nothing.
template <int TP> __device__ __forceinline__ void own3(Tgt3<TP> &t, const float4 s) {
    const float2 nx = make_float2(-s.x, -s.x), ny = make_float2(-s.y, -s.y),
                 nz = make_float2(-s.z, -s.z), q = make_float2(s.w, s.w);
#pragma unroll
    for (int i = 0; i < TP; ++i) {
        const float2 dx = __fadd2_rn(t.x[i], nx), dy = __fadd2_rn(t.y[i], ny),
                     dz = __fadd2_rn(t.z[i], nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 ri = make_float2(r2.x > 0.f ? rsqrtf(r2.x) : 0.f, r2.y > 0.f ? rsqrtf(r2.y) : 0.f);
        const float2 a = __fmul2_rn(q, ri), a3 = __fmul2_rn(a, __fmul2_rn(ri, ri));
        t.f[i] = __fadd2_rn(t.f[i], a);
        t.gx[i] = __ffma2_rn(a3, dx, t.gx[i]);
        t.gy[i] = __ffma2_rn(a3, dy, t.gy[i]);
        t.gz[i] = __ffma2_rn(a3, dz, t.gz[i]);
    }
}

// Sums v[0..3] over the lane's group of W = 16 or 32 lanes: every lane gets
// sum (lane mod W) / (W / 4).
template <int W>
__device__ __forceinline__ float sum4_3(float v0, float v1, float v2, float v3, int lane) {
    const bool h = lane & (W / 2);
    float a = (h ? v2 : v0) + __shfl_xor_sync(0xffffffffu, h ? v0 : v2, W / 2);
    const float b = (h ? v3 : v1) + __shfl_xor_sync(0xffffffffu, h ? v1 : v3, W / 2);
    const bool k = lane & (W / 4);
    a = (k ? b : a) + __shfl_xor_sync(0xffffffffu, k ? a : b, W / 4);
#pragma unroll
    for (int o = W / 8; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

constexpr float FAR3 = 64.f;   // a place no charge is near (leaf widths)
// sources left over after whole chunks of 32: up to this many one by one
constexpr int P3_REST = 16;

// A run of up to 64 targets of leaf A (t0 .. t1 of its sorted charges from
// a0) against the group's forward neighbours.  Both half-warps hold all the
// targets, four a lane, and 16 of the neighbour's charges each, which travel
// around the half by shuffles, the reaction on each accumulating as it
// travels: after 16 steps each has met every target and is home.  (With two
// targets a lane and whole-warp rings the eight shuffles of a step were a
// quarter of its instructions.)  first: the reactions are stored, else added
// to those of A's earlier runs (the same warp's).
__device__ __forceinline__ void pairs_run3(const Near3 &w, uint32_t most, int L,
                                           const uint32_t *__restrict__ start,
                                           const float4 *__restrict__ rec, uint32_t leaf, int g,
                                           uint32_t t0, uint32_t t1, bool first, int lane) {
    const int side = 1 << L;
    const int ix = int(compact3(leaf)), iy = int(compact3(leaf >> 1)), iz = int(compact3(leaf >> 2));
    const uint32_t a0 = start[leaf], a1 = start[leaf + 1];
    const uint32_t half = uint32_t(lane) >> 4, l = uint32_t(lane) & 15u;
    Tgt3<2> t;
    clear3(t);
    float4 r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t u = t0 + 16 * i + l;
        r[i] = u < t1 ? rec[u] : make_float4(FAR3, FAR3, FAR3, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        t.x[i] = make_float2(r[2 * i].x, r[2 * i + 1].x);
        t.y[i] = make_float2(r[2 * i].y, r[2 * i + 1].y);
        t.z[i] = make_float2(r[2 * i].z, r[2 * i + 1].z);
        t.q[i] = make_float2(r[2 * i].w, r[2 * i + 1].w);
    }
    if (g == 0 && pairwise3(w, most, a1 - a0))
#pragma unroll 2
        for (uint32_t j = a0 + half; j < a1; j += 2) own3(t, rec[j]);
    const int groups = groups3(a1 - a0);
    for (int k = group_first3(g, groups); k < group_first3(g + 1, groups); ++k) {
        int dx, dy, dz;
        fwd3(k, &dx, &dy, &dz);
        const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
        if (nx < 0 || ny < 0 || nz < 0 || nx >= side || ny >= side || nz >= side) continue;
        const uint32_t nb = morton3(uint32_t(nx), uint32_t(ny), uint32_t(nz));
        const uint32_t b0 = start[nb], b1 = start[nb + 1];
        if (!pairwise3(w, most, b1 - b0)) continue;
        float4 *out = w.slots + int64_t(P3_DIRS + k) * w.n;
        const float ox = float(dx), oy = float(dy), oz = float(dz);
        uint32_t c = b0;
        Src3 s;
        auto load = [&](uint32_t j) {
            const float4 u = j < b1 ? rec[j] : make_float4(-FAR3, -FAR3, -FAR3, 0.f);
            s.nx = -(u.x + ox);
            s.ny = -(u.y + oy);
            s.nz = -(u.z + oz);
            s.q = u.w;
            s.f = s.gx = s.gy = s.gz = 0.f;
        };
        for (; c + uint32_t(P3_REST) < b1; c += 32) {
            const uint32_t j = c + uint32_t(lane);
            load(j);
            const int from = (lane & 16) | ((lane + 1) & 15);
#pragma unroll
            for (int step = 0; step < 16; ++step) {
                // the next step's source on its way while this one computes
                const float nx2 = __shfl_sync(0xffffffffu, s.nx, from);
                const float ny2 = __shfl_sync(0xffffffffu, s.ny, from);
                const float nz2 = __shfl_sync(0xffffffffu, s.nz, from);
                const float q2 = __shfl_sync(0xffffffffu, s.q, from);
                pair3(t, s);
                s.f = __shfl_sync(0xffffffffu, s.f, from);
                s.gx = __shfl_sync(0xffffffffu, s.gx, from);
                s.gy = __shfl_sync(0xffffffffu, s.gy, from);
                s.gz = __shfl_sync(0xffffffffu, s.gz, from);
                s.nx = nx2;
                s.ny = ny2;
                s.nz = nz2;
                s.q = q2;
            }
            if (j < b1) {
                float4 o = make_float4(s.f, -s.gx, -s.gy, -s.gz);
                if (!first) {
                    const float4 p = out[j];
                    o = make_float4(p.x + o.x, p.y + o.y, p.z + o.z, p.w + o.w);
                }
                out[j] = o;
            }
        }
        for (; c < b1; c += 2) {  // the rest one by one, a half-warp each
            const uint32_t j = c + half;
            load(j);
            pair3(t, s);
            const float v = sum4_3<16>(s.f, -s.gx, -s.gy, -s.gz, lane);
            if ((lane & 3) == 0 && j < b1) {
                float *o = reinterpret_cast<float *>(out + j) + (l >> 2);
                *o = first ? v : *o + v;
            }
        }
        __syncwarp();  // a later run of this warp reads what other lanes wrote
    }
    // the halves' sums; half h writes targets 32 h ..
    float4 *own = w.slots + int64_t(g) * w.n;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        t.f[i].x += __shfl_xor_sync(0xffffffffu, t.f[i].x, 16);
        t.f[i].y += __shfl_xor_sync(0xffffffffu, t.f[i].y, 16);
        t.gx[i].x += __shfl_xor_sync(0xffffffffu, t.gx[i].x, 16);
        t.gx[i].y += __shfl_xor_sync(0xffffffffu, t.gx[i].y, 16);
        t.gy[i].x += __shfl_xor_sync(0xffffffffu, t.gy[i].x, 16);
        t.gy[i].y += __shfl_xor_sync(0xffffffffu, t.gy[i].y, 16);
        t.gz[i].x += __shfl_xor_sync(0xffffffffu, t.gz[i].x, 16);
        t.gz[i].y += __shfl_xor_sync(0xffffffffu, t.gz[i].y, 16);
        if (int(half) != i) continue;
        const uint32_t u = t0 + 32 * i + l, v = u + 16;
        if (u < t1) own[u] = make_float4(t.f[i].x, t.gx[i].x, t.gy[i].x, t.gz[i].x);
        if (v < t1) own[v] = make_float4(t.f[i].y, t.gx[i].y, t.gy[i].y, t.gz[i].y);
    }
}

// The targets left over after whole runs (up to 16), four at a time: the
// lanes hold the neighbours' charges, so that no lane idles for want of
// targets; the reactions are added to those of the leaf's first run.
__device__ __forceinline__ void pairs_rest3(const Near3 &w, uint32_t most, int L,
                                            const uint32_t *__restrict__ start,
                                            const float4 *__restrict__ rec, uint32_t leaf, int g,
                                            uint32_t t0, uint32_t t1, int lane) {
    const int side = 1 << L;
    const int ix = int(compact3(leaf)), iy = int(compact3(leaf >> 1)), iz = int(compact3(leaf >> 2));
    const uint32_t a0 = start[leaf], a1 = start[leaf + 1];
    const int groups = groups3(a1 - a0);
    for (uint32_t c = t0; c < t1; c += 4) {
        Tgt3<2> t;
        clear3(t);
        float4 r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            r[i] = c + i < t1 ? rec[c + i] : make_float4(FAR3, FAR3, FAR3, 0.f);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            t.x[i] = make_float2(r[2 * i].x, r[2 * i + 1].x);
            t.y[i] = make_float2(r[2 * i].y, r[2 * i + 1].y);
            t.z[i] = make_float2(r[2 * i].z, r[2 * i + 1].z);
            t.q[i] = make_float2(r[2 * i].w, r[2 * i + 1].w);
        }
        if (g == 0 && pairwise3(w, most, a1 - a0))
            for (uint32_t j = a0 + uint32_t(lane); j < a1; j += 32) own3(t, rec[j]);
        for (int k = group_first3(g, groups); k < group_first3(g + 1, groups); ++k) {
            int dx, dy, dz;
            fwd3(k, &dx, &dy, &dz);
            const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
            if (nx < 0 || ny < 0 || nz < 0 || nx >= side || ny >= side || nz >= side) continue;
            const uint32_t nb = morton3(uint32_t(nx), uint32_t(ny), uint32_t(nz));
            const uint32_t b0 = start[nb], b1 = start[nb + 1];
            if (!pairwise3(w, most, b1 - b0)) continue;
            float4 *out = w.slots + int64_t(P3_DIRS + k) * w.n;
            for (uint32_t j = b0 + uint32_t(lane); j < b1; j += 32) {
                const float4 u = rec[j], p = out[j];
                Src3 s;
                s.nx = -(u.x + float(dx));
                s.ny = -(u.y + float(dy));
                s.nz = -(u.z + float(dz));
                s.q = u.w;
                s.f = s.gx = s.gy = s.gz = 0.f;
                pair3(t, s);
                out[j] = make_float4(p.x + s.f, p.y - s.gx, p.z - s.gy, p.w - s.gz);
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = t.f[i / 2], x = t.gx[i / 2], y = t.gy[i / 2], z = t.gz[i / 2];
            const float v = i & 1 ? sum4_3<32>(f.y, x.y, y.y, z.y, lane)
                                  : sum4_3<32>(f.x, x.x, y.x, z.x, lane);
            if ((lane & 7) == 0 && c + i < t1)
                reinterpret_cast<float *>(w.slots + int64_t(g) * w.n + c + i)[lane >> 3] = v;
        }
    }
}

// Bound by the FP32 pipe (65 % busy, issue slots 64 %; a packed instruction
// holds the pipe two cycles): per target 18 operations, of which 11 packed, and
// 2 of a step's 8 shuffles; 23.3 instructions a pair in all.  Both near fields
// whole, on one GB300 (one-sided before / now):
//   2 M uniform charges (61 a leaf)           2.19 / 1.77 ms
//   2 M clustered charges (up to 600 a leaf)  11.2 / 8.6 ms
// Sweeps on the same two: 16 steps unrolled 1.77 / 8.56, by two 1.80 / 8.78;
// registers for 5, 6, 7 and 8 blocks an SM (steps by two) 1.80 / 8.71,
// 1.81 / 8.85, 1.80 / 8.77, 1.86 / 9.14; all scalar 1.83 / 8.76 at best; the
// reactions summed apart from the travelling sums 1.79 / 8.76.
__global__ void __launch_bounds__(128, 6) k3_pairs(int L, const uint32_t *__restrict__ start,
                                                const float4 *__restrict__ rec, const Near3 w) {
    const int lane = threadIdx.x & 31;
    const uint32_t it = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (it >= w.ctrl[C3_PAIRS]) return;
    const uint2 item = w.items[it];
    if (item.y == NO_GROUP3) return;
    const uint32_t leaf = item.x;
    if (!PF_IN(leaf, int64_t(1) << (3 * L))) return;
    const int g = int(item.y);
    const uint32_t a0 = start[leaf], a1 = start[leaf + 1];
    const uint32_t most = most3(w, a1 - a0);
    bool first = true;
    for (uint32_t t = a0; t < a1;) {
        const uint32_t left = a1 - t;
        if (left <= 16 && !first) {
            pairs_rest3(w, most, L, start, rec, leaf, g, t, a1, lane);
            break;
        }
        pairs_run3(w, most, L, start, rec, leaf, g, t, min(a1, t + 64), first, lane);
        t += 64;
        first = false;
    }
}

// The leaf pairs not evaluated pairwise, one way: a warp per work item (up to
// 32 targets of one leaf).  An item of k targets gives each target a group of
// rep lanes, rep the largest power of two with k rep <= 32, lane c of a group
// taking sources c, c + rep, ... of every range (a leaf's last, partly filled
// item keeps most lanes busy), the group's partial sums added by shuffles.
// Sources of the leaf and its neighbours in a fixed order (dz, dy, dx, then
// sorted rank), each read once per lane group (one address per group) in
// FP32 leaf units: d = xi_t - (xi_s + offset), 1/|d| from rsqrt, self and
// coincident pairs (|d| = 0, own leaf only: the records are capped below
// 0.5 - 2^-24) skipped.
__global__ void __launch_bounds__(W3 * 32, 4) k3_near_directed(int L,
                                                               const uint32_t *__restrict__ start,
                                                               const float4 *__restrict__ rec,
                                                               const Near3 w) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t it = int64_t(blockIdx.x) * W3 + wid;
    if (it >= int64_t(w.ctrl[C3_DIRECTED])) return;
    // one item: the targets s0 .. s1 - 1 of leaf b
    const uint2 item = w.directed[it];
    const int64_t b = item.x;
    if (!PF_IN(b, int64_t(1) << (3 * L))) return;
    const uint32_t s0 = item.y;
    const uint32_t nme = start[b + 1] - start[b];
    const uint32_t most = most3(w, nme);
    const uint32_t s1 = min(start[b + 1], s0 + 32u);
    const int k = int(s1 - s0);  // 1..32 (an item holds at least one target)
    int lg = 0;
    while (lg < 5 && (k << (lg + 1)) <= 32) ++lg;
    const uint32_t rep = 1u << lg, c = uint32_t(lane) & (rep - 1u);
    const uint32_t i = s0 + uint32_t(lane >> lg);
    const bool live = i < s1;
    const int ix = int(compact3(uint32_t(b))), iy = int(compact3(uint32_t(b) >> 1)),
              iz = int(compact3(uint32_t(b) >> 2));
    const int side = 1 << L;
    const float4 tg = live ? rec[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    float f = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
                if (nx < 0 || ny < 0 || nz < 0 || nx >= side || ny >= side || nz >= side)
                    continue;
                const uint32_t nb = morton3(uint32_t(nx), uint32_t(ny), uint32_t(nz));
                const uint32_t a = start[nb], e = start[nb + 1];
                if (pairwise3(w, most, e - a)) continue;
                const float ox = tg.x - float(dx), oy = tg.y - float(dy), oz = tg.z - float(dz);
                // |d| = 0 only within the target's own leaf (self, and
                // coincident particles, which bin to the same leaf); the
                // record cap keeps it from pairs across a leaf face
                auto pair = [&](const float4 sr, bool guard) {
                    const float ddx = ox - sr.x, ddy = oy - sr.y, ddz = oz - sr.z;
                    const float r2 = fmaf(ddx, ddx, fmaf(ddy, ddy, ddz * ddz));
                    float ri = guard ? rsqrtf(r2) : rsqrt_normal(r2);
                    if (guard) ri = r2 > 0.f ? ri : 0.f;
                    const float qr = sr.w * ri;
                    const float qr3 = qr * ri * ri;
                    f += qr;
                    gx = fmaf(qr3, ddx, gx);
                    gy = fmaf(qr3, ddy, gy);
                    gz = fmaf(qr3, ddz, gz);
                };
                // full items (rep = 1) on the plain loop (the strided one
                // measured slower there), both unrolled eight / two deep
                const bool own = dx == 0 && dy == 0 && dz == 0;
                if (rep == 1u) {
                    if (own)
                        for (uint32_t j = a; j < e; ++j) pair(rec[j], true);
                    else {
#pragma unroll 8
                        for (uint32_t j = a; j < e; ++j) pair(rec[j], false);
                    }
                } else {
                    const float4 *sp = rec + a + c, *se = rec + e;
                    if (own)
                        for (; sp < se; sp += rep) pair(*sp, true);
                    else {
#pragma unroll 2
                        for (; sp < se; sp += rep) pair(*sp, false);
                    }
                }
            }
    for (uint32_t o = 1; o < rep; o <<= 1) {
        f += __shfl_xor_sync(0xffffffffu, f, int(o));
        gx += __shfl_xor_sync(0xffffffffu, gx, int(o));
        gy += __shfl_xor_sync(0xffffffffu, gy, int(o));
        gz += __shfl_xor_sync(0xffffffffu, gz, int(o));
    }
    if (c == 0 && live) w.own[i] = make_float4(f, gx, gy, gz);
}

// The parts of each charge and L2P, in the caller's order.
template <typename TOut>
__global__ void __launch_bounds__(256) k3_near_final(int L, int p, double w,
                                                     const uint32_t *__restrict__ skeys,
                                                     const uint32_t *__restrict__ start,
                                                     const float4 *__restrict__ rec,
                                                     const float2 *__restrict__ le,
                                                     const uint32_t *__restrict__ perm,
                                                     const Near3 nr, void *phi, void *ex, void *ey,
                                                     void *ez) {
    const int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x;
    if (i >= nr.n) return;
    const uint32_t b = skeys[i];
    if (!PF_IN(b, int64_t(1) << (3 * L))) return;
    const uint32_t flags = nr.flags[b];
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](const float4 v) {
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
    };
    if (flags & LF3_OWN) add(nr.own[i]);
    if (flags & LF3_FWD) {
        const int groups = groups3(start[b + 1] - start[b]);
        for (int g = 0; g < groups; ++g) add(nr.slots[int64_t(g) * nr.n + i]);
    }
#pragma unroll
    for (int k = 0; k < P3_DIRS; ++k)
        if ((flags >> k) & 1u) add(nr.slots[int64_t(P3_DIRS + k) * nr.n + i]);
    float ff = 0.f, fx = 0.f, fy = 0.f, fz = 0.f;
    if (L >= 2) {
        const float4 r = rec[i];
        l2p3<float, float2>(le + (lvl_off3(L) + int64_t(b)) * nc3(p), p, r.x, r.y, r.z, ff, fx, fy, fz);
    }
    const float inv_w = float(1.0 / w), inv_w2 = float(1.0 / (w * w));
    const int64_t o = perm[i];
    if (!PF_IN(o, nr.n)) return;
    store3<TOut>(phi, o, double((s.x + ff) * inv_w));
    store3<TOut>(ex, o, double((s.y - fx) * inv_w2));
    store3<TOut>(ey, o, double((s.z - fy) * inv_w2));
    store3<TOut>(ez, o, double((s.w - fz) * inv_w2));
}

// 1/sqrt(x): the hardware's approximation y and one step of Householder's
// third-order iteration, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y^2
// (|e| < 2^-18 leaves |e|^3 below 2^-54; within 1.5 ulp,
// tests/test_gpu_factors.py): five FP64 operations, where a
// division by sqrt took about thirty.  Subnormal, infinite and NaN x (the
// approximation flushes or saturates there) by division.
__device__ __forceinline__ double rsqrt_f64(double x) {
    const uint32_t h = uint32_t(__double2hiint(x));
    if (h - 0x00100000u >= 0x7fe00000u) return 1.0 / sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

__global__ void __launch_bounds__(256) k3_rsqrt64(const double *__restrict__ x,
                                                  double *__restrict__ y, int64_t n) {
    const int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x;
    if (i < n) y[i] = rsqrt_f64(x[i]);
}

// The FP64 path's leaf pairs not evaluated pairwise: global coordinates; work
// items, and lanes shared out over an item's few targets, as in the mixed
// kernel.  Bound by the FP64 pipe (two lanes a cycle and SM): 18 operations a
// pair.  Measured with every leaf pair (one GB300, 262,144 uniform charges, L =
// 4): 32.9 ms with a division and a square root per pair and a warp per leaf ->
// 16.6 ms.
__global__ void __launch_bounds__(W3 * 32) k3_near_directed64(int L,
                                                              const uint32_t *__restrict__ start,
                                                              const Dbl4 *__restrict__ xs,
                                                              const Near3 w,
                                                              Dbl4 *__restrict__ own) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t it = int64_t(blockIdx.x) * W3 + wid;
    if (it >= int64_t(w.ctrl[C3_DIRECTED])) return;
    // one item: the targets s0 .. s1 - 1 of leaf b, rep lanes each
    const uint2 item = w.directed[it];
    const int64_t b = item.x;
    if (!PF_IN(b, int64_t(1) << (3 * L))) return;
    const uint32_t nme = start[b + 1] - start[b];
    const uint32_t most = most3(w, nme);
    const uint32_t s0 = item.y, s1 = min(start[b + 1], s0 + 32u);
    const int k = int(s1 - s0);
    int lg = 0;
    while (lg < 5 && (k << (lg + 1)) <= 32) ++lg;
    const uint32_t rep = 1u << lg, c = uint32_t(lane) & (rep - 1u);
    const uint32_t i = s0 + uint32_t(lane >> lg);
    const bool live = i < s1;
    const int ix = int(compact3(uint32_t(b))), iy = int(compact3(uint32_t(b) >> 1)),
              iz = int(compact3(uint32_t(b) >> 2));
    const int side = 1 << L;
    const Dbl4 tg = xs[live ? i : s0];
    double f = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
                if (nx < 0 || ny < 0 || nz < 0 || nx >= side || ny >= side || nz >= side)
                    continue;
                const uint32_t nb = morton3(uint32_t(nx), uint32_t(ny), uint32_t(nz));
                const uint32_t a = start[nb], e = start[nb + 1];
                if (pairwise3(w, most, e - a)) continue;
#pragma unroll 2
                for (uint32_t j = a + c; j < e; j += rep) {
                    const Dbl4 s = xs[j];
                    const double ddx = tg.x - s.x, ddy = tg.y - s.y, ddz = tg.z - s.z;
                    const double r2 = fma(ddx, ddx, fma(ddy, ddy, ddz * ddz));
                    // self and coincident pairs (r2 = 0, tested on the bits)
                    const bool pair = (__double2hiint(r2) | __double2loint(r2)) != 0;
                    const double ri = pair ? rsqrt_f64(r2) : 0.0;
                    const double q = pair ? s.w : 0.0;  // (an infinite charge adds 0 to itself)
                    const double qr = q * ri, qr3 = qr * (ri * ri);
                    f = fma(q, ri, f);
                    gx = fma(qr3, ddx, gx);
                    gy = fma(qr3, ddy, gy);
                    gz = fma(qr3, ddz, gz);
                }
            }
    for (uint32_t o = 1; o < rep; o <<= 1) {
        f += __shfl_xor_sync(0xffffffffu, f, int(o));
        gx += __shfl_xor_sync(0xffffffffu, gx, int(o));
        gy += __shfl_xor_sync(0xffffffffu, gy, int(o));
        gz += __shfl_xor_sync(0xffffffffu, gz, int(o));
    }
    if (c == 0 && live) own[i] = Dbl4{f, gx, gy, gz};
}

// ---------------------------------------------------------------------------
// FP64 near field, pairwise: a warp per pair item (leaf A, group of forward
// directions, as k3_near_items lists them with pmin = 1; the leaf pairs above
// limit left out).  The charges of the group's neighbours, and of A itself in
// one group, form one list; each lane
// takes one of 32 and keeps its reaction in registers while A's targets pass
// by: lane l meets target (l + step) mod 32 of a run of 32, so that the sums of
// the targets, in shared memory, have one writer a step.  A last run of c < 32
// targets is shared by groups of c lanes, each with its own copy of the sums,
// and no lane idles for want of targets.  Targets go 128 at a time (the
// reactions of later passes are added to those of the first).
// Bound by the FP64 pipe (two lanes a cycle and SM): 24 operations a pair for
// both charges, where the one-sided sums take 18 for each; loads, shuffles and
// selects cost nothing beside it.
// The near field whole, one GB300, one-sided / now: 262,144 uniform charges, 64
// a leaf, 16.4 / 9.7 ms (the pipe busy throughout); 8 a leaf, 6.2 / 2.3 ms;
// 200,000 clustered charges, up to 760 a leaf, 61.2 / 41.1 ms (47 with the leaf
// itself in its first group, 58 with 24 warps an SM instead of 8 besides).
constexpr int PW64 = 2;               // warps a block
constexpr int PT64 = 128;             // targets of a pass
constexpr int PA64 = PT64 + 32;       // sums of a pass, copies of the last run's among them
// Shared memory asked for per block, so that no more than four are resident:
// two warps a scheduler keep the pipe busy, and with more the heaviest items
// all start at once and the schedulers that got them end last.
constexpr size_t kPairs64Smem = 56 * 1024;

// f, gx, gy, gz of target and source: one pair, both ways (d = target -
// source); self, coincident and padding pairs add nothing.
__device__ __forceinline__ void pair64(const Dbl4 &t, const Dbl4 &s, bool live, Dbl4 &ta, Dbl4 &sa) {
    const double dx = t.x - s.x, dy = t.y - s.y, dz = t.z - s.z;
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const bool pair = live && (__double2hiint(r2) | __double2loint(r2)) != 0;
    const double ri = pair ? rsqrt_f64(r2) : 0.0;
    const double qs = pair ? s.w : 0.0, qt = pair ? t.w : 0.0;
    const double r3 = ri * ri * ri, a = qs * r3, c = qt * r3;
    ta.x = fma(qs, ri, ta.x);
    ta.y = fma(a, dx, ta.y);
    ta.z = fma(a, dy, ta.z);
    ta.w = fma(a, dz, ta.w);
    sa.x = fma(qt, ri, sa.x);
    sa.y = fma(-c, dx, sa.y);
    sa.z = fma(-c, dy, sa.z);
    sa.w = fma(-c, dz, sa.w);
}

__global__ void __launch_bounds__(PW64 * 32) k3_pairs_f64(int L, const uint32_t *__restrict__ start,
                                                    const Dbl4 *__restrict__ xs, const Near3 w,
                                                    Dbl4 *__restrict__ slots) {
    __shared__ Dbl4 stgt[PW64][PT64], sacc[PW64][PA64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t it = blockIdx.x * PW64 + wid;
    if (it >= w.ctrl[C3_PAIRS]) return;
    const uint2 item = w.items[it];
    if (item.y == NO_GROUP3) return;
    const uint32_t leaf = item.x;
    if (!PF_IN(leaf, int64_t(1) << (3 * L))) return;
    const int g = int(item.y), side = 1 << L;
    const int ix = int(compact3(leaf)), iy = int(compact3(leaf >> 1)), iz = int(compact3(leaf >> 2));
    const uint32_t a0 = start[leaf], a1 = start[leaf + 1];
    const int groups = groups3<P3_GROUPS64>(a1 - a0);
    const int k0 = group_first3(g, groups), nk = group_first3(g + 1, groups) - k0;
    Dbl4 *tgt = stgt[wid], *acc = sacc[wid];
    const uint32_t most = most3(w, a1 - a0);
    // lane 0: the leaf itself (its group only); lane 1 + i: forward direction k0 + i
    uint32_t beg = 0, cnt = 0;
    if (lane == 0 && g == own_group3(groups)) {
        beg = a0;
        cnt = a1 - a0;
    } else if (lane >= 1 && lane <= nk) {
        int dx, dy, dz;
        fwd3(k0 + lane - 1, &dx, &dy, &dz);
        const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
        if (nx >= 0 && ny >= 0 && nz >= 0 && nx < side && ny < side && nz < side) {
            const uint32_t nb = morton3(uint32_t(nx), uint32_t(ny), uint32_t(nz));
            beg = start[nb];
            cnt = start[nb + 1] - beg;
        }
    }
    if (!pairwise3(w, most, cnt)) cnt = 0;
    uint32_t end = cnt;  // of the lane's range in the list
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += v;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, end, 31);
    for (uint32_t t0 = a0; t0 < a1; t0 += PT64) {
        const uint32_t nt = min(a1 - t0, uint32_t(PT64)), whole = nt & ~31u, c = nt & 31u;
        for (uint32_t i = lane; i < nt; i += 32) tgt[i] = xs[t0 + i];
        for (uint32_t i = lane; i < PA64; i += 32) acc[i] = Dbl4{0.0, 0.0, 0.0, 0.0};
        __syncwarp();
        for (uint32_t m0 = 0; m0 < total; m0 += 32) {
            const uint32_t m = m0 + uint32_t(lane);
            const bool live = m < total;
            int r = 0;  // the range that holds entry m
            for (int i = 0; i <= nk; ++i) r += m >= __shfl_sync(0xffffffffu, end, i);
            r = min(r, nk);
            const uint32_t j = __shfl_sync(0xffffffffu, beg + cnt - end, r) + m;
            const Dbl4 s = live ? xs[j] : tgt[0];
            Dbl4 sa{0.0, 0.0, 0.0, 0.0};
            for (uint32_t b = 0; b < whole; b += 32)
                for (uint32_t st = 0; st < 32; ++st) {
                    const uint32_t i = b + ((uint32_t(lane) + st) & 31u);
                    Dbl4 ta = acc[i];
                    pair64(tgt[i], s, live, ta, sa);
                    acc[i] = ta;
                    __syncwarp();
                }
            if (c) {
                const uint32_t copy = uint32_t(lane) / c * c;
                uint32_t i = uint32_t(lane) - copy;
                for (uint32_t st = 0; st < c; ++st) {
                    Dbl4 ta = acc[whole + copy + i];
                    pair64(tgt[whole + i], s, live, ta, sa);
                    acc[whole + copy + i] = ta;
                    __syncwarp();
                    i = i + 1 == c ? 0 : i + 1;
                }
            }
            if (live && r > 0 && PF_IN(j, w.n)) {
                Dbl4 *o = slots + int64_t(P3_GROUPS64 + k0 + r - 1) * w.n + j;
                if (t0 != a0) {
                    const Dbl4 p = *o;
                    sa = Dbl4{p.x + sa.x, p.y + sa.y, p.z + sa.z, p.w + sa.w};
                }
                *o = sa;
            }
        }
        for (uint32_t i = lane; i < nt; i += 32) {
            Dbl4 v = acc[i];
            if (i >= whole)
                for (uint32_t o = c; o < 32; o += c) {
                    const Dbl4 u = acc[i + o];
                    v = Dbl4{v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w};
                }
            slots[int64_t(g) * w.n + t0 + i] = v;
        }
        __syncwarp();
    }
}

// The parts of each charge and L2P, in the caller's order.
template <typename TOut>
__global__ void __launch_bounds__(128) k3_final_f64(int L, int p, Dom3 d,
                                                    const uint32_t *__restrict__ skeys,
                                                    const uint32_t *__restrict__ start,
                                                    const Dbl4 *__restrict__ xs,
                                                    const double2 *__restrict__ le,
                                                    const uint32_t *__restrict__ perm,
                                                    const Near3 nr, const Dbl4 *__restrict__ slots,
                                                    const Dbl4 *__restrict__ own, void *phi,
                                                    void *ex, void *ey, void *ez) {
    const int64_t i = int64_t(blockIdx.x) * 128 + threadIdx.x;
    if (i >= nr.n) return;
    const uint32_t b = skeys[i];
    if (!PF_IN(b, int64_t(1) << (3 * L))) return;
    const uint32_t flags = nr.flags[b];
    Dbl4 s{0.0, 0.0, 0.0, 0.0};
    auto add = [&](const Dbl4 v) {
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
    };
    if (flags & LF3_OWN) add(own[i]);
    if (flags & LF3_FWD) {
        const int groups = groups3<P3_GROUPS64>(start[b + 1] - start[b]);
        for (int g = 0; g < groups; ++g) add(slots[int64_t(g) * nr.n + i]);
    }
#pragma unroll
    for (int k = 0; k < P3_DIRS; ++k)
        if ((flags >> k) & 1u) add(slots[int64_t(P3_GROUPS64 + k) * nr.n + i]);
    const double w = d.width / double(1 << L);
    double ff = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
    if (L >= 2) {
        const double cx = d.x0 + (int(compact3(b)) + 0.5) * w,
                     cy = d.y0 + (int(compact3(b >> 1)) + 0.5) * w,
                     cz = d.z0 + (int(compact3(b >> 2)) + 0.5) * w;
        const Dbl4 t = xs[i];
        l2p3<double, double2>(le + (lvl_off3(L) + int64_t(b)) * nc3(p), p, (t.x - cx) / w,
                              (t.y - cy) / w, (t.z - cz) / w, ff, fx, fy, fz);
    }
    const int64_t o = perm[i];
    if (!PF_IN(o, nr.n)) return;
    store3<TOut>(phi, o, s.x + ff / w);
    store3<TOut>(ex, o, s.y - fx / (w * w));
    store3<TOut>(ey, o, s.z - fy / (w * w));
    store3<TOut>(ez, o, s.w - fz / (w * w));
}

// ---------------------------------------------------------------------------
// Host: operator tables in FP64 from the same recurrences.
// ---------------------------------------------------------------------------
using cd = std::complex<double>;

// R_n^m(v), n < P, m >= 0: out[n (n + 1) / 2 + m]
void host_rec_r(double x, double y, double z, int P, cd *out) {
    const double r2 = x * x + y * y + z * z;
    cd rmm(1.0, 0.0);
    for (int m = 0; m < P; ++m) {
        if (m > 0) rmm *= cd(x, y) / double(2 * m);
        cd r1 = rmm, r0(0.0, 0.0);
        for (int n = m; n < P; ++n) {
            cd rn = r1;
            if (n > m) {
                rn = (double(2 * n - 1) * z * r1 - r2 * r0) / double(n * n - m * m);
                r0 = r1;
                r1 = rn;
            }
            out[n * (n + 1) / 2 + m] = rn;
        }
    }
}

// I_n^m(v), n < P, m >= 0
void host_rec_i(double x, double y, double z, int P, cd *out) {
    const double r2 = x * x + y * y + z * z;
    cd imm(1.0 / std::sqrt(r2), 0.0);
    for (int m = 0; m < P; ++m) {
        if (m > 0) imm *= double(2 * m - 1) * cd(x, y) / r2;
        cd i1 = imm, i0(0.0, 0.0);
        for (int n = m; n < P; ++n) {
            cd in = i1;
            if (n > m) {
                in = (double(2 * n - 1) * z * i1 - double((n - 1) * (n - 1) - m * m) * i0) / r2;
                i0 = i1;
                i1 = in;
            }
            out[n * (n + 1) / 2 + m] = in;
        }
    }
}

// The mixed path's M2L operator for one offset delta in the real basis of a
// real potential's degree-< p coefficients (real index r < p (p + 1) / 2: Re
// of coefficient r = n (n + 1) / 2 + m; r >= p (p + 1) / 2: Im of the
// coefficients with m > 0, in order), from the M2L sum written per stored
// (n, m >= 0) input: L~_k^l gets alpha M~_n^m + beta conj(M~_n^m) with
// alpha = (-1)^k I_{n+k}^{m+l}(delta) and, for m > 0, beta =
// (-1)^(k+m) I_{n+k}^{l-m}(delta) (the -m term).  iv: I_j^s(delta), j < 2p - 1,
// s >= 0; a[k_in * p^2 + r_out] = d(output r_out) / d(input k_in), FP64.
void host_m2l_real(int p, const cd *iv, double *a) {
    const int nc = p * (p + 1) / 2, nr = p * p;
    std::vector<int> imidx(size_t(nc), -1);
    for (int n = 0, r = nc; n < p; ++n)
        for (int m = 1; m <= n; ++m) imidx[size_t(n * (n + 1) / 2 + m)] = r++;
    auto ival = [&](int j, int sg) {  // I_j^sg from the stored s >= 0
        if (sg >= 0) return iv[j * (j + 1) / 2 + sg];
        const cd v = std::conj(iv[j * (j + 1) / 2 - sg]);
        return (sg & 1) ? -v : v;
    };
    std::fill(a, a + size_t(nr) * nr, 0.0);
    for (int k = 0; k < p; ++k)
        for (int lo = 0; lo <= k; ++lo) {
            const int jo = k * (k + 1) / 2 + lo;
            for (int n = 0; n < p; ++n)
                for (int m = 0; m <= n; ++m) {
                    const int ji = n * (n + 1) / 2 + m;
                    const double sk = (k & 1) ? -1.0 : 1.0;
                    const cd al = sk * ival(n + k, m + lo);
                    const cd be =
                        m > 0 ? sk * ((m & 1) ? -1.0 : 1.0) * ival(n + k, lo - m) : cd(0.0, 0.0);
                    // input a (real part): L += (al + be) a; input b (imaginary
                    // part): L += i (al - be) b
                    const cd vr = al + be, vi = cd(0.0, 1.0) * (al - be);
                    a[size_t(ji) * nr + jo] = vr.real();
                    if (lo > 0) a[size_t(ji) * nr + imidx[size_t(jo)]] = vr.imag();
                    if (m > 0) {
                        a[size_t(imidx[size_t(ji)]) * nr + jo] = vi.real();
                        if (lo > 0) a[size_t(imidx[size_t(ji)]) * nr + imidx[size_t(jo)]] = vi.imag();
                    }
                }
        }
}

// v rounded to TF32 (10 mantissa bits; to nearest, ties away from zero)
float host_tf32_rna(float v) {
    uint32_t bits;
    std::memcpy(&bits, &v, 4);
    if ((bits & 0x7F800000u) != 0x7F800000u) bits += 0x1000u;  // finite: round the magnitude
    bits &= 0xFFFFE000u;
    float r;
    std::memcpy(&r, &bits, 4);
    return r;
}

// Coefficient (n, m) of a stored m >= 0 series, m < 0 by symmetry.
cd host_coef(const cd *a, int n, int m) {
    if (m >= 0) return a[n * (n + 1) / 2 + m];
    const cd v = std::conj(a[n * (n + 1) / 2 - m]);
    return (m & 1) ? -v : v;
}

// The M2M sum for one child (rt: R_k^l of the child's offset) of a series mc
// whose only degree is n0: out_n^m = sum_l conj(R_k^l) M_{n0}^{m-l} 2^-n0,
// k = n - n0.
void host_m2m_one(int p, int n0, const cd *rt, const cd *mc, cd *out) {
    std::fill(out, out + p * (p + 1) / 2, cd(0.0, 0.0));
    for (int n = n0; n < p; ++n)
        for (int m = 0; m <= n; ++m) {
            const int k = n - n0;
            cd s(0.0, 0.0);
            for (int ll = std::max(-k, m - n0); ll <= std::min(k, m + n0); ++ll)
                s += std::conj(host_coef(rt, k, ll)) * host_coef(mc, n0, m - ll);
            out[n * (n + 1) / 2 + m] = s * std::ldexp(1.0, -n0);
        }
}

// The L2L sum for one child of a series lp whose only degree is n0:
// out_j^s = 2^-(j+1) sum_l conj(R_k^l) L_{n0}^{s+l}, k = n0 - j.
void host_l2l_one(int p, int n0, const cd *rt, const cd *lp, cd *out) {
    std::fill(out, out + p * (p + 1) / 2, cd(0.0, 0.0));
    for (int j = 0; j <= n0; ++j)
        for (int s = 0; s <= j; ++s) {
            const int k = n0 - j;
            cd acc(0.0, 0.0);
            for (int ll = std::max(-k, -n0 - s); ll <= std::min(k, n0 - s); ++ll)
                acc += std::conj(host_coef(rt, k, ll)) * host_coef(lp, n0, s + ll);
            out[j * (j + 1) / 2 + s] = acc * std::ldexp(1.0, -(j + 1));
        }
}

// The real p^2 x p^2 matrix of a map of real-potential series (the basis
// of host_m2l_real), by applying it to each basis vector:
// a[k_in * p^2 + r_out], FP64.
template <typename F> void host_real_matrix(int p, F apply, double *a) {
    const int nc = p * (p + 1) / 2, nr = p * p;
    // real index -> (coefficient, imaginary part?)
    std::vector<int> jof(static_cast<size_t>(nr)), imof(static_cast<size_t>(nr), 0);
    std::vector<int> nof(static_cast<size_t>(nr));  // its degree
    std::vector<int> imidx(size_t(nc), -1);
    for (int n = 0, r = nc; n < p; ++n)
        for (int m = 0; m <= n; ++m) {
            const int j = n * (n + 1) / 2 + m;
            jof[size_t(j)] = j;
            nof[size_t(j)] = n;
            if (m > 0) {
                imidx[size_t(j)] = r;
                jof[size_t(r)] = j;
                nof[size_t(r)] = n;
                imof[size_t(r++)] = 1;
            }
        }
    std::vector<cd> in(static_cast<size_t>(nc)), out(static_cast<size_t>(nc));
    for (int k = 0; k < nr; ++k) {
        std::fill(in.begin(), in.end(), cd(0.0, 0.0));
        in[size_t(jof[size_t(k)])] = imof[size_t(k)] ? cd(0.0, 1.0) : cd(1.0, 0.0);
        apply(nof[size_t(k)], in.data(), out.data());
        for (int j = 0; j < nc; ++j) {
            a[size_t(k) * nr + j] = out[size_t(j)].real();
            if (imidx[size_t(j)] >= 0) a[size_t(k) * nr + imidx[size_t(j)]] = out[size_t(j)].imag();
        }
    }
}

// The real M2M (kind 0: child of the octant -> parent) or L2L (kind 1:
// parent -> child of the octant) operator of order p, FP64.
void host_shift_real(int p, int kind, int octant, double *a) {
    std::vector<cd> ro(static_cast<size_t>(p * (p + 1) / 2));
    host_rec_r((octant & 1) ? 0.25 : -0.25, (octant & 2) ? 0.25 : -0.25,
               (octant & 4) ? 0.25 : -0.25, p, ro.data());
    if (kind == 0)
        host_real_matrix(p, [&](int n, const cd *in, cd *out) { host_m2m_one(p, n, ro.data(), in, out); }, a);
    else
        host_real_matrix(p, [&](int n, const cd *in, cd *out) { host_l2l_one(p, n, ro.data(), in, out); }, a);
}

// Default of PETFMM3D_OPT_PAIR_BYTES, the most bytes for the planes of the
// pairwise sums (67M charges of the mixed path, 32M of the FP64 path); above it,
// or where that memory cannot be had, leaf pairs are summed one-sided.
constexpr size_t kPairs3MaxBytes = (size_t(1) << 26) * P3_SLOTS * sizeof(float4);

struct DevBuf3 {
    void *p = nullptr;
    size_t cap = 0;
};

int ensure3(DevBuf3 &b, size_t bytes, cudaStream_t st) {
    if (bytes == 0) bytes = 16;
    if (b.cap >= bytes) return PETFMM_OK;
    if (b.p) {
        if (cudaStreamSynchronize(st) != cudaSuccess) return PETFMM_ECUDA;
        cudaFree(b.p);
        b.p = nullptr;
        b.cap = 0;
    }
    if (cudaMalloc(&b.p, bytes) != cudaSuccess) {
        cudaGetLastError();
        b.p = nullptr;
        return PETFMM_ENOMEM;
    }
    b.cap = bytes;
    return PETFMM_OK;
}

// A table, copied on the context's stream: the launches that follow there find it
// complete.
int upload3(DevBuf3 &b, const void *src, size_t bytes, cudaStream_t st) {
    const int rc = ensure3(b, bytes, st);
    if (rc) return rc;
    if (copy_table(b.p, src, bytes, st) == cudaSuccess) return PETFMM_OK;
    cudaGetLastError();
    return PETFMM_ECUDA;
}

int free3(DevBuf3 &b, cudaStream_t st) {
    if (!b.p) return PETFMM_OK;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PETFMM_ECUDA;
    cudaFree(b.p);
    b = DevBuf3();
    return PETFMM_OK;
}

}  // namespace

struct petfmm3d_ctx {
    petfmm_domain3d dom{};
    int L = 0, p = 0, precision = 0, dtype = 0;
    cudaStream_t stream = nullptr;
    DevBuf3 keysA, keysB, valsA, valsB, sortw, start, recu, rec, xs, me, le, status;
    // near field: one-sided and pair items, parts of the charges' sums, flags, counters
    DevBuf3 nitems, pitems, slots, nown, nflags, nctrl;
    bool no_pairs = false;  // no room for the planes of pairwise sums
    size_t pair_bytes = kPairs3MaxBytes;  // PETFMM3D_OPT_PAIR_BYTES
    // operator tables of the context's precision only
    DevBuf3 orbits, atab32, rmap, parity;  // M2L operators: by orbit, by offset
    DevBuf3 shift, order;  // the M2M and L2L operators of octant 0, rows by parity class
    Shift3 sh{};
    DevBuf3 tcimg;  // p <= 8: TF32 hi / lo images of the M2L operators (tensor-core M2L)
    int m2l_tc = 2;  // PETFMM3D_OPT_M2L_TC
    bool timing = false, ev_recorded = false;
    cudaEvent_t ev[PETFMM3D_STAGE_COUNT + 1] = {};
    uint64_t launches = 0, evaluations = 0;
    int64_t last_n = 0;
    bool sorted_in_first = true;
};

namespace {

#define P3_TRY(x) do { int rc_ = (x); if (rc_) return rc_; } while (0)
#define P3_CUDA(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { cudaGetLastError(); \
    return e_ == cudaErrorMemoryAllocation ? PETFMM_ENOMEM : PETFMM_ECUDA; } } while (0)

// M2L by reflection orbits: FP64, p > 8, and by default the mixed path's trees
// of up to four levels, where the tensor-core kernel waits on its serial chain
// of offsets (us, tensor cores / orbits: L = 3, p = 8 653 / 90; L = 4, p = 8
// 733 / 549, p = 5 496 / 170; L = 5, p = 8 799 / 4132, p = 5 518 / 983).  p > 8,
// against a SIMT GEMM over every offset: L = 4, p = 12 7.87 / 2.84 ms, L = 5,
// p = 16 181 / 51 ms.
bool use_orbits3(const petfmm3d_ctx *c) {
    return c->precision == PETFMM_FP64 || c->p > TC3_MAXP || (c->m2l_tc == 2 && c->L <= 4);
}

// The real basis of the M2L matrices: real index r < nc is Re of coefficient r, r
// >= nc Im of the coefficients with m > 0 in order; parity: bit d set if the
// solid harmonic changes sign with axis d.
void real_basis3(int p, std::vector<short2> &rm, std::vector<uint8_t> &par) {
    rm.resize(size_t(p) * p);
    par.resize(size_t(p) * p);
    for (int n = 0, r = nc3(p); n < p; ++n)
        for (int m = 0; m <= n; ++m) {
            const int j = n * (n + 1) / 2 + m;
            rm[size_t(j)] = make_short2(short(j), short(m == 0 ? 2 : 0));
            par[size_t(j)] = uint8_t((m & 1) | (((n + m) & 1) << 2));
            if (m > 0) {
                par[size_t(r)] = uint8_t(((m + 1) & 1) | 2 | (((n + m) & 1) << 2));
                rm[size_t(r++)] = make_short2(short(j), 1);
            }
        }
}

// The M2L operators of the kernel that the options and the tree choose, made the
// first time they are needed: by orbit, or for every offset the tensor cores'
// images or the SIMT GEMM's matrices.
int m2l_tables(petfmm3d_ctx *c) {
    const int p = c->p, nc = nc3(p), nr = p * p, nrp = mg_nrp(p);
    const bool f64 = c->precision == PETFMM_FP64, by_orbit = use_orbits3(c);
    if (c->L < 2 || (by_orbit ? c->orbits : c->m2l_tc ? c->tcimg : c->atab32).p) return PETFMM_OK;
    std::vector<cd> iv(static_cast<size_t>(nci3(p)));
    // the orbits' operators [|dx| + 4 |dy| + 16 |dz|][k_in][r_out]
    std::vector<double> orb(size_t(64) * nr * nr, 0.0);
    for (int o = 0; o < 64; ++o) {
        const int dx = o & 3, dy = (o >> 2) & 3, dz = o >> 4;
        if (dx < 2 && dy < 2 && dz < 2) continue;
        host_rec_i(dx, dy, dz, 2 * p - 1, iv.data());
        host_m2l_real(p, iv.data(), orb.data() + size_t(o) * nr * nr);
    }
    if (by_orbit) {
        if (f64) return upload3(c->orbits, orb.data(), orb.size() * sizeof(double), c->stream);
        const std::vector<float> orb32(orb.begin(), orb.end());
        return upload3(c->orbits, orb32.data(), orb32.size() * sizeof(float), c->stream);
    }
    // Each offset's operator is its orbit's between the signs of the reflected
    // axes.  atab32: FP32, ap[k_in * nrp + r_out].  tcimg: TF32 hi / lo images for
    // the tensor cores: [slot][hi, lo][k / 4][n][k mod 4] = A[k][n] (zero
    // padding), K in the input basis of the tensor-core M2L (coefficient by
    // coefficient: Re, then Im if m > 0), N in the M2L matrices' basis.
    std::vector<short2> rm;
    std::vector<uint8_t> par;
    real_basis3(p, rm, par);
    std::vector<int> tc3_kin(static_cast<size_t>(nr));
    for (int n = 0, k = 0, t = 0; n < p; ++n)
        for (int m = 0; m <= n; ++m) {
            tc3_kin[size_t(k++)] = n * (n + 1) / 2 + m;
            if (m > 0) tc3_kin[size_t(k++)] = nc + t++;
        }
    const size_t mat = size_t(nrp) * nrp;
    std::vector<double> sign(static_cast<size_t>(nr));
    std::vector<float> tab(size_t(NSLOT3) * mat * (c->m2l_tc ? 2 : 1), 0.f);
    for (int slot = 0; slot < NSLOT3; ++slot) {
        const int dx = slot % 7 - 3, dy = (slot / 7) % 7 - 3, dz = slot / 49 - 3;
        if (std::max(std::abs(dx), std::max(std::abs(dy), std::abs(dz))) < 2) continue;
        const int o = std::abs(dx) + 4 * std::abs(dy) + 16 * std::abs(dz);
        const double *ao = orb.data() + size_t(o) * nr * nr;
        const int refl = (dx < 0) | (dy < 0) << 1 | (dz < 0) << 2;
        for (int r = 0; r < nr; ++r)
            sign[size_t(r)] = __builtin_popcount(par[size_t(r)] & refl) & 1 ? -1.0 : 1.0;
        auto entry = [&](int k, int r) {
            return ao[size_t(k) * nr + r] * (sign[size_t(k)] * sign[size_t(r)]);
        };
        if (!c->m2l_tc) {
            float *ap = tab.data() + size_t(slot) * mat;
            for (int k = 0; k < nr; ++k)
                for (int r = 0; r < nr; ++r) ap[size_t(k) * nrp + r] = float(entry(k, r));
            continue;
        }
        float *hi = tab.data() + size_t(slot) * 2 * mat, *lo = hi + mat;
        for (int k = 0; k < nr; ++k) {
            const int kin = tc3_kin[size_t(k)];
            for (int n = 0; n < nr; ++n) {
                const double a = entry(kin, n);
                const float h = host_tf32_rna(float(a));
                const size_t at = (size_t(k / 4) * nrp + n) * 4 + size_t(k % 4);
                hi[at] = h;
                lo[at] = host_tf32_rna(float(a - double(h)));
            }
        }
    }
    return upload3(c->m2l_tc ? c->tcimg : c->atab32, tab.data(), tab.size() * sizeof(float), c->stream);
}

int upload_tables(petfmm3d_ctx *c) {
    const int p = c->p, nr = p * p;
    std::vector<short2> rm;
    std::vector<uint8_t> par;
    real_basis3(p, rm, par);
    P3_TRY(upload3(c->rmap, rm.data(), rm.size() * sizeof(short2), c->stream));
    P3_TRY(upload3(c->parity, par.data(), par.size(), c->stream));
    std::vector<double> a64(size_t(nr) * nr);
    // M2M [k_in][r_out], then L2L with the rows k_in by parity class
    c->sh = Shift3{p, nr, std::max(1, 256 / nr), {}};
    std::vector<uint16_t> order;
    for (int f = 0; f < 8; ++f) {
        c->sh.cls[f] = int(order.size());
        for (int r = 0; r < nr; ++r)
            if (par[size_t(r)] == f) order.push_back(uint16_t(r));
    }
    c->sh.cls[8] = nr;
    std::vector<double> ops(size_t(2) * nr * nr);
    host_shift_real(p, 0, 0, ops.data());
    host_shift_real(p, 1, 0, a64.data());
    for (int k = 0; k < nr; ++k)
        std::copy_n(a64.data() + size_t(order[size_t(k)]) * nr, nr,
                    ops.data() + size_t(nr + k) * nr);
    const std::vector<float> ops32(ops.begin(), ops.end());
    const bool f64 = c->precision == PETFMM_FP64;
    const size_t es = f64 ? sizeof(double) : sizeof(float);
    P3_TRY(upload3(c->shift, f64 ? static_cast<const void *>(ops.data()) : ops32.data(),
                   ops.size() * es, c->stream));
    P3_TRY(upload3(c->order, order.data(), order.size() * sizeof(uint16_t), c->stream));
    return m2l_tables(c);
}

Dom3 make_dom3(const petfmm_domain3d &dom, int L) {
    Dom3 d{};
    d.x0 = dom.x0;
    d.y0 = dom.y0;
    d.z0 = dom.z0;
    d.width = dom.width;
    d.scale = std::ldexp(1.0, L) / dom.width;
    d.x0h = float(d.x0);
    d.x0l = float(d.x0 - double(d.x0h));
    d.y0h = float(d.y0);
    d.y0l = float(d.y0 - double(d.y0h));
    d.z0h = float(d.z0);
    d.z0l = float(d.z0 - double(d.z0h));
    d.sh = float(d.scale);
    d.sl = float(d.scale - double(d.sh));
    return d;
}

void mark3(petfmm3d_ctx *c, int s) {
    if (c->timing) cudaEventRecord(c->ev[s], c->stream);
}

unsigned grid_w(int64_t warps) { return unsigned((warps + W3 - 1) / W3); }

template <int P>
cudaError_t m2l_gemm_p(int L, const uint32_t *start, const float *atab, const float2 *me,
                       float2 *le, cudaStream_t st) {
    constexpr int R = MG_PIPE_ROWS;
    constexpr size_t smem = mgp_smem_bytes<P, R>();
    static bool pattr = false;
    if (!pattr) {
        cudaError_t e = cudaFuncSetAttribute(k3_m2l_pipe<P, R>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        pattr = true;
    }
    int64_t grid = 0;
    for (int k = 2; k <= L; ++k) grid += mg_blocks(k, R);
    k3_m2l_pipe<P, R><<<unsigned(grid), MG_THREADS, smem, st>>>(L, start, atab, me, le);
    return cudaGetLastError();
}

template <int P>
cudaError_t m2l_tc_p(int L, const uint32_t *start, const float *bimg, const float2 *me, float2 *le,
                     int *status, cudaStream_t st) {
    if constexpr (mg_nrp(P) <= 64 && mg_nrp(P) % 16 == 0) {
        constexpr size_t smem = tc3_smem_bytes<P>();
        static bool attr = false;
        if (!attr) {
            cudaError_t e = cudaFuncSetAttribute(k3_m2l_tc<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 int(smem));
            if (e != cudaSuccess) return e;
            attr = true;
        }
        int64_t grid = 0;
        for (int k = 2; k <= L; ++k) grid += tc3_blocks(k);
        k3_m2l_tc<P><<<unsigned(grid), TC3_THREADS, smem, st>>>(L, start, bimg, me, le, 1LL << 26,
                                                                status);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

// all levels 2..L in one launch, p <= 8
cudaError_t launch_m2l_tc3(int p, int L, const uint32_t *start, const float *bimg, const float2 *me,
                           float2 *le, int *status, cudaStream_t st) {
    switch (p) {
#define TC3_CASE(P) case P: return m2l_tc_p<P>(L, start, bimg, me, le, status, st);
        TC3_CASE(1) TC3_CASE(2) TC3_CASE(3) TC3_CASE(4) TC3_CASE(5) TC3_CASE(6) TC3_CASE(7)
        TC3_CASE(8)
#undef TC3_CASE
        default: return cudaErrorInvalidValue;
    }
}

// all levels 2..L in one launch, p <= 8
cudaError_t launch_m2l_gemm(int p, int L, const uint32_t *start, const float *atab,
                            const float2 *me, float2 *le, cudaStream_t st) {
    switch (p) {
#define MG_CASE(P) case P: return m2l_gemm_p<P>(L, start, atab, me, le, st);
        MG_CASE(1) MG_CASE(2) MG_CASE(3) MG_CASE(4) MG_CASE(5) MG_CASE(6) MG_CASE(7) MG_CASE(8)
#undef MG_CASE
        default: return cudaErrorInvalidValue;
    }
}

template <typename T>
int expansions3(petfmm3d_ctx *c, const uint32_t *start) {
    using V = typename C3<T>::V;
    const int L = c->L, p = c->p;
    cudaStream_t st = c->stream;
    V *me = static_cast<V *>(c->me.p), *le = static_cast<V *>(c->le.p);
    const Dom3 d = make_dom3(c->dom, L);
    mark3(c, PETFMM3D_STAGE_P2M);
    using Rec = std::conditional_t<sizeof(T) == 4, float4, Dbl4>;
    const Rec *rec = static_cast<const Rec *>(sizeof(T) == 4 ? c->rec.p : c->xs.p);
    if (p <= 8)
        P3_CUDA(launch_p2m_lanes<T>(p, L, d, start, rec, me, st));
    else
        k3_p2m<T, Rec><<<grid_w(int64_t(1) << (3 * L)), W3 * 32, 0, st>>>(L, p, d, start, rec, me);
    P3_CUDA(cudaGetLastError());
    c->launches++;
    mark3(c, PETFMM3D_STAGE_M2M);
    const T *op = static_cast<const T *>(c->shift.p);
    const short2 *rmap = static_cast<const short2 *>(c->rmap.p);
    const uint8_t *par = static_cast<const uint8_t *>(c->parity.p);
    const uint16_t *order = static_cast<const uint16_t *>(c->order.p);
    for (int l = L - 1; l >= 2; --l) {
        P3_CUDA((launch_shift3<T, false>(l, L, c->sh, start, op, rmap, par, order, me, st)));
        c->launches++;
    }
    P3_TRY(m2l_tables(c));  // (after an option changed the kernel)
    mark3(c, PETFMM3D_STAGE_M2L);
    if (use_orbits3(c)) {
        P3_CUDA(launch_m2l_orbits<T>(L, p, start, static_cast<const T *>(c->orbits.p), rmap, par, me,
                                     le, st));
    } else if constexpr (sizeof(T) == 4) {
        if (c->m2l_tc)
            P3_CUDA(launch_m2l_tc3(p, L, start, static_cast<const float *>(c->tcimg.p), me, le,
                                   static_cast<int *>(c->status.p), st));
        else
            P3_CUDA(launch_m2l_gemm(p, L, start, static_cast<const float *>(c->atab32.p), me, le, st));
    }
    c->launches++;
    mark3(c, PETFMM3D_STAGE_L2L);
    for (int l = 2; l < L; ++l) {
        P3_CUDA((launch_shift3<T, true>(l, L, c->sh, start, op + size_t(c->sh.nr) * c->sh.nr, rmap,
                                        par, order, le, st)));
        c->launches++;
    }
    return PETFMM_OK;
}

// One-sided work items of up to 32 targets: at most min(8^L, n) + n / 32.
int64_t directed_cap3(int64_t n, int64_t nleaf) { return std::min(nleaf, n) + n / 32 + 1; }

// The buffers that an evaluation of n charges cannot do without: those of the
// tree and the expansions, those of the near field.
int tree_buffers3(petfmm3d_ctx *c, int64_t n) {
    cudaStream_t st = c->stream;
    const bool mixed = c->precision == PETFMM_MIXED;
    const int64_t nleaf = int64_t(1) << (3 * c->L), nbox = lvl_off3(c->L + 1);
    const size_t series = size_t(nbox) * nc3(c->p) * (mixed ? sizeof(float2) : sizeof(double2));
    P3_TRY(ensure3(c->keysA, size_t(n) * 4, st));
    P3_TRY(ensure3(c->keysB, size_t(n) * 4, st));
    P3_TRY(ensure3(c->valsA, size_t(n) * 4, st));
    P3_TRY(ensure3(c->valsB, size_t(n) * 4, st));
    P3_TRY(ensure3(c->sortw, size_t(radix_scratch_words(n)) * 4, st));
    P3_TRY(ensure3(c->start, size_t(nleaf + 1) * 4, st));
    P3_TRY(ensure3(c->me, series, st));
    P3_TRY(ensure3(c->le, series, st));
    if (mixed) {
        P3_TRY(ensure3(c->recu, size_t(n) * sizeof(float4), st));
        P3_TRY(ensure3(c->rec, size_t(n) * sizeof(float4), st));
    } else {
        P3_TRY(ensure3(c->xs, size_t(n) * sizeof(Dbl4), st));
    }
    return PETFMM_OK;
}
int near_buffers3(petfmm3d_ctx *c, int64_t n) {
    cudaStream_t st = c->stream;
    const int64_t nleaf = int64_t(1) << (3 * c->L);
    P3_TRY(ensure3(c->nown, size_t(n) * (c->precision == PETFMM_MIXED ? sizeof(float4) : sizeof(Dbl4)),
                   st));
    P3_TRY(ensure3(c->nitems, size_t(directed_cap3(n, nleaf)) * sizeof(uint2), st));
    P3_TRY(ensure3(c->nflags, size_t(nleaf) * 4, st));
    P3_TRY(ensure3(c->nctrl, C3_WORDS * 4, st));
    return PETFMM_OK;
}

// Either of them; the planes of the pairwise sums give way where a needed buffer
// cannot be had beside them.
int needed3(petfmm3d_ctx *c, int64_t n, int (*buffers)(petfmm3d_ctx *, int64_t)) {
    const int rc = buffers(c, n);
    if (rc != PETFMM_ENOMEM || !c->slots.p) return rc;
    P3_TRY(free3(c->slots, c->stream));
    c->no_pairs = true;
    return buffers(c, n);
}

// The near field's buffers: where they are allowed and there is room, the planes
// and items of the pairwise sums too (*icap of them), else nr->pmin stays all
// ones and every leaf pair is summed one-sided.
int near3(petfmm3d_ctx *c, int64_t n, Near3 *nr, int64_t *icap) {
    cudaStream_t st = c->stream;
    const bool mixed = c->precision == PETFMM_MIXED;
    const int64_t nleaf = int64_t(1) << (3 * c->L);
    const uint32_t pmin = mixed ? P3_PAIR_MIN : 1;
    const size_t parts = mixed ? P3_SLOTS * sizeof(float4) : P3_SLOTS64 * sizeof(Dbl4);
    nr->n = n;
    nr->pmin = ~0u;
    nr->share = mixed ? P3_SHARE : P3_SHARE64;
    nr->enough = mixed ? P3_ENOUGH : P3_ENOUGH64;
    P3_TRY(needed3(c, n, near_buffers3));
    // (up to n^2 pairs of charges, a half octave's taken for up to 3/2 of them: too
    // few charges for any pairwise sum need no lists of them)
    const bool enough = uint64_t(n) * uint64_t(n) / 2 * 3 >= nr->enough;
    if (n >= 2 * int64_t(pmin) && enough && n * parts <= c->pair_bytes && !c->no_pairs) {
        // up to 2 groups of a leaf of at least pmin, 4 above 96 charges, 14 above 384
        *icap = 2 * std::min<int64_t>(nleaf, n / pmin) + 2 * (n / 97) + 10 * (n / 385) + 1;
        int rc = ensure3(c->pitems, size_t(*icap) * sizeof(uint2), st);
        if (rc == PETFMM_OK) rc = ensure3(c->slots, n * parts, st);
        if (rc == PETFMM_OK) {
            nr->pmin = pmin;
        } else if (rc == PETFMM_ENOMEM) {
            P3_TRY(free3(c->slots, st));
            P3_TRY(free3(c->pitems, st));
            c->no_pairs = true;
        } else {
            return rc;
        }
    }
    nr->own = static_cast<float4 *>(c->nown.p);
    nr->slots = static_cast<float4 *>(c->slots.p);
    nr->flags = static_cast<uint32_t *>(c->nflags.p);
    nr->ctrl = static_cast<uint32_t *>(c->nctrl.p);
    nr->directed = static_cast<uint2 *>(c->nitems.p);
    nr->items = static_cast<uint2 *>(c->pitems.p);
    P3_CUDA(cudaMemsetAsync(nr->ctrl, 0, C3_WORDS * 4, st));
    return PETFMM_OK;
}

int evaluate3(petfmm3d_ctx *c, int64_t n, const void *x, const void *y, const void *z,
              const void *q, void *phi, void *ex, void *ey, void *ez) {
    cudaStream_t st = c->stream;
    const int L = c->L, p = c->p;
    const bool mixed = c->precision == PETFMM_MIXED, f32 = c->dtype == PETFMM_F32;
    P3_TRY(ensure3(c->status, 16, st));
    P3_CUDA(cudaMemsetAsync(c->status.p, 0, sizeof(int), st));
    c->last_n = n;
    c->ev_recorded = false;
    if (n == 0) return PETFMM_OK;
    const int64_t nleaf = int64_t(1) << (3 * L);
    P3_TRY(needed3(c, n, tree_buffers3));
    uint32_t *kA = static_cast<uint32_t *>(c->keysA.p), *kB = static_cast<uint32_t *>(c->keysB.p);
    uint32_t *vA = static_cast<uint32_t *>(c->valsA.p), *vB = static_cast<uint32_t *>(c->valsB.p);
    uint32_t *start = static_cast<uint32_t *>(c->start.p);
    int *status = static_cast<int *>(c->status.p);
    const Dom3 d = make_dom3(c->dom, L);
    const unsigned gp = unsigned((n + 255) / 256);
    float4 *recu = mixed ? static_cast<float4 *>(c->recu.p) : nullptr;

    mark3(c, PETFMM3D_STAGE_BIN);
    if (f32)
        k3_bin<float><<<gp, 256, 0, st>>>(n, static_cast<const float *>(x), static_cast<const float *>(y),
                                          static_cast<const float *>(z), static_cast<const float *>(q),
                                          d, L, kA, recu, status);
    else
        k3_bin<double><<<gp, 256, 0, st>>>(n, static_cast<const double *>(x), static_cast<const double *>(y),
                                           static_cast<const double *>(z), static_cast<const double *>(q),
                                           d, L, kA, recu, status);
    P3_CUDA(cudaGetLastError());
    c->launches++;
    mark3(c, PETFMM3D_STAGE_SORT);
    bool in_first = true;
    P3_CUDA(radix_sort(kA, vA, kB, vB, n, 3 * L, static_cast<uint32_t *>(c->sortw.p), &in_first, st,
                       &c->launches));
    c->sorted_in_first = in_first;
    const uint32_t *skeys = in_first ? kA : kB;
    const uint32_t *perm = in_first ? vA : vB;
    k3_leaf_start<<<unsigned((nleaf + 1 + 255) / 256), 256, 0, st>>>(skeys, n, nleaf, start);
    P3_CUDA(cudaGetLastError());
    c->launches++;
    mark3(c, PETFMM3D_STAGE_GATHER);
    if (mixed) {
        P3_CUDA(launch_gather_mixed(recu, perm, static_cast<float4 *>(c->rec.p), n, st, &c->launches));
    } else {
        Dbl4 *xs = static_cast<Dbl4 *>(c->xs.p);
        if (f32)
            k3_gather_f64<float><<<gp, 256, 0, st>>>(n, perm, static_cast<const float *>(x),
                                                     static_cast<const float *>(y),
                                                     static_cast<const float *>(z),
                                                     static_cast<const float *>(q), xs);
        else
            k3_gather_f64<double><<<gp, 256, 0, st>>>(n, perm, static_cast<const double *>(x),
                                                      static_cast<const double *>(y),
                                                      static_cast<const double *>(z),
                                                      static_cast<const double *>(q), xs);
        P3_CUDA(cudaGetLastError());
        c->launches++;
    }
    if (L >= 2) {
        if (mixed)
            P3_TRY(expansions3<float>(c, start));
        else
            P3_TRY(expansions3<double>(c, start));
    } else {
        for (int s = PETFMM3D_STAGE_P2M; s <= PETFMM3D_STAGE_L2L; ++s) mark3(c, s);
    }
    mark3(c, PETFMM3D_STAGE_NEAR);
    const double w = c->dom.width / double(int64_t(1) << L);
    const unsigned gb = unsigned((nleaf + 255) / 256);
    const unsigned gi = grid_w(directed_cap3(n, nleaf));
    Near3 nr{};
    int64_t icap = 0;
    P3_TRY(near3(c, n, &nr, &icap));
    const bool pairs = nr.pmin != ~0u;
    if (mixed) {
        const float4 *rec = static_cast<const float4 *>(c->rec.p);
        const float2 *le = static_cast<const float2 *>(c->le.p);
        if (pairs) {
            k3_near_items<false, P3_DIRS><<<gb, 256, 0, st>>>(L, start, nr);
            P3_CUDA(cudaGetLastError());
            c->launches++;
        }
        k3_near_items<true, P3_DIRS><<<gb, 256, 0, st>>>(L, start, nr);
        P3_CUDA(cudaGetLastError());
        if (pairs) {
            k3_pairs<<<unsigned((icap + 3) / 4), 128, 0, st>>>(L, start, rec, nr);
            P3_CUDA(cudaGetLastError());
            c->launches++;
        }
        k3_near_directed<<<gi, W3 * 32, 0, st>>>(L, start, rec, nr);
        P3_CUDA(cudaGetLastError());
        c->launches += 2;
        if (f32)
            k3_near_final<float><<<gp, 256, 0, st>>>(L, p, w, skeys, start, rec, le, perm, nr, phi,
                                                     ex, ey, ez);
        else
            k3_near_final<double><<<gp, 256, 0, st>>>(L, p, w, skeys, start, rec, le, perm, nr, phi,
                                                      ex, ey, ez);
    } else {
        const Dbl4 *xs = static_cast<const Dbl4 *>(c->xs.p);
        const double2 *le = static_cast<const double2 *>(c->le.p);
        Dbl4 *slots = static_cast<Dbl4 *>(c->slots.p), *own = static_cast<Dbl4 *>(c->nown.p);
        if (pairs) {
            k3_near_items<false, P3_GROUPS64><<<gb, 256, 0, st>>>(L, start, nr);
            P3_CUDA(cudaGetLastError());
            c->launches++;
        }
        k3_near_items<true, P3_GROUPS64><<<gb, 256, 0, st>>>(L, start, nr);
        P3_CUDA(cudaGetLastError());
        if (pairs) {
            constexpr int pad = int(kPairs64Smem - PW64 * (PT64 + PA64) * sizeof(Dbl4));
            P3_CUDA(cudaFuncSetAttribute(k3_pairs_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         pad));
            k3_pairs_f64<<<unsigned((icap + PW64 - 1) / PW64), PW64 * 32, pad, st>>>(L, start, xs, nr,
                                                                                   slots);
            P3_CUDA(cudaGetLastError());
            c->launches++;
        }
        k3_near_directed64<<<gi, W3 * 32, 0, st>>>(L, start, xs, nr, own);
        P3_CUDA(cudaGetLastError());
        c->launches += 2;
        const unsigned gf = unsigned((n + 127) / 128);
        if (f32)
            k3_final_f64<float><<<gf, 128, 0, st>>>(L, p, d, skeys, start, xs, le, perm, nr, slots,
                                                    own, phi, ex, ey, ez);
        else
            k3_final_f64<double><<<gf, 128, 0, st>>>(L, p, d, skeys, start, xs, le, perm, nr, slots,
                                                     own, phi, ex, ey, ez);
    }
    P3_CUDA(cudaGetLastError());
    c->launches++;
    mark3(c, PETFMM3D_STAGE_COUNT);
    c->ev_recorded = c->timing;
    return PETFMM_OK;
}

}  // namespace

extern "C" {

int petfmm3d_create(const petfmm_domain3d *dom, int levels, int order, int precision, int dtype,
                    void *cuda_stream, petfmm3d_ctx **out) {
    if (!out) return PETFMM_EINVAL;
    *out = nullptr;
    if (!dom || !(dom->width > 0.0) || !std::isfinite(dom->width) || !std::isfinite(dom->x0) ||
        !std::isfinite(dom->y0) || !std::isfinite(dom->z0))
        return PETFMM_EINVAL;
    if (levels < 1 || levels > L3_MAX || order < 1 || order > P3_MAX) return PETFMM_EINVAL;
    if (precision != PETFMM_FP64 && precision != PETFMM_MIXED) return PETFMM_EINVAL;
    if (dtype != PETFMM_F64 && dtype != PETFMM_F32) return PETFMM_EINVAL;
    petfmm3d_ctx *c = new (std::nothrow) petfmm3d_ctx;
    if (!c) return PETFMM_ENOMEM;
    c->dom = *dom;
    c->L = levels;
    c->p = order;
    c->precision = precision;
    c->dtype = dtype;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    int rc = upload_tables(c);
    for (int i = 0; !rc && i <= PETFMM3D_STAGE_COUNT; ++i)
        if (cudaEventCreate(&c->ev[i]) != cudaSuccess) rc = PETFMM_ECUDA;
    if (rc) {
        cudaGetLastError();
        petfmm3d_destroy(c);
        return rc;
    }
    *out = c;
    return PETFMM_OK;
}

int petfmm3d_evaluate(petfmm3d_ctx *c, int64_t n, const void *x, const void *y, const void *z,
                      const void *q, void *phi, void *ex, void *ey, void *ez) {
    if (!c || n < 0 || n > int64_t(0xffffffffu) / 4) return PETFMM_EINVAL;
    if (n > 0 && (!x || !y || !z || !q || !phi || !ex || !ey || !ez)) return PETFMM_EINVAL;
    const int rc = evaluate3(c, n, x, y, z, q, phi, ex, ey, ez);
    if (!rc) c->evaluations++;
    return rc;
}

int petfmm3d_sync(petfmm3d_ctx *c) {
    if (!c) return PETFMM_EINVAL;
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) {
        cudaGetLastError();
        return PETFMM_ECUDA;
    }
    if (!c->status.p) return PETFMM_OK;
    int s = 0;
    if (cudaMemcpy(&s, c->status.p, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return PETFMM_ECUDA;
    }
    return s;
}

int petfmm3d_set_option(petfmm3d_ctx *c, int option, int64_t value) {
    if (!c) return PETFMM_EINVAL;
    switch (option) {
        case PETFMM3D_OPT_TIMING: c->timing = value != 0; return PETFMM_OK;
        case PETFMM3D_OPT_M2L_TC:
            if (value < 0 || value > 2) return PETFMM_EINVAL;
            c->m2l_tc = int(value);
            return PETFMM_OK;
        case PETFMM3D_OPT_PAIR_BYTES:
            if (value < 0) return PETFMM_EINVAL;
            c->pair_bytes = size_t(value);
            c->no_pairs = false;
            // (planes above the new limit are given back)
            return c->slots.cap > c->pair_bytes ? free3(c->slots, c->stream) : PETFMM_OK;
        default: return PETFMM_EINVAL;
    }
}

int petfmm3d_stage_times(petfmm3d_ctx *c, float *ms, int cap) {
    if (!c || !ms || cap < 0) return PETFMM_EINVAL;
    if (!c->ev_recorded) return PETFMM_ENOTREADY;
    const int k = std::min(cap, int(PETFMM3D_STAGE_COUNT));
    for (int s = 0; s < k; ++s) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, c->ev[s], c->ev[s + 1]) != cudaSuccess) {
            cudaGetLastError();
            return PETFMM_ECUDA;
        }
        ms[s] = t;
    }
    return k;
}

int petfmm3d_debug_tree(petfmm3d_ctx *c, int64_t n, uint32_t *skeys, uint32_t *perm,
                        uint32_t *start) {
    if (!c || n != c->last_n || n <= 0 || !skeys || !perm || !start) return PETFMM_EINVAL;
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return PETFMM_ECUDA;
    const void *k = c->sorted_in_first ? c->keysA.p : c->keysB.p;
    const void *v = c->sorted_in_first ? c->valsA.p : c->valsB.p;
    const size_t nleaf = size_t(1) << (3 * c->L);
    if (cudaMemcpy(skeys, k, size_t(n) * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(perm, v, size_t(n) * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(start, c->start.p, (nleaf + 1) * 4, cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return PETFMM_ECUDA;
    }
    return PETFMM_OK;
}

uint64_t petfmm3d_launches(const petfmm3d_ctx *c) { return c ? c->launches : 0; }

int petfmm3d_debug_m2l_operator(int order, int dx, int dy, int dz, double *out, int64_t cap) {
    if (order < 1 || order > P3_MAX || !out) return PETFMM_EINVAL;
    if (std::abs(dx) > 3 || std::abs(dy) > 3 || std::abs(dz) > 3 ||
        std::max(std::abs(dx), std::max(std::abs(dy), std::abs(dz))) < 2)
        return PETFMM_EINVAL;
    const int64_t nr = int64_t(order) * order;
    if (cap < nr * nr) return PETFMM_EINVAL;
    std::vector<cd> iv(size_t(nci3(order)));
    host_rec_i(dx, dy, dz, 2 * order - 1, iv.data());
    host_m2l_real(order, iv.data(), out);
    return PETFMM_OK;
}

int petfmm3d_debug_shift_operator(int order, int kind, int octant, double *out, int64_t cap) {
    if (order < 1 || order > P3_MAX || !out) return PETFMM_EINVAL;
    if ((kind != PETFMM3D_SHIFT_M2M && kind != PETFMM3D_SHIFT_L2L) || octant < 0 || octant > 7)
        return PETFMM_EINVAL;
    const int64_t nr = int64_t(order) * order;
    if (cap < nr * nr) return PETFMM_EINVAL;
    host_shift_real(order, kind == PETFMM3D_SHIFT_M2M ? 0 : 1, octant, out);
    return PETFMM_OK;
}

int petfmm3d_debug_rsqrt(petfmm3d_ctx *c, int64_t n, const double *x, double *y) {
    if (!c || n < 0 || (n > 0 && (!x || !y))) return PETFMM_EINVAL;
    if (n > 0) k3_rsqrt64<<<unsigned((n + 255) / 256), 256, 0, c->stream>>>(x, y, n);
    return cudaGetLastError() == cudaSuccess ? PETFMM_OK : PETFMM_ECUDA;
}

int petfmm3d_destroy(petfmm3d_ctx *c) {
    if (!c) return PETFMM_EINVAL;
    if (c->stream) cudaStreamSynchronize(c->stream);
    DevBuf3 *bufs[] = {&c->nitems, &c->pitems, &c->slots,
                       &c->nown, &c->nflags, &c->nctrl,
                       &c->keysA, &c->keysB, &c->valsA, &c->valsB, &c->sortw, &c->start,
                       &c->recu,  &c->rec,   &c->xs,    &c->me,    &c->le,    &c->status,
                       &c->orbits, &c->atab32, &c->parity, &c->rmap,
                       &c->shift, &c->order, &c->tcimg};
    for (DevBuf3 *b : bufs)
        if (b->p) cudaFree(b->p);
    for (int i = 0; i <= PETFMM3D_STAGE_COUNT; ++i)
        if (c->ev[i]) cudaEventDestroy(c->ev[i]);
    cudaGetLastError();
    delete c;
    return PETFMM_OK;
}

}  // extern "C"
