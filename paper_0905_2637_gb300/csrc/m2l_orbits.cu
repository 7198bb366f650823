// m2l_orbits.cu -- M2L by orbits of quarter turns (Sec. 2.2): the FP64 path, and
// the levels of the mixed path that the tensor cores do not take.
//
// Vortex kernel: c^_m = sum_delta sum_k R[k][m] delta^-(k+m+1) a~_k, R[k][m] =
// (-1)^(k+1) C(k+m, k), over the 27 offsets delta of the interaction list:
//  - Offsets that are quarter turns of one another, delta = i^r delta_0, share
//    one product: with H_j[k] = sum_r i^(-r j) a~_k^(r) (a four-point Fourier
//    sum, additions only) their part is sum_k R[k][m] delta_0^-(k+m+1)
//    H_{(k+m+1) mod 4}[k].  The 27 offsets form 10 such orbits.
//  - delta_0^-k is applied to the sources and delta_0^-(m+1) to the sum, so
//    the product itself is a real matrix on complex vectors, the same R for
//    every orbit: 2 p^2 operations instead of 4 p^2.
// At p = 17 an interior box takes about 9,500 operations against 31,200 for
// 27 complex products.  The Laplace kernel has delta^-(k+m) and its own R; its
// term log(-delta) a~_0 of c^_0 is added apart.
//
// A block takes a run of consecutive (z-order) parent cells' children of one
// class; its (box, coefficient) pairs lie flat over the threads, NI each, so
// no lane idles.  The FP64 pipe (two lanes a cycle and SM on this part) bounds
// the FP64 path.  On the mixed path the coarse levels hold few boxes and the
// time is latency: the sources of all orbits are looked up at once, and with
// NI = 1 the next orbit's coefficients are loaded while the current one
// multiplies.
// Measured on one GB300.  FP64, against a warp per box with 27 complex
// products: 1,048,576 blobs, L = 8, p = 17: 13.8 -> 1.9 ms; 10,000 blobs, L = 4,
// p = 12: 0.56 -> 0.04 ms.  Mixed, against tiled complex products
// of the 27 offsets (a launch of 64 to 128 boxes a block, 12 barriers in turn):
// 4,096 blobs, L = 4, p = 17: 0.094 -> 0.014 ms for the whole M2L; 1,048,576
// blobs, L = 8, levels 2 to 7: 0.113 -> 0.06 ms, and half the error (a 300 x 300
// lattice: 1.9e-7 -> 1.3e-7 of the FP64 path).
#include <algorithm>
#include <cmath>
#include <vector>

#include "kernels.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

namespace {

constexpr int ORB_THREADS = 128;
constexpr int ORBITS = 10;
// representatives of the orbits, as (dx, dy) = source - target
__constant__ int8_t c_orbit[ORBITS][2] = {{2, 0}, {2, 1}, {2, -1}, {2, 2}, {3, 0},
                                          {3, 1}, {3, -1}, {3, 2}, {3, -2}, {3, 3}};
const int kOrbit[ORBITS][2] = {{2, 0}, {2, 1}, {2, -1}, {2, 2}, {3, 0},
                               {3, 1}, {3, -1}, {3, 2}, {3, -2}, {3, 3}};

// target boxes of a block
__host__ __device__ __forceinline__ int orb_rows(int p, int ni) {
    const int r = ORB_THREADS * ni / p;
    return r < 64 ? r : 64;
}

// delta_0 turned by r quarter turns
__device__ __forceinline__ void turned(int o, int r, int *dx, int *dy) {
    const int x = c_orbit[o][0], y = c_orbit[o][1];
    *dx = r == 0 ? x : r == 1 ? -y : r == 2 ? -x : y;
    *dy = r == 0 ? y : r == 1 ? x : r == 2 ? -y : -x;
}

// The complex products with their roundings spelled out: the instances of the
// kernel must give the same bits (a batch and a tree alone).
template <typename C2> __device__ __forceinline__ C2 orb_mul(C2 a, C2 b) {
    C2 r;
    r.x = fma(a.x, b.x, -(a.y * b.y));
    r.y = fma(a.x, b.y, a.y * b.x);
    return r;
}
template <typename C2> __device__ __forceinline__ C2 orb_fma(C2 a, C2 b, C2 c) {
    C2 r;
    r.x = fma(a.x, b.x, fma(-a.y, b.y, c.x));
    r.y = fma(a.x, b.y, fma(a.y, b.x, c.y));
    return r;
}
template <typename C2, typename R> __device__ __forceinline__ C2 orb_c(R x, R y) {
    C2 r;
    r.x = x;
    r.y = y;
    return r;
}

}  // namespace

// Reals: R ([k][m]); per orbit delta_0^-j for j = 0..p as complex; per orbit
// and turn log(-delta) (Laplace kernel; else zero).
void host_m2l_orbit_table(int p, int kernel, std::vector<double> &out) {
    const bool lap = kernel == KERNEL_LAPLACE;
    out.assign(size_t(p) * p + size_t(ORBITS) * (p + 1) * 2 + ORBITS * 8, 0.0);
    for (int k = 0; k < p; ++k)
        for (int m = 0; m < p; ++m) {
            // C(k + m, k); Laplace kernel: C(k + m - 1, k - 1), -1 / m for k = 0
            const int a = lap ? k - 1 : k;
            double c = 1.0;
            for (int i = 1; i <= a; ++i) c = c * double(m + i) / double(i);
            c = std::nearbyint(c);
            double v = (k & 1) ? c : -c;
            if (lap) v = k ? ((k & 1) ? -c : c) : m ? -1.0 / m : 0.0;
            out[size_t(k) * p + m] = v;
        }
    double *pw = out.data() + size_t(p) * p, *lg = pw + size_t(ORBITS) * (p + 1) * 2;
    for (int o = 0; o < ORBITS; ++o) {
        const long double x = kOrbit[o][0], y = kOrbit[o][1], n = x * x + y * y;
        long double re = 1.0L, im = 0.0L;
        for (int j = 0; j <= p; ++j) {
            pw[(size_t(o) * (p + 1) + j) * 2] = double(re);
            pw[(size_t(o) * (p + 1) + j) * 2 + 1] = double(im);
            const long double t = (re * x + im * y) / n;  // times 1 / delta_0
            im = (im * x - re * y) / n;
            re = t;
        }
        for (int r = 0; lap && r < 4; ++r) {
            const double dx = r == 0 ? kOrbit[o][0] : r == 1 ? -kOrbit[o][1] : r == 2 ? -kOrbit[o][0] : kOrbit[o][1];
            const double dy = r == 0 ? kOrbit[o][1] : r == 1 ? kOrbit[o][0] : r == 2 ? -kOrbit[o][1] : -kOrbit[o][0];
            lg[(o * 4 + r) * 2] = 0.5 * std::log(double(n));
            lg[(o * 4 + r) * 2 + 1] = std::atan2(-dy, -dx);
        }
    }
}

int64_t m2l_orbit_units(int p, int level, int ni) {
    const int64_t np = int64_t(1) << (2 * (level - 1));
    const int rows = orb_rows(p, ni);
    return (np + rows - 1) / rows * 4;
}

template <typename R, int NI>
__global__ void __launch_bounds__(ORB_THREADS) k_m2l_orbits(
    const Task *__restrict__ tasks, int ntasks, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const typename Cplx<R>::T *__restrict__ me,
    typename Cplx<R>::T *__restrict__ le) {
    using C2 = typename Cplx<R>::T;
    extern __shared__ __align__(16) unsigned char orb_smem[];
    __shared__ uint32_t s_act;
    const int tid = threadIdx.x;
    const Task t = tasks[find_task(tasks, ntasks, blockIdx.x)];
    const InstDesc &d = insts[t.inst];
    const int p = d.p, l = t.level, nside = 1 << l;
    const int rows = orb_rows(p, NI), js = rows * p + 1;  // one of padding: four H, four banks
    const int64_t unit = int64_t(blockIdx.x) - t.block0;
    const int c = int(unit & 3);
    const int64_t np = int64_t(1) << (2 * (l - 1)), p0 = (unit >> 2) * rows;
    const bool lap = d.kernel == KERNEL_LAPLACE;
    const int ex = lap ? 0 : 1;  // delta^-(k + m + ex)
    C2 *h = reinterpret_cast<C2 *>(orb_smem);         // [4][js]
    C2 *pw = h + 4 * js;                               // [orbit][p + 1]
    C2 *lg = pw + ORBITS * (p + 1);                    // [orbit][turn]
    C2 *lsum = lg + ORBITS * 4;                        // [box]: this orbit's log terms
    R *rm = reinterpret_cast<R *>(lsum + rows);        // [k][m]
    int *srow = reinterpret_cast<int *>(rm + p * p);  // [orbit][box][turn], -1: none
    const uint32_t *st = start + d.soff;
    if (tid == 0) s_act = 0;
    bool mine = false;
    for (int b = tid; b < rows; b += ORB_THREADS)
        if (p0 + b < np) mine |= box_count(st, d.L, l, uint32_t((p0 + b) * 4 + c)) != 0;
    if (!__syncthreads_or(mine)) return;  // no target box holds particles
    const R *tab = static_cast<const R *>(d.t_m2l);
    for (int i = tid; i < p * p; i += ORB_THREADS) rm[i] = tab[i];
    for (int i = tid; i < 2 * (ORBITS * (p + 1) + ORBITS * 4); i += ORB_THREADS)
        reinterpret_cast<R *>(pw)[i] = tab[p * p + i];
    // every orbit's sources: the turns in the class's interaction list
    const int lo_x = (c & 1) ? -3 : -2, lo_y = (c >> 1) ? -3 : -2;
    uint32_t act = 0;
    for (int e = tid; e < ORBITS * 4 * rows; e += ORB_THREADS) {
        const int r = e & 3, b = (e >> 2) % rows, o = (e >> 2) / rows;
        int dx, dy, src = -1;
        turned(o, r, &dx, &dy);
        if (p0 + b < np && dx >= lo_x && dx <= lo_x + 5 && dy >= lo_y && dy <= lo_y + 5) {
            const uint32_t pc = uint32_t(p0 + b);
            const int sx = 2 * int(compact_bits(pc)) + (c & 1) + dx;
            const int sy = 2 * int(compact_bits(pc >> 1)) + (c >> 1) + dy;
            if (sx >= 0 && sy >= 0 && sx < nside && sy < nside &&
                box_count(st, d.L, l, morton_key(uint32_t(sx), uint32_t(sy)))) {
                src = int(box_index(l, uint32_t(sx), uint32_t(sy)));
                act |= 1u << o;
            }
        }
        srow[e] = src;
    }
    if (act) atomicOr(&s_act, act);
    __syncthreads();
    act = s_act;
    int it_b[NI], it_m[NI];
    C2 acc[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int e = tid + i * ORB_THREADS;
        const bool in = e < rows * p;
        it_b[i] = in ? e / p : 0;
        it_m[i] = in ? e - it_b[i] * p : 0;
        acc[i] = orb_c<C2>(R(0), R(0));
    }
    const C2 *lev = me + d.eoff + lvl_off(l) * p;
    // the four sources of (box, coefficient) e in orbit o
    auto load = [&](int o, int b, int k, C2 (&a)[4]) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int s = srow[(o * rows + b) * 4 + r];
            a[r] = s >= 0 && PF_IN(s, int64_t(1) << (2 * l)) ? lev[int64_t(s) * p + k]
                                                              : orb_c<C2>(R(0), R(0));
        }
    };
    C2 ahead[4];
    if (NI == 1 && act && tid < rows * p) load(__ffs(act) - 1, it_b[0], it_m[0], ahead);
    while (act) {
        const int o = __ffs(act) - 1;
        act &= act - 1;
        int turns = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            int dx, dy;
            turned(o, r, &dx, &dy);
            if (dx >= lo_x && dx <= lo_x + 5 && dy >= lo_y && dy <= lo_y + 5) turns |= 1 << r;
        }
        const bool real_pw = c_orbit[o][1] == 0;
        const bool even = (turns & 5) != 0, odd = (turns & 10) != 0;
        __syncthreads();  // the previous orbit's products are done
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int e = tid + i * ORB_THREADS;
            if (e >= rows * p) continue;
            const int b = it_b[i], k = it_m[i];
            const C2 w = pw[o * (p + 1) + k];
            C2 a[4];
            if (NI == 1) {
#pragma unroll
                for (int r = 0; r < 4; ++r) a[r] = ahead[r];
            } else {
                load(o, b, k, a);
            }
            if (lap && k == 0) {
                C2 s = orb_c<C2>(R(0), R(0));
#pragma unroll
                for (int r = 0; r < 4; ++r) s = orb_fma(lg[o * 4 + r], a[r], s);
                lsum[b] = s;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if ((turns >> r) & 1)
                    a[r] = real_pw ? orb_c<C2>(a[r].x * w.x, a[r].y * w.x) : orb_mul(a[r], w);
            // sums and differences of opposite turns (of one alone: itself)
            C2 ep = a[0], em = a[0], op = a[1], om = a[1];
            if ((turns & 5) == 5) {
                ep = orb_c<C2>(a[0].x + a[2].x, a[0].y + a[2].y);
                em = orb_c<C2>(a[0].x - a[2].x, a[0].y - a[2].y);
            } else if (turns & 4) {
                ep = a[2];
                em = orb_c<C2>(-a[2].x, -a[2].y);
            }
            if ((turns & 10) == 10) {
                op = orb_c<C2>(a[1].x + a[3].x, a[1].y + a[3].y);
                om = orb_c<C2>(a[1].x - a[3].x, a[1].y - a[3].y);
            } else if (turns & 8) {
                op = a[3];
                om = orb_c<C2>(-a[3].x, -a[3].y);
            }
            C2 h0 = ep, h1 = em, h2 = ep, h3 = em;
            if (even && odd) {
                h0 = orb_c<C2>(ep.x + op.x, ep.y + op.y);
                h2 = orb_c<C2>(ep.x - op.x, ep.y - op.y);
                h1 = orb_c<C2>(em.x + om.y, em.y - om.x);  // em - i om
                h3 = orb_c<C2>(em.x - om.y, em.y + om.x);  // em + i om
            } else if (odd) {
                h0 = op;
                h2 = orb_c<C2>(-op.x, -op.y);
                h1 = orb_c<C2>(om.y, -om.x);
                h3 = orb_c<C2>(-om.y, om.x);
            }
            C2 *hb = h + b * p + k;
            hb[0] = h0;
            hb[js] = h1;
            hb[2 * js] = h2;
            hb[3 * js] = h3;
        }
        __syncthreads();
        if (NI == 1 && act && tid < rows * p) load(__ffs(act) - 1, it_b[0], it_m[0], ahead);
        C2 s[NI];
        int off[NI][4];  // H_{(k + m + ex) mod 4} of k = 0..3
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            s[i] = orb_c<C2>(R(0), R(0));
#pragma unroll
            for (int q = 0; q < 4; ++q)
                off[i][q] = ((it_m[i] + ex + q) & 3) * js + it_b[i] * p + q;
        }
        auto step = [&](int k0, int q) {
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const C2 v = h[off[i][q] + k0];
                const R r = rm[(k0 + q) * p + it_m[i]];
                s[i].x = fma(r, v.x, s[i].x);
                s[i].y = fma(r, v.y, s[i].y);
            }
        };
        int k0 = 0;
        for (; k0 + 4 <= p; k0 += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q) step(k0, q);
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (k0 + q < p) step(k0, q);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const C2 w = pw[o * (p + 1) + it_m[i] + ex];
            if (real_pw) {
                acc[i].x = fma(w.x, s[i].x, acc[i].x);
                acc[i].y = fma(w.x, s[i].y, acc[i].y);
            } else {
                acc[i] = orb_fma(w, s[i], acc[i]);
            }
            if (lap && it_m[i] == 0) {
                acc[i].x += lsum[it_b[i]].x;
                acc[i].y += lsum[it_b[i]].y;
            }
        }
    }
    C2 *dst = le + d.eoff + lvl_off(l) * p;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int64_t b = p0 + it_b[i];
        if (tid + i * ORB_THREADS >= rows * p || b >= np) continue;
        const uint32_t ix = 2 * compact_bits(uint32_t(b)) + uint32_t(c & 1),
                       iy = 2 * compact_bits(uint32_t(b) >> 1) + uint32_t(c >> 1);
        dst[box_index(l, ix, iy) * p + it_m[i]] = acc[i];
    }
}

size_t m2l_orbit_smem(int p, int ni, bool fp64) {
    const size_t rows = size_t(orb_rows(p, ni)), r = fp64 ? 8 : 4;
    return (4 * (rows * p + 1) + size_t(ORBITS) * (p + 1) + ORBITS * 4 + rows) * 2 * r +
           size_t(p) * p * r + size_t(ORBITS) * 4 * rows * sizeof(int);
}

template <typename R>
cudaError_t launch_m2l_orbits(const Task *tasks, int ntasks, int64_t nblocks, int ni, size_t smem,
                              const InstDesc *insts, const uint32_t *start,
                              const typename Cplx<R>::T *me, typename Cplx<R>::T *le,
                              cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    auto *k = k_m2l_orbits<R, 1>;
    if (sizeof(R) == 8 && ni != 1) k = k_m2l_orbits<R, sizeof(R) == 8 ? M2L_ORBIT_NI_MAX : 1>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    k<<<unsigned(nblocks), ORB_THREADS, smem, st>>>(tasks, ntasks, insts, start, me, le);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}
template cudaError_t launch_m2l_orbits<double>(const Task *, int, int64_t, int, size_t,
                                               const InstDesc *, const uint32_t *, const double2 *,
                                               double2 *, cudaStream_t, uint64_t *);
template cudaError_t launch_m2l_orbits<float>(const Task *, int, int64_t, int, size_t,
                                              const InstDesc *, const uint32_t *, const float2 *,
                                              float2 *, cudaStream_t, uint64_t *);

PF_DEFINE_CHECK_READER(orbits)

}  // namespace petfmm
