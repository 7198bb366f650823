// m2l64.cu -- M2L of the FP64 path (vortex kernel, Sec. 2.2).
//
// c^_m = sum_delta sum_k R[k][m] delta^-(k+m+1) a~_k, R[k][m] = (-1)^(k+1)
// C(k+m, k), over the 27 offsets delta of the interaction list.  The FP64
// pipe of this part (two lanes a cycle and SM) bounds it, so the operations
// are cut and no lane idles:
//  - Offsets that are quarter turns of one another, delta = i^r delta_0, share
//    one product: with H_j[k] = sum_r i^(-r j) a~_k^(r) (a four-point Fourier
//    sum, additions only) their part is sum_k R[k][m] delta_0^-(k+m+1)
//    H_{(k+m+1) mod 4}[k].  The 27 offsets form 10 such orbits.
//  - delta_0^-k is applied to the sources and delta_0^-(m+1) to the sum, so
//    the product itself is a real matrix on complex vectors, the same R for
//    every orbit: 2 p^2 FP64 operations instead of 4 p^2.
// At p = 17 an interior box takes about 9,500 operations against 31,200 for
// 27 complex products.  A block takes a run of consecutive (z-order) parent
// cells' children of one class; its (box, coefficient) pairs lie flat over
// the threads.  Measured on one GB300, against a
// warp per box with 27 complex products: 1,048,576 blobs, L = 8, p = 17: 13.8 ->
// 1.9 ms; 10,000 blobs, L = 4, p = 12: 0.56 -> 0.042 ms.
#include <cmath>
#include <vector>

#include "kernels.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

namespace {

constexpr int M64_THREADS = 128;
constexpr int M64_ORBITS = 10;
// representatives of the orbits, as (dx, dy) = source - target
__constant__ int8_t c_orbit[M64_ORBITS][2] = {{2, 0}, {2, 1}, {2, -1}, {2, 2}, {3, 0},
                                              {3, 1}, {3, -1}, {3, 2}, {3, -2}, {3, 3}};
const int kOrbit[M64_ORBITS][2] = {{2, 0}, {2, 1}, {2, -1}, {2, 2}, {3, 0},
                                   {3, 1}, {3, -1}, {3, 2}, {3, -2}, {3, 3}};

__host__ __device__ __forceinline__ int m64_rows(int p, int ni) { return M64_THREADS * ni / p; }

// delta_0 turned by r quarter turns
__device__ __forceinline__ void turned(int o, int r, int *dx, int *dy) {
    const int x = c_orbit[o][0], y = c_orbit[o][1];
    *dx = r == 0 ? x : r == 1 ? -y : r == 2 ? -x : y;
    *dy = r == 0 ? y : r == 1 ? x : r == 2 ? -y : -x;
}

// The complex products with their roundings spelled out: the two instances
// of the kernel must give the same bits (a batch and a tree alone).
__device__ __forceinline__ double2 mul64(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 fma64(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

}  // namespace

// R (p x p, [k][m]) then, per orbit, delta_0^-j for j = 0..p as complex.
void host_m2l64_table(int p, std::vector<double> &out) {
    out.assign(size_t(p) * p + size_t(M64_ORBITS) * (p + 1) * 2, 0.0);
    for (int k = 0; k < p; ++k)
        for (int m = 0; m < p; ++m) {
            double c = 1.0;  // C(k + m, k)
            for (int i = 1; i <= k; ++i) c = c * double(m + i) / double(i);
            out[size_t(k) * p + m] = (k & 1) ? std::nearbyint(c) : -std::nearbyint(c);
        }
    double *pw = out.data() + size_t(p) * p;
    for (int o = 0; o < M64_ORBITS; ++o) {
        const long double x = kOrbit[o][0], y = kOrbit[o][1], n = x * x + y * y;
        long double re = 1.0L, im = 0.0L;
        for (int j = 0; j <= p; ++j) {
            pw[(size_t(o) * (p + 1) + j) * 2] = double(re);
            pw[(size_t(o) * (p + 1) + j) * 2 + 1] = double(im);
            const long double t = (re * x + im * y) / n;  // times 1 / delta_0
            im = (im * x - re * y) / n;
            re = t;
        }
    }
}

int64_t m2l64_units(int p, int level, int ni) {
    const int64_t np = int64_t(1) << (2 * (level - 1));
    const int rows = m64_rows(p, ni);
    return (np + rows - 1) / rows * 4;
}

template <int NI>
__global__ void __launch_bounds__(M64_THREADS) k_m2l64(const Task *__restrict__ tasks, int ntasks,
                                                       const InstDesc *__restrict__ insts,
                                                       const uint32_t *__restrict__ start,
                                                       const double2 *__restrict__ me,
                                                       double2 *__restrict__ le) {
    extern __shared__ __align__(16) unsigned char m64_smem[];
    const int tid = threadIdx.x;
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const InstDesc &d = insts[t.inst];
    const int p = d.p, l = t.level, nside = 1 << l;
    const int rows = m64_rows(p, NI), js = rows * p + 1;  // one of padding: four H, four banks
    const int64_t unit = int64_t(blockIdx.x) - t.block0;
    const int c = int(unit & 3);
    const int64_t np = int64_t(1) << (2 * (l - 1)), p0 = (unit >> 2) * rows;
    double2 *h = reinterpret_cast<double2 *>(m64_smem);  // [4][js]
    double2 *pw = h + 4 * js;                             // [orbit][p + 1]
    double *rm = reinterpret_cast<double *>(pw + M64_ORBITS * (p + 1));  // [k][m]
    int *srow = reinterpret_cast<int *>(rm + p * p);      // [box][turn]
    const uint32_t *st = start + d.soff;
    bool mine = false;
    for (int b = tid; b < rows; b += M64_THREADS)
        if (p0 + b < np) mine |= box_count(st, d.L, l, uint32_t((p0 + b) * 4 + c)) != 0;
    if (!__syncthreads_or(mine)) return;  // no target box holds particles
    const double *tab = static_cast<const double *>(d.t_m2l);
    for (int i = tid; i < p * p; i += M64_THREADS) rm[i] = tab[i];
    for (int i = tid; i < M64_ORBITS * (p + 1); i += M64_THREADS)
        pw[i] = make_double2(tab[p * p + 2 * i], tab[p * p + 2 * i + 1]);
    int it_b[NI], it_m[NI];
    double2 acc[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int e = tid + i * M64_THREADS;
        const bool in = e < rows * p;
        it_b[i] = in ? e / p : 0;
        it_m[i] = in ? e % p : 0;
        acc[i] = make_double2(0.0, 0.0);
    }
    const double2 *lev = me + d.eoff + lvl_off(l) * p;
    const int lo_x = (c & 1) ? -3 : -2, lo_y = (c >> 1) ? -3 : -2;
    for (int o = 0; o < M64_ORBITS; ++o) {
        // the turns of this orbit in the class's interaction list
        int turns = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            int dx, dy;
            turned(o, r, &dx, &dy);
            if (dx >= lo_x && dx <= lo_x + 5 && dy >= lo_y && dy <= lo_y + 5) turns |= 1 << r;
        }
        __syncthreads();  // the previous orbit's products are done
        bool have = false;
        for (int e = tid; e < 4 * rows; e += M64_THREADS) {
            const int r = e & 3;
            const int64_t b = p0 + (e >> 2);
            int src = -1;
            if (b < np && ((turns >> r) & 1)) {
                int dx, dy;
                turned(o, r, &dx, &dy);
                const int sx = 2 * int(compact_bits(uint32_t(b))) + (c & 1) + dx;
                const int sy = 2 * int(compact_bits(uint32_t(b) >> 1)) + (c >> 1) + dy;
                if (sx >= 0 && sy >= 0 && sx < nside && sy < nside &&
                    box_count(st, d.L, l, morton_key(uint32_t(sx), uint32_t(sy))))
                    src = int(box_index(l, uint32_t(sx), uint32_t(sy)));
            }
            srow[e] = src;
            have |= src >= 0;
        }
        if (!__syncthreads_or(have)) continue;
        const bool real_pw = c_orbit[o][1] == 0;
        const bool even = (turns & 5) != 0, odd = (turns & 10) != 0;
        for (int e = tid; e < rows * p; e += M64_THREADS) {
            const int b = e / p, k = e - b * p;
            const double2 w = pw[o * (p + 1) + k];
            double2 a[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int s = srow[4 * b + r];
                a[r] = s >= 0 ? lev[int64_t(s) * p + k] : make_double2(0.0, 0.0);
                if ((turns >> r) & 1)
                    a[r] = real_pw ? make_double2(a[r].x * w.x, a[r].y * w.x) : mul64(a[r], w);
            }
            // sums and differences of opposite turns (of one alone: itself)
            double2 ep = a[0], em = a[0], op = a[1], om = a[1];
            if ((turns & 5) == 5) {
                ep = make_double2(a[0].x + a[2].x, a[0].y + a[2].y);
                em = make_double2(a[0].x - a[2].x, a[0].y - a[2].y);
            } else if (turns & 4) {
                ep = a[2];
                em = make_double2(-a[2].x, -a[2].y);
            }
            if ((turns & 10) == 10) {
                op = make_double2(a[1].x + a[3].x, a[1].y + a[3].y);
                om = make_double2(a[1].x - a[3].x, a[1].y - a[3].y);
            } else if (turns & 8) {
                op = a[3];
                om = make_double2(-a[3].x, -a[3].y);
            }
            double2 h0 = ep, h1 = em, h2 = ep, h3 = em;
            if (even && odd) {
                h0 = make_double2(ep.x + op.x, ep.y + op.y);
                h2 = make_double2(ep.x - op.x, ep.y - op.y);
                h1 = make_double2(em.x + om.y, em.y - om.x);  // em - i om
                h3 = make_double2(em.x - om.y, em.y + om.x);  // em + i om
            } else if (odd) {
                h0 = op;
                h2 = make_double2(-op.x, -op.y);
                h1 = make_double2(om.y, -om.x);
                h3 = make_double2(-om.y, om.x);
            }
            h[e] = h0;
            h[js + e] = h1;
            h[2 * js + e] = h2;
            h[3 * js + e] = h3;
        }
        __syncthreads();
        double2 s[NI];
        int ha[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            s[i] = make_double2(0.0, 0.0);
            ha[i] = it_b[i] * p;
        }
#pragma unroll 2
        for (int k = 0; k < p; ++k)
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const double2 v = h[((k + it_m[i] + 1) & 3) * js + ha[i] + k];
                const double r = rm[k * p + it_m[i]];
                s[i].x = fma(r, v.x, s[i].x);
                s[i].y = fma(r, v.y, s[i].y);
            }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const double2 w = pw[o * (p + 1) + it_m[i] + 1];
            if (real_pw) {
                acc[i].x = fma(w.x, s[i].x, acc[i].x);
                acc[i].y = fma(w.x, s[i].y, acc[i].y);
            } else {
                acc[i] = fma64(w, s[i], acc[i]);
            }
        }
    }
    double2 *dst = le + d.eoff + lvl_off(l) * p;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int64_t b = p0 + it_b[i];
        if (tid + i * M64_THREADS >= rows * p || b >= np) continue;
        const uint32_t ix = 2 * compact_bits(uint32_t(b)) + uint32_t(c & 1),
                       iy = 2 * compact_bits(uint32_t(b) >> 1) + uint32_t(c >> 1);
        dst[box_index(l, ix, iy) * p + it_m[i]] = acc[i];
    }
}

size_t m2l64_smem(int p, int ni) {
    const size_t rows = size_t(m64_rows(p, ni));
    return 4 * (rows * p + 1) * 16 + size_t(M64_ORBITS) * (p + 1) * 16 + size_t(p) * p * 8 +
           4 * rows * sizeof(int);
}

template <int NI>
static cudaError_t m2l64_launch(const Task *tasks, int ntasks, int64_t nblocks,
                                const InstDesc *insts, const uint32_t *start, const double2 *me,
                                double2 *le, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_m2l64<NI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(smem));
    if (e != cudaSuccess) return e;
    k_m2l64<NI><<<unsigned(nblocks), M64_THREADS, smem, st>>>(tasks, ntasks, insts, start, me, le);
    return cudaGetLastError();
}

cudaError_t launch_m2l64(const Task *tasks, int ntasks, int64_t nblocks, int ni, size_t smem,
                         const InstDesc *insts, const uint32_t *start, const double2 *me,
                         double2 *le, cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    PF_LAUNCHED(1);
    return ni == 1 ? m2l64_launch<1>(tasks, ntasks, nblocks, insts, start, me, le, smem, st)
                   : m2l64_launch<M2L64_NI_MAX>(tasks, ntasks, nblocks, insts, start, me, le, smem, st);
}

}  // namespace petfmm
