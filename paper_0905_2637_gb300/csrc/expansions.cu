// expansions.cu -- the upward and downward sweeps of Sec. 2.2 (Fig. 2):
// P2M, the per-box M2L of the mixed path's sparse units, and the operator
// tables of all translations (M2M and L2L: shifts.cu; the other M2L kernels:
// m2l_tc.cu, m2l_orbits.cu).
//
// Series (Cauchy kernel; the paper leaves the mathematics to Greengard-
// Rokhlin, Sec. 2.2).  With z = x + i y, the far field is
// w(z) = sum_j gamma_j / (z - z_j) and (u, v) = (Im w, Re w) / 2pi.  Rescaled
// coefficients, r = width of the box that owns the expansion:
//   P2M  a~_k = sum_j gamma_j zeta_j^k,       zeta_j = (z_j - z_c) / r
//   M2M  a~'_l = 2^-l sum_{k<=l} C(l,k) e^(l-k) a~_k,  e = (child - parent
//        centre) / r_child in {+-1/2 +- i/2}
//   M2L  c^_m = sum_k (-1)^(k+1) C(k+m,k) delta^-(k+m+1) a~_k,  delta = (source
//        - target centre) / r, one of 40 fixed offsets
//   L2L  c^'_n = sum_{m>=n} 2^-(m+1) C(m,n) e^(m-n) c^_m
//   L2P  w(z) = r^-1 sum_m c^_m zeta^m
// Costs (Sec. 5.2): P2M O(N_i p) per leaf, M2M and L2L O(p^2) per child,
// M2L O(p^2 n_IL) per box with n_IL <= 27.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <utility>
#include <vector>

#include "kernels.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

// ----------------------------------------------------------------------------
// Interaction-list table.  For a target of child class c = (cx, cy) the
// sources are the children of the parent's 3x3 neighbourhood that are not
// within one box of the target: per axis dx in [-2, 3] if cx = 0 and [-3, 2]
// if cx = 1 (same for y), minus the 3x3 block around the target -- 27
// offsets.  Each offset maps to one of the 40 vectors of [-3, 3]^2 \ [-1, 1]^2.
// ----------------------------------------------------------------------------
struct IlTable {
    IlEntry e[4][27];
};
constexpr IlTable il_table() {
    IlTable t{};
    for (int c = 0; c < 4; ++c) {
        const int x_lo = (c & 1) ? -3 : -2, y_lo = (c >> 1) ? -3 : -2;
        int n = 0;
        for (int dy = y_lo; dy <= y_lo + 5; ++dy)
            for (int dx = x_lo; dx <= x_lo + 5; ++dx) {
                if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1) continue;
                t.e[c][n].dx = int8_t(dx);
                t.e[c][n].dy = int8_t(dy);
                t.e[c][n].op = int8_t(m2l_op_index(dx, dy));
                ++n;
            }
    }
    return t;
}
static constexpr IlTable kIl = il_table();
__constant__ IlTable c_il = il_table();

int host_interaction_list(int level, int ix, int iy, int32_t *out) {
    if (level < 0 || level > MAX_L) return -1;
    const int nside = 1 << level;
    if (ix < 0 || iy < 0 || ix >= nside || iy >= nside) return -1;
    if (level < 2) return 0;
    const IlEntry *e = kIl.e[(ix & 1) | ((iy & 1) << 1)];
    int n = 0;
    for (int i = 0; i < 27; ++i) {
        const int sx = ix + e[i].dx, sy = iy + e[i].dy;
        if (sx < 0 || sy < 0 || sx >= nside || sy >= nside) continue;
        out[2 * n] = sx;
        out[2 * n + 1] = sy;
        ++n;
    }
    return n;
}

int64_t m2l_pair_count(int L) {
    int64_t tot = 0;
    for (int l = 2; l <= L; ++l) {
        const int64_t n = int64_t(1) << l;
        tot += (6 * n - 8) * (6 * n - 8) - (3 * n - 2) * (3 * n - 2);
    }
    return tot;
}

// ----------------------------------------------------------------------------
// Operator tables, built in FP64 on the host.
// ----------------------------------------------------------------------------
struct HC { double re, im; };
static HC hmul(HC a, HC b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }

static std::vector<double> binomials(int nmax) {
    // Pascal's triangle, nmax + 1 rows
    std::vector<double> c(size_t(nmax + 1) * (nmax + 1), 0.0);
    for (int n = 0; n <= nmax; ++n) {
        c[size_t(n) * (nmax + 1)] = 1.0;
        for (int k = 1; k <= n; ++k)
            c[size_t(n) * (nmax + 1) + k] =
                c[size_t(n - 1) * (nmax + 1) + k - 1] + (k <= n - 1 ? c[size_t(n - 1) * (nmax + 1) + k] : 0.0);
    }
    return c;
}

void host_m2l_table(int p, double *out) {
    const int nb = 2 * p;
    std::vector<double> C = binomials(nb);
    auto binom = [&](int n, int k) { return C[size_t(n) * (nb + 1) + k]; };
    int op = 0;
    for (int y = -3; y <= 3; ++y)
        for (int x = -3; x <= 3; ++x) {
            if (x >= -1 && x <= 1 && y >= -1 && y <= 1) continue;
            // powers of 1/delta
            const double den = double(x) * x + double(y) * y;
            const HC inv = {double(x) / den, -double(y) / den};
            std::vector<HC> ip(size_t(2 * p + 1));
            ip[0] = {1.0, 0.0};
            for (int i = 1; i <= 2 * p; ++i) ip[i] = hmul(ip[i - 1], inv);
            for (int k = 0; k < p; ++k)
                for (int m = 0; m < p; ++m) {
                    const double s = ((k & 1) ? 1.0 : -1.0) * binom(k + m, k);
                    const HC t = ip[k + m + 1];
                    double *o = out + ((size_t(op) * p + k) * p + m) * 2;
                    o[0] = s * t.re;
                    o[1] = s * t.im;
                }
            ++op;
        }
}

static void host_m2m_table(int p, double *out /* [c][l][k] */) {
    std::vector<double> C = binomials(p);
    for (int c = 0; c < 4; ++c) {
        const HC e = {(c & 1) - 0.5, (c >> 1) - 0.5};
        std::vector<HC> ep(size_t(p + 1));
        ep[0] = {1.0, 0.0};
        for (int i = 1; i <= p; ++i) ep[i] = hmul(ep[i - 1], e);
        for (int l = 0; l < p; ++l)
            for (int k = 0; k < p; ++k) {
                double *o = out + ((size_t(c) * p + l) * p + k) * 2;
                if (k > l) { o[0] = o[1] = 0.0; continue; }
                const double s = std::ldexp(C[size_t(l) * (p + 1) + k], -l);
                o[0] = s * ep[l - k].re;
                o[1] = s * ep[l - k].im;
            }
    }
}

static void host_l2l_table(int p, double *out /* [c][n][m] */) {
    std::vector<double> C = binomials(p);
    for (int c = 0; c < 4; ++c) {
        const HC e = {(c & 1) - 0.5, (c >> 1) - 0.5};
        std::vector<HC> ep(size_t(p + 1));
        ep[0] = {1.0, 0.0};
        for (int i = 1; i <= p; ++i) ep[i] = hmul(ep[i - 1], e);
        for (int n = 0; n < p; ++n)
            for (int m = 0; m < p; ++m) {
                double *o = out + ((size_t(c) * p + n) * p + m) * 2;
                if (m < n) { o[0] = o[1] = 0.0; continue; }
                const double s = std::ldexp(C[size_t(m) * (p + 1) + n], -(m + 1));
                o[0] = s * ep[m - n].re;
                o[1] = s * ep[m - n].im;
            }
    }
}

// Laplace kernel (log potential), rescaled like the Cauchy series: ME
// a~_0 = a_0, a~_k = a_k / w^k; LE b^_m = b_m w^m (w the box width).  With
// e the child centre's offset from the parent's in child widths and delta the
// source centre's offset from the target's in box widths, the translations
// do not depend on the level, except the constant of M2L, whose a_0 log w
// term the M2L kernel adds.
//   M2M  [c][l][k]: l = 0: a~_0; l >= 1: -a~_0 e^l / (l 2^l)
//                   + sum_{1<=k<=l} C(l-1, k-1) e^(l-k) 2^-l a~_k
//   L2L  [c][n][m]: C(m, n) e^(m-n) 2^-m, m >= n
//   M2L  [op][k][m]: k = 0: m = 0 log(-delta), m >= 1 -1 / (m delta^m);
//                   k >= 1: (-1)^k C(m+k-1, k-1) / delta^(k+m)
static void host_lap_m2m_table(int p, double *out /* [c][l][k] */) {
    std::vector<double> C = binomials(p);
    for (int c = 0; c < 4; ++c) {
        const HC e = {(c & 1) - 0.5, (c >> 1) - 0.5};
        std::vector<HC> ep(size_t(p + 1));
        ep[0] = {1.0, 0.0};
        for (int i = 1; i <= p; ++i) ep[i] = hmul(ep[i - 1], e);
        for (int l = 0; l < p; ++l)
            for (int k = 0; k < p; ++k) {
                double *o = out + ((size_t(c) * p + l) * p + k) * 2;
                o[0] = o[1] = 0.0;
                if (k > l) continue;
                if (l == 0) {
                    o[0] = 1.0;
                } else if (k == 0) {
                    const double s = -std::ldexp(1.0, -l) / double(l);
                    o[0] = s * ep[l].re;
                    o[1] = s * ep[l].im;
                } else {
                    const double s = std::ldexp(C[size_t(l - 1) * (p + 1) + k - 1], -l);
                    o[0] = s * ep[l - k].re;
                    o[1] = s * ep[l - k].im;
                }
            }
    }
}

static void host_lap_l2l_table(int p, double *out /* [c][n][m] */) {
    std::vector<double> C = binomials(p);
    for (int c = 0; c < 4; ++c) {
        const HC e = {(c & 1) - 0.5, (c >> 1) - 0.5};
        std::vector<HC> ep(size_t(p + 1));
        ep[0] = {1.0, 0.0};
        for (int i = 1; i <= p; ++i) ep[i] = hmul(ep[i - 1], e);
        for (int n = 0; n < p; ++n)
            for (int m = 0; m < p; ++m) {
                double *o = out + ((size_t(c) * p + n) * p + m) * 2;
                if (m < n) { o[0] = o[1] = 0.0; continue; }
                const double s = std::ldexp(C[size_t(m) * (p + 1) + n], -m);
                o[0] = s * ep[m - n].re;
                o[1] = s * ep[m - n].im;
            }
    }
}

void host_lap_m2l_table(int p, double *out /* [op][k][m] */) {
    const int nb = 2 * p;
    std::vector<double> C = binomials(nb);
    auto binom = [&](int n, int k) { return C[size_t(n) * (nb + 1) + k]; };
    int op = 0;
    for (int y = -3; y <= 3; ++y)
        for (int x = -3; x <= 3; ++x) {
            if (x >= -1 && x <= 1 && y >= -1 && y <= 1) continue;
            const double den = double(x) * x + double(y) * y;
            const HC inv = {double(x) / den, -double(y) / den};
            std::vector<HC> ip(size_t(2 * p + 1));
            ip[0] = {1.0, 0.0};
            for (int i = 1; i <= 2 * p; ++i) ip[i] = hmul(ip[i - 1], inv);
            for (int k = 0; k < p; ++k)
                for (int m = 0; m < p; ++m) {
                    double *o = out + ((size_t(op) * p + k) * p + m) * 2;
                    HC t;
                    if (k == 0 && m == 0) {
                        // log(-delta), principal branch (only Re enters the result)
                        t = {0.5 * std::log(den), std::atan2(-double(y), -double(x))};
                    } else if (k == 0) {
                        const double s = -1.0 / double(m);
                        t = {s * ip[m].re, s * ip[m].im};
                    } else {
                        const double s = ((k & 1) ? -1.0 : 1.0) * binom(m + k - 1, k - 1);
                        t = {s * ip[k + m].re, s * ip[k + m].im};
                    }
                    o[0] = t.re;
                    o[1] = t.im;
                }
            ++op;
        }
}

void host_op_table(int p, int kernel, int which, std::vector<double> &out) {
    const bool lap = kernel == KERNEL_LAPLACE;
    out.assign(size_t(which == 2 ? 40 : 4) * p * p * 2, 0.0);
    if (which == 0) (lap ? host_lap_m2m_table : host_m2m_table)(p, out.data());
    else if (which == 1) (lap ? host_lap_l2l_table : host_l2l_table)(p, out.data());
    else (lap ? host_lap_m2l_table : host_m2l_table)(p, out.data());
}

// A table on its stream, which the launches that use it follow.  The source goes
// with the caller's frame, and a device that reads pageable memory itself need
// not have it staged when the copy returns: wait for it.
cudaError_t copy_table(void *dst, const void *src, size_t bytes, cudaStream_t st) {
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaError_t build_op_tables(int p, int kernel, bool fp64, OpTables *t, cudaStream_t st) {
    t->p = p;
    std::vector<double> shift, orbit;
    host_shift_table(p, kernel, shift);
    host_m2l_orbit_table(p, kernel, orbit);
    // one allocation and one copy for all of them
    std::vector<float> shift32, orbit32, m2l32;
    struct Part {
        void **dst;
        const void *src;
        size_t bytes;
    };
    std::vector<Part> parts;
    if (fp64) {
        parts = {{(void **)&t->shift64, shift.data(), shift.size() * 8},
                 {(void **)&t->orbit64, orbit.data(), orbit.size() * 8}};
    } else {
        std::vector<double> m2l(size_t(2) * 40 * p * p);
        (kernel == KERNEL_LAPLACE ? host_lap_m2l_table : host_m2l_table)(p, m2l.data());
        shift32.assign(shift.begin(), shift.end());
        orbit32.assign(orbit.begin(), orbit.end());
        m2l32.assign(m2l.begin(), m2l.end());
        parts = {{(void **)&t->shift32, shift32.data(), shift32.size() * 4},
                 {(void **)&t->orbit32, orbit32.data(), orbit32.size() * 4},
                 {(void **)&t->m2l32, m2l32.data(), m2l32.size() * 4}};
    }
    size_t total = 0;
    for (const Part &x : parts) total += (x.bytes + 255) / 256 * 256;
    std::vector<unsigned char> blob(total);
    cudaError_t e = cudaMalloc(&t->blob, total);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    size_t at = 0;
    for (const Part &x : parts) {
        std::memcpy(blob.data() + at, x.src, x.bytes);
        *x.dst = static_cast<unsigned char *>(t->blob) + at;
        at += (x.bytes + 255) / 256 * 256;
    }
    return copy_table(t->blob, blob.data(), total, st);
}

cudaError_t build_tc_image(int kernel, bool blocks, OpTables *t, cudaStream_t st) {
    float *&dst = blocks ? t->m2l_tcb : t->m2l_tc;
    if (dst) return cudaSuccess;
    std::vector<float> img;
    (blocks ? host_m2l_tcb_images : host_m2l_tc_images)(t->p, kernel, img);
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, img.size() * 4);
    if (e == cudaSuccess) e = copy_table(p, img.data(), img.size() * 4, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        cudaFree(p);
    } else {
        dst = static_cast<float *>(p);
    }
    return e;
}

void free_op_tables(OpTables *t) {
    cudaFree(t->blob);
    cudaFree(t->m2l_tc);
    cudaFree(t->m2l_tcb);
    *t = OpTables();
}

// ----------------------------------------------------------------------------
// P2M: one warp per occupied leaf.  k_occ_list collects the occupied leaves
// (in no particular order); a persistent grid of warps strides over that
// list, so no block is spent on an empty leaf and the dense leaves of a
// cluster spread over all SMs.  Per leaf, lanes take 32 particles at a time,
// write the gamma * zeta^k powers to shared memory, and lane k sums column k
// in a fixed order: each leaf's expansion does not depend on which warp or
// in which order the leaves were processed.  Two leaves of at most 16 blobs
// share a warp: the FP64 pipe, two lanes a cycle and SM, bounds the FP64 path,
// and half of the lanes held no blob (1M blobs, 16 a leaf, p = 17: 583 -> 294
// us).
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_occ_list(const Task *__restrict__ tasks, int ntasks,
                                                  const InstDesc *__restrict__ insts,
                                                  const uint32_t *__restrict__ start,
                                                  uint2 *__restrict__ occ, uint32_t *ctrl) {
    const int lane = threadIdx.x & 31;
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    bool o = false;
    if (m < t.count) {
        const uint32_t *st = start + insts[t.inst].soff;
        o = st[m + 1] > st[m];
    }
    const uint32_t b = __ballot_sync(0xffffffffu, o);
    uint32_t base = 0;
    if (lane == 0 && b) base = atomicAdd(ctrl + CTRL_NOCC, uint32_t(__popc(b)));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (o) occ[base + __popc(b & ((1u << lane) - 1u))] = make_uint2(uint32_t(t.inst), uint32_t(m));
}

cudaError_t launch_occ_list(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, uint2 *occ, uint32_t *ctrl, cudaStream_t st,
                            uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_occ_list<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, occ, ctrl);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

template <typename R>
__device__ __forceinline__ typename Cplx<R>::T mk2(R a, R b) {
    typename Cplx<R>::T r;
    r.x = a;
    r.y = b;
    return r;
}

template <typename R>
__global__ void __launch_bounds__(P2M_WARPS * 32) k_p2m(
    const uint2 *__restrict__ occ, const uint32_t *ctrl, const InstDesc *__restrict__ insts,
    int pmax, const uint32_t *__restrict__ start, const double *__restrict__ xs,
    const double *__restrict__ ys, const double *__restrict__ gs, const float4 *__restrict__ rec,
    typename Cplx<R>::T *__restrict__ me) {
    using C2 = typename Cplx<R>::T;
    extern __shared__ unsigned char smem_raw[];
    C2 *buf = reinterpret_cast<C2 *>(smem_raw) + size_t(threadIdx.x >> 5) * 32 * pmax;
    const int lane = threadIdx.x & 31;
    const uint32_t nocc = ctrl[CTRL_NOCC];
    const uint32_t nwarps = gridDim.x * P2M_WARPS;
    // leaf range of occupied-leaf entry i (empty past the end, and in the
    // checked build when it lies outside its instance)
    auto range = [&](uint32_t i, uint2 &e, uint32_t &s0, uint32_t &s1) {
        e = occ[min(i, nocc - 1)];
        const InstDesc &d = insts[e.x];
        s0 = start[d.soff + e.y];
        s1 = i < nocc ? start[d.soff + e.y + 1] : s0;
        if (!(PF_IN(e.y, int64_t(1) << (2 * d.L)) && PF_IN(int64_t(s0) - d.poff, d.n + 1) &&
              PF_IN(int64_t(s1) - d.poff, d.n + 1)) || s1 < s0)
            s1 = s0;
    };
    // gamma zeta^k of sorted blob j (nothing from end on) in this lane's row;
    // Laplace: q, then -q zeta^k / k.  (Explicit multiply-adds: the same bits
    // wherever this is inlined.)
    auto powers = [&](const InstDesc &d, uint32_t leaf, uint32_t j, uint32_t end) {
        C2 z = mk2<R>(R(0), R(0)), w = z;
        if (j < end) {
            if (rec) {
                const float4 r = rec[j];
                z = mk2<R>(R(r.x), R(r.y));
                w = mk2<R>(R(r.z), R(0));
            } else {
                const double cx = fma(double(compact_bits(leaf)) + 0.5, d.wleaf, d.x0);
                const double cy = fma(double(compact_bits(leaf >> 1)) + 0.5, d.wleaf, d.y0);
                z = mk2<R>(R((xs[j] - cx) * d.scale), R((ys[j] - cy) * d.scale));
                w = mk2<R>(R(gs[j]), R(0));
            }
        }
        const bool lap = d.kernel == KERNEL_LAPLACE;
        for (int k = 0; k < d.p; ++k) {
            C2 wk = w;
            if (lap && k) {
                const R s = R(-1) / R(k);
                wk = mk2<R>(w.x * s, w.y * s);
            }
            buf[lane * pmax + k] = wk;
            w = mk2<R>(fma(w.x, z.x, -(w.y * z.y)), fma(w.x, z.y, w.y * z.x));
        }
    };
    auto add_rows = [&](C2 &acc, int k, int row, uint32_t rows) {
#pragma unroll 4
        for (uint32_t q = 0; q < rows; ++q) {
            const C2 b = buf[(row + q) * pmax + k];
            acc.x += b.x;
            acc.y += b.y;
        }
    };
    auto series = [&](const InstDesc &d, uint32_t leaf) {
        return me + d.eoff +
               (lvl_off(d.L) + box_index(d.L, compact_bits(leaf), compact_bits(leaf >> 1))) * d.p;
    };
    // two entries at a time once there are more than warps
    const uint32_t per = nocc > nwarps ? 2 : 1;
    for (uint32_t i = per * (blockIdx.x * P2M_WARPS + (threadIdx.x >> 5)); i < nocc;
         i += per * nwarps) {
        uint2 e[2];
        uint32_t s0[2], s1[2];
        range(i, e[0], s0[0], s1[0]);
        range(per == 2 ? i + 1 : nocc, e[1], s0[1], s1[1]);
        if (per == 2 && s1[0] - s0[0] <= 16 && s1[1] - s0[1] <= 16) {
            // a half-warp each
            const int h = lane >> 4;
            powers(insts[h ? e[1].x : e[0].x], h ? e[1].y : e[0].y,
                   (h ? s0[1] : s0[0]) + uint32_t(lane & 15), h ? s1[1] : s1[0]);
            __syncwarp();
            const int p0 = insts[e[0].x].p, cols = p0 + insts[e[1].x].p;
            for (int c = lane; c < cols; c += 32) {
                const int u = c >= p0, k = u ? c - p0 : c;
                const uint32_t rows = u ? s1[1] - s0[1] : s1[0] - s0[0];
                C2 acc = mk2<R>(R(0), R(0));
                add_rows(acc, k, 16 * u, rows);
                if (!u || i + 1 < nocc) series(insts[u ? e[1].x : e[0].x], u ? e[1].y : e[0].y)[k] = acc;
            }
            __syncwarp();
            continue;
        }
        for (uint32_t u = 0; u < per && i + u < nocc; ++u) {
            const InstDesc &d = insts[e[u].x];
            C2 acc0 = mk2<R>(R(0), R(0)), acc1 = acc0;
            for (uint32_t c0 = s0[u]; c0 < s1[u]; c0 += 32) {
                const uint32_t rows = min(32u, s1[u] - c0);
                powers(d, e[u].y, c0 + uint32_t(lane), s1[u]);
                __syncwarp();
                if (lane < d.p) add_rows(acc0, lane, 0, rows);
                if (lane + 32 < d.p) add_rows(acc1, lane + 32, 0, rows);
                __syncwarp();
            }
            C2 *dst = series(d, e[u].y);
            if (lane < d.p) dst[lane] = acc0;
            if (lane + 32 < d.p) dst[lane + 32] = acc1;
        }
    }
}

// Leaves of at most this many blobs are summed by one lane each (k_p2m_reg).
constexpr uint32_t P2M_LANE_MAX = 16;

// Mixed path, p <= PM: each lane keeps the running sums of its particles'
// gamma zeta^k in registers over all chunks of the leaf, and the warp adds
// the 32 lanes' sums once per leaf (transposed through shared memory, lane k
// adding column k: even rows and odd rows separately, then the two).  About a
// third of the instructions of the per-chunk transpose above.
// Bound by latency.  765k leaves of one blob, p = 17: 41 us; 200 us when each
// lane wrote its leaf's coefficients by itself (32 rows a store instruction,
// 60 us of it) and each warp looked its larger leaves up one by one (100 us).
template <int PM>
__global__ void __launch_bounds__(P2M_WARPS * 32) k_p2m_reg(
    const uint2 *__restrict__ occ, const uint32_t *ctrl, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const float4 *__restrict__ rec, float2 *__restrict__ me) {
    constexpr int SP = PM | 1;  // odd row stride: conflict-free 8-byte accesses
    __shared__ float2 buf[P2M_WARPS][32 * SP];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t nocc = ctrl[CTRL_NOCC];
    const uint32_t gw = blockIdx.x * P2M_WARPS + wid, nwarps = gridDim.x * P2M_WARPS;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // leaf range of occupied-leaf entry i (empty in the checked build when
    // it lies outside its instance)
    auto range = [&](uint32_t i, const InstDesc *&dp, uint32_t &m, uint32_t &s0, uint32_t &s1) {
        const uint2 e = occ[i];
        dp = insts + e.x;
        m = e.y;
        s0 = start[dp->soff + m];
        s1 = start[dp->soff + m + 1];
        if (!(PF_IN(m, int64_t(1) << (2 * dp->L)) && PF_IN(int64_t(s0) - dp->poff, dp->n + 1) &&
              PF_IN(int64_t(s1) - dp->poff, dp->n + 1)) || s1 < s0)
            s1 = s0;
    };
    // 1. Leaves of at most P2M_LANE_MAX blobs, one per lane, 32 entries per
    //    warp at a time: the lane sums its few blobs' series by itself and
    //    the warp writes the 32 leaves' coefficients (a warp and a 32-row
    //    reduction per leaf of one or a few blobs would be mostly idle).
    for (uint32_t base = gw * 32; base < nocc; base += nwarps * 32) {
        const uint32_t i = base + lane;
        const InstDesc *dp = nullptr;
        uint32_t m = 0, s0 = 0, s1 = 0;
        if (i < nocc) range(i, dp, m, s0, s1);
        const bool mine = s1 > s0 && s1 - s0 <= P2M_LANE_MAX;
        int p = 0;
        float2 *dst = nullptr;
        if (mine) {
            const InstDesc &d = *dp;
            p = d.p;
            float2 acc[PM];
#pragma unroll
            for (int k = 0; k < PM; ++k) acc[k] = make_float2(0.f, 0.f);
            for (uint32_t j = s0; j < s1; ++j) {
                const float4 r = rec[j];
                float2 w = make_float2(r.z, 0.f);
                const float2 z = make_float2(r.x, r.y);
#pragma unroll
                for (int k = 0; k < PM; ++k) {
                    if (k < p) {
                        acc[k].x += w.x;
                        acc[k].y += w.y;
                        w = cmul(w, z);
                    }
                }
            }
            const uint32_t ix = compact_bits(m), iy = compact_bits(m >> 1);
            dst = me + d.eoff + (lvl_off(d.L) + box_index(d.L, ix, iy)) * p;
            const bool lap = d.kernel == KERNEL_LAPLACE;
#pragma unroll
            for (int k = 0; k < PM; ++k) {
                if (k < p) {
                    // Laplace kernel: a_k = -(1/k) sum q zeta^k for k >= 1
                    const float sc = (lap && k) ? -1.0f / float(k) : 1.0f;
                    buf[wid][lane * SP + k] = make_float2(sc * acc[k].x, sc * acc[k].y);
                }
            }
        }
        __syncwarp();
        // the 32 leaves' coefficients as one run: consecutive lanes write
        // consecutive coefficients of a leaf
        const int pw = __reduce_max_sync(0xffffffffu, p);
        const uint64_t dst64 = reinterpret_cast<uint64_t>(dst);
        for (int q = 0, e = lane; q < pw; ++q, e += 32) {
            const int leaf = e / pw, k = e - leaf * pw;
            const uint64_t to = __shfl_sync(0xffffffffu, dst64, leaf);
            const int pl = __shfl_sync(0xffffffffu, p, leaf);
            if (k < pl) reinterpret_cast<float2 *>(to)[k] = buf[wid][leaf * SP + k];
        }
        __syncwarp();
    }
    // 2. Larger leaves, one per warp, entry i by warp i mod nwarps so that a
    //    cluster's leaves spread over all of them; the lanes look up 32 of the
    //    warp's entries at a time.
    for (uint64_t base = gw; base < nocc; base += uint64_t(nwarps) * 32) {
        const uint64_t mine = base + uint64_t(nwarps) * lane;
        const InstDesc *dp = nullptr;
        uint32_t m = 0, s0 = 0, s1 = 0;
        if (mine < nocc) range(uint32_t(mine), dp, m, s0, s1);
        uint32_t todo = __ballot_sync(0xffffffffu, s1 > s0 && s1 - s0 > P2M_LANE_MAX);
        for (; todo; todo &= todo - 1) {
            range(uint32_t(base + uint64_t(nwarps) * (__ffs(todo) - 1)), dp, m, s0, s1);
            const InstDesc &d = *dp;
            const int p = d.p, L = d.L;
            float2 acc[PM];
#pragma unroll
            for (int k = 0; k < PM; ++k) acc[k] = make_float2(0.f, 0.f);
            // Leaves of more than 32 blobs: two blobs per lane per step (two
            // independent power chains), and the next step's two records
            // requested before this step's arithmetic: up to four 16-byte loads
            // in flight per lane.  Smaller leaves take one step of one blob per
            // lane (a second chain would only add padding).
            if (s1 - s0 <= 32) {
                const float4 r = s0 + lane < s1 ? rec[s0 + lane] : z4;
                float2 w = make_float2(r.z, 0.f);
                const float2 z = make_float2(r.x, r.y);
#pragma unroll
                for (int k = 0; k < PM; ++k) {
                    if (k < p) {
                        acc[k].x += w.x;
                        acc[k].y += w.y;
                        w = cmul(w, z);
                    }
                }
            }
            float4 na = z4, nb = z4;
            if (s1 - s0 > 32) {
                na = rec[s0 + lane];
                nb = s0 + 32 + lane < s1 ? rec[s0 + 32 + lane] : z4;
            }
            for (uint32_t c0 = s0; s1 - s0 > 32 && c0 < s1; c0 += 64) {
                const float4 ra = na, rb = nb;
                const uint32_t jn = c0 + 64 + lane;
                na = jn < s1 ? rec[jn] : z4;
                nb = jn + 32 < s1 ? rec[jn + 32] : z4;
                float2 wa = make_float2(ra.z, 0.f), wb = make_float2(rb.z, 0.f);
                const float2 za = make_float2(ra.x, ra.y), zb = make_float2(rb.x, rb.y);
#pragma unroll
                for (int k = 0; k < PM; ++k) {
                    if (k < p) {
                        acc[k].x += wa.x;
                        acc[k].y += wa.y;
                        acc[k].x += wb.x;
                        acc[k].y += wb.y;
                        wa = cmul(wa, za);
                        wb = cmul(wb, zb);
                    }
                }
            }
            float2 *row = buf[wid] + lane * SP;
#pragma unroll
            for (int k = 0; k < PM; ++k)
                if (k < p) row[k] = acc[k];
            __syncwarp();
            if (lane < p) {
                float2 se = make_float2(0.f, 0.f), so = make_float2(0.f, 0.f);
#pragma unroll 4
                for (int q = 0; q < 32; q += 2) {
                    const float2 a = buf[wid][q * SP + lane], b = buf[wid][(q + 1) * SP + lane];
                    se.x += a.x;
                    se.y += a.y;
                    so.x += b.x;
                    so.y += b.y;
                }
                const uint32_t ix = compact_bits(m), iy = compact_bits(m >> 1);
                // Laplace kernel: a_k = -(1/k) sum q zeta^k for k >= 1
                const float s = (d.kernel == KERNEL_LAPLACE && lane) ? -1.0f / float(lane) : 1.0f;
                me[d.eoff + (lvl_off(L) + box_index(L, ix, iy)) * p + lane] =
                    make_float2(s * (se.x + so.x), s * (se.y + so.y));
            }
            __syncwarp();
        }
    }
}

template <int PM, typename C2>
cudaError_t launch_p2m_reg(const uint2 *occ, const uint32_t *ctrl, int64_t max_occ,
                           const InstDesc *insts, const uint32_t *start, const float4 *rec,
                           C2 *me, cudaStream_t st) {
    if constexpr (std::is_same<C2, float2>::value) {
        int per_sm = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2m_reg<PM>, P2M_WARPS * 32, 0);
        if (per_sm < 1) per_sm = 1;
        const int64_t grid = std::min<int64_t>((max_occ + P2M_WARPS - 1) / P2M_WARPS,
                                               int64_t(per_sm) * device_sm_count());
        k_p2m_reg<PM><<<unsigned(grid), P2M_WARPS * 32, 0, st>>>(occ, ctrl, insts, start, rec, me);
        return cudaGetLastError();
    } else {
        return cudaErrorNotSupported;
    }
}

template <typename R>
cudaError_t launch_p2m(const uint2 *occ, const uint32_t *ctrl, int64_t max_occ,
                       const InstDesc *insts, int pmax, const uint32_t *start, const double *xs,
                       const double *ys, const double *gs, const float4 *rec,
                       typename Cplx<R>::T *me, cudaStream_t st, uint64_t *launches) {
    if (max_occ <= 0) return cudaSuccess;
    const size_t smem = size_t(P2M_WARPS) * 32 * pmax * sizeof(typename Cplx<R>::T);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_p2m<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(smem));
        if (e != cudaSuccess) return e;
    }
    if (rec) {
        // mixed path: the register-accumulating kernel for the smallest
        // compiled bound on p
        cudaError_t e = cudaErrorNotSupported;
        if (pmax <= 8) e = launch_p2m_reg<8>(occ, ctrl, max_occ, insts, start, rec, me, st);
        else if (pmax <= 12) e = launch_p2m_reg<12>(occ, ctrl, max_occ, insts, start, rec, me, st);
        else if (pmax <= 17) e = launch_p2m_reg<17>(occ, ctrl, max_occ, insts, start, rec, me, st);
        else if (pmax <= 24) e = launch_p2m_reg<24>(occ, ctrl, max_occ, insts, start, rec, me, st);
        if (e != cudaErrorNotSupported) {
            PF_LAUNCHED(1);
            return e;
        }
    }
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2m<R>, P2M_WARPS * 32, smem);
    if (per_sm < 1) per_sm = 1;
    const int64_t grid = std::min<int64_t>((max_occ + P2M_WARPS - 1) / P2M_WARPS,
                                           int64_t(per_sm) * device_sm_count());
    k_p2m<R><<<unsigned(grid), P2M_WARPS * 32, smem, st>>>(occ, ctrl, insts, pmax, start, xs, ys,
                                                          gs, rec, me);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// M2L (SIMT): one warp per target box; lane m owns output coefficient m (and
// m + 32).  The source ME is staged in per-warp shared memory and read as a
// broadcast; operator rows come through L1.  Task = (instance, level l),
// units = 4^l target boxes, row-major.
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(M2L_WARPS * 32) k_m2l(const Task *__restrict__ tasks,
                                                        int ntasks,
                                                        const InstDesc *__restrict__ insts,
                                                        const uint32_t *__restrict__ start,
                                                        const float2 *__restrict__ me,
                                                        float2 *__restrict__ le,
                                                        const uint32_t *__restrict__ ucount,
                                                        int dense_pct) {
    using R = float;
    using C2 = float2;
    __shared__ C2 sa[M2L_WARPS][MAX_P];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t box0 = ((int64_t(blockIdx.x) - t.block0) * M2L_WARPS + wid) * BOX_RUN;
    if (box0 >= t.count) return;
    const InstDesc &d = insts[t.inst];
    const int p = d.p, l = t.level;
    const int nside = 1 << l;
    const uint32_t *st = start + d.soff;
    // the run's target boxes that hold particles and are not left to the
    // tensor cores (levels that also run there leave the dense units to them)
    bool mine = false;
    if (lane < BOX_RUN && box0 + lane < t.count) {
        const int64_t bx = box0 + lane;
        const int jx = int(bx & (nside - 1)), jy = int(bx >> l);
        mine = box_count(st, d.L, l, morton_key(uint32_t(jx), uint32_t(jy))) != 0;
        if (mine && d.tc_unit0[l] >= 0) {
            const int jc = (jx & 1) | ((jy & 1) << 1);
            int nbox;
            const int64_t u = d.tc_unit0[l] + unit_of(d, l, jc, jy >> 1, jx >> 1, &nbox);
            mine = !tc_unit_dense(ucount[u], nbox, dense_pct);
        }
    }
    uint32_t todo = __ballot_sync(0xffffffffu, mine);
    while (todo) {
        const int64_t box = box0 + (__ffs(todo) - 1);
        todo &= todo - 1;
        const int ix = int(box & (nside - 1)), iy = int(box >> l);
        const int c = (ix & 1) | ((iy & 1) << 1);
        const C2 *tab = static_cast<const C2 *>(d.t_m2l_box);
        const C2 *lev = me + d.eoff + lvl_off(l) * p;
        C2 acc0 = mk2<R>(R(0), R(0)), acc1 = mk2<R>(R(0), R(0));
        for (int e = 0; e < 27; ++e) {
            const IlEntry en = c_il.e[c][e];
            const int sx = ix + en.dx, sy = iy + en.dy;
            if (sx < 0 || sy < 0 || sx >= nside || sy >= nside) continue;
            if (!box_count(st, d.L, l, morton_key(uint32_t(sx), uint32_t(sy)))) continue;
            const C2 *src = lev + box_index(l, uint32_t(sx), uint32_t(sy)) * p;
            if (lane < p) sa[wid][lane] = src[lane];
            if (lane + 32 < p) sa[wid][lane + 32] = src[lane + 32];
            __syncwarp();
            const C2 *T = tab + size_t(en.op) * p * p;
            if (lane < p) {
                for (int k = 0; k < p; ++k) acc0 = cfma(T[k * p + lane], sa[wid][k], acc0);
            }
            if (lane + 32 < p) {
                for (int k = 0; k < p; ++k) acc1 = cfma(T[k * p + lane + 32], sa[wid][k], acc1);
            }
            __syncwarp();
        }
        C2 *dst = le + d.eoff + (lvl_off(l) + box_index(l, uint32_t(ix), uint32_t(iy))) * p;
        if (lane < p) dst[lane] = acc0;
        if (lane + 32 < p) dst[lane + 32] = acc1;
    }
}

cudaError_t launch_m2l(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                       const uint32_t *start, const float2 *me, float2 *le, const uint32_t *ucount,
                       int dense_pct, cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_m2l<<<unsigned(nblocks), M2L_WARPS * 32, 0, st>>>(tasks, ntasks, insts, start, me, le, ucount,
                                                       dense_pct);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Laplace kernel, the level-dependent constant of M2L: the rescaled
// operators carry log(-delta); the a~_0 log w_l part is added here, after all
// M2L kernels of the evaluation: b^_0(t) += log w_l * sum over the occupied
// interaction-list sources s of a~_0(s).  One thread per target box (task =
// instance, level; units = 4^l boxes, row-major), occupied targets only.
// ----------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256) k_m2l_logterm(const Task *__restrict__ tasks, int ntasks,
                                                     const InstDesc *__restrict__ insts,
                                                     const uint32_t *__restrict__ start,
                                                     const typename Cplx<R>::T *__restrict__ me,
                                                     typename Cplx<R>::T *__restrict__ le) {
    using C2 = typename Cplx<R>::T;
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t box = (int64_t(blockIdx.x) - t.block0) * 256 + threadIdx.x;
    if (box >= t.count) return;
    const InstDesc &d = insts[t.inst];
    const int p = d.p, l = t.level, nside = 1 << l;
    const uint32_t *st = start + d.soff;
    const int ix = int(box & (nside - 1)), iy = int(box >> l);
    if (!box_count(st, d.L, l, morton_key(uint32_t(ix), uint32_t(iy)))) return;
    const int c = (ix & 1) | ((iy & 1) << 1);
    const C2 *lev = me + d.eoff + lvl_off(l) * p;
    R sr = R(0), si = R(0);
    for (int e = 0; e < 27; ++e) {
        const IlEntry en = c_il.e[c][e];
        const int sx = ix + en.dx, sy = iy + en.dy;
        if (sx < 0 || sy < 0 || sx >= nside || sy >= nside) continue;
        if (!box_count(st, d.L, l, morton_key(uint32_t(sx), uint32_t(sy)))) continue;
        const C2 a0 = lev[box_index(l, uint32_t(sx), uint32_t(sy)) * p];
        sr += a0.x;
        si += a0.y;
    }
    const R logw = R(d.logw0 - double(l) * 0.69314718055994530942);
    C2 *dst = le + d.eoff + (lvl_off(l) + box_index(l, uint32_t(ix), uint32_t(iy))) * p;
    C2 o = *dst;
    o.x += logw * sr;
    o.y += logw * si;
    *dst = o;
}

template <typename R>
cudaError_t launch_m2l_logterm(const Task *tasks, int ntasks, int64_t nblocks,
                               const InstDesc *insts, const uint32_t *start,
                               const typename Cplx<R>::T *me, typename Cplx<R>::T *le,
                               cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_m2l_logterm<R><<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, me, le);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}
template cudaError_t launch_m2l_logterm<double>(const Task *, int, int64_t, const InstDesc *,
                                                const uint32_t *, const double2 *, double2 *,
                                                cudaStream_t, uint64_t *);
template cudaError_t launch_m2l_logterm<float>(const Task *, int, int64_t, const InstDesc *,
                                               const uint32_t *, const float2 *, float2 *,
                                               cudaStream_t, uint64_t *);

template cudaError_t launch_p2m<double>(const uint2 *, const uint32_t *, int64_t,
                                        const InstDesc *, int, const uint32_t *, const double *,
                                        const double *, const double *, const float4 *, double2 *,
                                        cudaStream_t, uint64_t *);
template cudaError_t launch_p2m<float>(const uint2 *, const uint32_t *, int64_t, const InstDesc *,
                                       int, const uint32_t *, const double *, const double *,
                                       const double *, const float4 *, float2 *, cudaStream_t,
                                       uint64_t *);

PF_DEFINE_CHECK_READER(expansions)

}  // namespace petfmm
