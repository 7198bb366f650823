// shifts.cu -- M2M and L2L of Sec. 2.2 (both precisions, both kernels).
//
// The centres of a box's four children are quarter turns of one another about
// its own centre, e_r = e_0 i^r (e_0 = (1 + i) / 2, in child widths), so the
// four translations share one real triangular matrix:
//   M2M  a'_l = e_0^l sum_k B[l][k] H_{(l-k) mod 4}[k],
//        H_j[k] = e_0^-k sum_r i^(r j) a_k^(r)
//   L2L  c'^(r)_n = e_0^-n sum_t i^(r t) G_{(t+n) mod 4},
//        G_s = sum_{m = s mod 4} B[n][m] (e_0^m c_m)
// with B[l][k] = 2^-l C(l, k) (M2M) and 2^-(m+1) C(m, n) (L2L) for the vortex
// kernel, the like for the Laplace kernel.  e_0^-k = (1 - i)^k, exact.  A
// parent costs p (p + 1) / 2 real-by-complex products and a few additions per
// coefficient, where four complex triangular products took eight times that.
// A block takes a run of parents (a row of the parent grid, so that each child
// class is one contiguous read), keeps the occupied ones, and lays the
// (parent, coefficient) pairs flat over its threads, the coefficients l and
// p - 1 - l together: every thread has about the same triangle to sum.
// Bound by latency at the upper levels (on the mixed path levels up to
// kShiftTop run in one launch, a block per instance) and by memory and
// shared-memory reads below.  Measured on one GB300, against a thread per (box,
// coefficient) with complex triangular products: mixed, 765,625 blobs, L = 10,
// p = 17: M2M 0.41 -> 0.17 ms, L2L 0.44 -> 0.21 ms; 512 uneven trees: 0.36 ->
// 0.13, 0.46 -> 0.18 ms; FP64, 1,048,576 blobs, L = 8: 0.58 -> 0.10, 0.44 ->
// 0.13 ms.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "kernels.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

namespace {

constexpr int SH_THREADS = 256;      // each phase of a block in one or two rounds
constexpr int SH_TOP_THREADS = 1024;  // a block of 64 parents: all of level kShiftTop = 3
constexpr int SH_TOP_BOXES = 1 << (2 * kShiftTop);

// row length of the matrices and of a box in shared memory
__host__ __device__ __forceinline__ int sh_row(int p) { return (p + 3) & ~3; }
// parents of a block
__host__ __device__ __forceinline__ int sh_boxes(int p) {
    const int b = 256 / p;
    return b < 1 ? 1 : b > 32 ? 32 : b;
}
// class of the child at e_0 i^r
__device__ __forceinline__ int turned_class(int r) { return r == 0 ? 3 : r == 1 ? 2 : r == 2 ? 0 : 1; }

template <typename R> __device__ __forceinline__ R fma_of(R a, R b, R c) { return fma(a, b, c); }

// Complex helpers with their roundings spelled out: the level kernels and the
// top kernel must give the same bits.
template <typename C2> __device__ __forceinline__ C2 sh_mul(C2 a, C2 b) {
    C2 r;
    r.x = fma_of(a.x, b.x, -(a.y * b.y));
    r.y = fma_of(a.x, b.y, a.y * b.x);
    return r;
}
template <typename C2> __device__ __forceinline__ C2 sh_add(C2 a, C2 b) {
    a.x += b.x;
    a.y += b.y;
    return a;
}
template <typename C2> __device__ __forceinline__ C2 sh_sub(C2 a, C2 b) {
    a.x -= b.x;
    a.y -= b.y;
    return a;
}
template <typename C2> __device__ __forceinline__ C2 sh_addi(C2 a, C2 b) {  // a + i b
    C2 r;
    r.x = a.x - b.y;
    r.y = a.y + b.x;
    return r;
}
template <typename C2> __device__ __forceinline__ C2 sh_subi(C2 a, C2 b) {  // a - i b
    C2 r;
    r.x = a.x + b.y;
    r.y = a.y - b.x;
    return r;
}

// Shared memory of `boxes` parents: the matrix, the powers, the parents' rows
// (M2M: the four H; L2L: one), the parents and their children.
template <typename R>
struct ShMem {
    using C2 = typename Cplx<R>::T;
    R *b;        // [p][row]
    C2 *ep, *em; // e_0^k, e_0^-k
    C2 *h;       // [4][js] or [1][js]
    int *box;    // [boxes]: row-major index of each kept parent
    int *child;  // [boxes][4]: index of its child at turn r within the level, or -1
    int *count;
    int js;
    __device__ ShMem(unsigned char *s, int p, int boxes, int planes) {
        const int row = sh_row(p);
        js = boxes * row + 1;  // one of padding: the four planes on different banks
        h = reinterpret_cast<C2 *>(s);
        ep = h + planes * js;
        em = ep + row;
        b = reinterpret_cast<R *>(em + row);
        box = reinterpret_cast<int *>(b + p * row);
        child = box + boxes;
        count = child + 4 * boxes;
    }
};

template <typename R>
size_t sh_bytes(int p, int boxes, int planes) {
    const size_t row = size_t(sh_row(p)), c = 2 * sizeof(R);
    return (planes * (boxes * row + 1) + 2 * row) * c + p * row * sizeof(R) +
           (5 * size_t(boxes) + 1) * sizeof(int);
}

// The instance's table (host_shift_table): [M2M B][L2L B][e_0^k][e_0^-k].
template <typename R>
__device__ __forceinline__ void sh_tables(const ShMem<R> &m, const void *tab, int p, bool l2l) {
    const int row = sh_row(p);
    const R *t = static_cast<const R *>(tab);
    for (int i = threadIdx.x; i < p * row; i += blockDim.x) m.b[i] = t[(l2l ? p * row : 0) + i];
    const R *e = t + 2 * p * row;
    R *ep = reinterpret_cast<R *>(m.ep);
    for (int i = threadIdx.x; i < 4 * row; i += blockDim.x) ep[i] = e[i];
}

// Keeps the occupied parents of first .. first + boxes - 1 (row-major, level
// l, depth L) and finds their occupied children: a parent's and its children's
// counts are differences of five leaf starts, loaded together.
template <typename R>
__device__ __forceinline__ int sh_parents(const ShMem<R> &m, const uint32_t *st, int L, int l,
                                          int64_t first, int boxes) {
    const int64_t np = int64_t(1) << (2 * l);
    if (threadIdx.x == 0) *m.count = 0;
    __syncthreads();
    const int64_t q = first + threadIdx.x;
    if (int(threadIdx.x) < boxes && q < np) {
        const uint64_t pm = morton_key(uint32_t(q & ((int64_t(1) << l) - 1)), uint32_t(q >> l));
        const int sh = 2 * (L - l - 1);
        uint32_t s[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) s[c] = st[(4 * pm + uint64_t(c)) << sh];
        if (s[4] > s[0]) {
            // any order: a box's sums do not depend on its place
            const int o = atomicAdd(m.count, 1);
            m.box[o] = int(q);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                // class c of parent (Px, Py) is at c 4^l + Py 2^l + Px
                const int c = turned_class(r);
                m.child[4 * o + r] = s[c + 1] > s[c] ? int(int64_t(c) * np + q) : -1;
            }
        }
    }
    __syncthreads();
    return *m.count;
}

template <typename R>
__device__ __forceinline__ void sh_m2m(const ShMem<R> &m, const InstDesc &d, int l, int n,
                                       typename Cplx<R>::T *me) {
    using C2 = typename Cplx<R>::T;
    const int p = d.p, row = sh_row(p), half = (p + 1) / 2;
    const C2 *kids = me + d.eoff + lvl_off(l + 1) * p;
    for (int e = threadIdx.x; e < n * p; e += blockDim.x) {
        const int b = e / p, k = e - b * p;
        C2 a[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            a[r].x = a[r].y = R(0);
            const int c = m.child[4 * b + r];
            if (c >= 0 && PF_IN(c, int64_t(4) << (2 * l))) a[r] = kids[int64_t(c) * p + k];
        }
        const C2 s02 = sh_add(a[0], a[2]), d02 = sh_sub(a[0], a[2]);
        const C2 s13 = sh_add(a[1], a[3]), d13 = sh_sub(a[1], a[3]);
        const C2 w = m.em[k];
        const int o = b * row + k;
        m.h[o] = sh_mul(sh_add(s02, s13), w);
        m.h[m.js + o] = sh_mul(sh_addi(d02, d13), w);
        m.h[2 * m.js + o] = sh_mul(sh_sub(s02, s13), w);
        m.h[3 * m.js + o] = sh_mul(sh_subi(d02, d13), w);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * half; e += blockDim.x) {
        const int b = e / half, l1 = e - b * half, l2 = p - 1 - l1;
        const int steps = l1 == l2 ? l1 + 1 : p + 1;
        C2 s, s1;
        s.x = s.y = s1.x = s1.y = R(0);
        const C2 *hb = m.h + b * row;
        // coefficient l1, then l2, as one run of steps
#pragma unroll 4
        for (int t = 0; t < steps; ++t) {
            const bool one = t <= l1;
            const int k = one ? t : t - l1 - 1, lc = one ? l1 : l2;
            const C2 v = hb[((lc - k) & 3) * m.js + k];
            const R w = m.b[lc * row + k];
            s.x = fma_of(w, v.x, s.x);
            s.y = fma_of(w, v.y, s.y);
            if (t == l1) {
                s1 = s;
                s.x = s.y = R(0);
            }
        }
        const int64_t q = m.box[b];
        const uint32_t ix = uint32_t(q & ((int64_t(1) << l) - 1)), iy = uint32_t(q >> l);
        C2 *dst = me + d.eoff + (lvl_off(l) + box_index(l, ix, iy)) * p;
        dst[l1] = sh_mul(s1, m.ep[l1]);
        if (l1 != l2) dst[l2] = sh_mul(s, m.ep[l2]);
    }
}

template <typename R>
__device__ __forceinline__ void sh_l2l(const ShMem<R> &m, const InstDesc &d, int l, int n,
                                       typename Cplx<R>::T *le) {
    // l: the parents' level
    using C2 = typename Cplx<R>::T;
    const int p = d.p, row = sh_row(p), half = (p + 1) / 2;
    for (int e = threadIdx.x; e < n * row; e += blockDim.x) {
        const int b = e / row, k = e - b * row;
        C2 v;
        v.x = v.y = R(0);
        if (k < p) {
            const int64_t q = m.box[b];
            const uint32_t ix = uint32_t(q & ((int64_t(1) << l) - 1)), iy = uint32_t(q >> l);
            v = sh_mul(le[d.eoff + (lvl_off(l) + box_index(l, ix, iy)) * p + k], m.ep[k]);
        }
        m.h[e] = v;
    }
    __syncthreads();
    C2 *kids = le + d.eoff + lvl_off(l + 1) * p;
    for (int e = threadIdx.x; e < n * half; e += blockDim.x) {
        const int b = e / half, n1 = e - b * half, n2 = p - 1 - n1;
        const C2 *hb = m.h + b * row;
        // the children's own parts, requested before the sums
        C2 own[2][4];
#pragma unroll
        for (int which = 0; which < 2; ++which)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int kid = m.child[4 * b + r];
                own[which][r].x = own[which][r].y = R(0);
                if (kid >= 0 && PF_IN(kid, int64_t(4) << (2 * l))) own[which][r] = kids[int64_t(kid) * p + (which ? n2 : n1)];
            }
#pragma unroll
        for (int which = 0; which < 2; ++which) {
            const int c = which ? n2 : n1;
            if (which && n1 == n2) break;
            C2 g[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) g[s].x = g[s].y = R(0);
            // (the matrix is zero below the diagonal and in its padding)
#pragma unroll 2
            for (int k0 = c & ~3; k0 < row; k0 += 4)
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const C2 v = hb[k0 + s];
                    const R w = m.b[c * row + k0 + s];
                    g[s].x = fma_of(w, v.x, g[s].x);
                    g[s].y = fma_of(w, v.y, g[s].y);
                }
            // F_t = G_{(t + c) mod 4}
            if (c & 1) {
                const C2 x = g[0];
                g[0] = g[1];
                g[1] = g[2];
                g[2] = g[3];
                g[3] = x;
            }
            if (c & 2) {
                C2 x = g[0];
                g[0] = g[2];
                g[2] = x;
                x = g[1];
                g[1] = g[3];
                g[3] = x;
            }
            const C2 s02 = sh_add(g[0], g[2]), d02 = sh_sub(g[0], g[2]);
            const C2 s13 = sh_add(g[1], g[3]), d13 = sh_sub(g[1], g[3]);
            const C2 f[4] = {sh_add(s02, s13), sh_addi(d02, d13), sh_sub(s02, s13),
                             sh_subi(d02, d13)};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int kid = m.child[4 * b + r];
                if (kid >= 0 && PF_IN(kid, int64_t(4) << (2 * l)))
                    kids[int64_t(kid) * p + c] = sh_add(own[which][r], sh_mul(f[r], m.em[c]));
            }
        }
    }
}

template <typename R, bool L2L>
__global__ void __launch_bounds__(SH_THREADS) k_shift(const Task *__restrict__ tasks, int ntasks,
                                                      const InstDesc *__restrict__ insts,
                                                      const uint32_t *__restrict__ start,
                                                      typename Cplx<R>::T *ex) {
    extern __shared__ __align__(16) unsigned char sh_smem[];
    const Task t = tasks[find_task(tasks, ntasks, blockIdx.x)];
    const InstDesc &d = insts[t.inst];
    const int boxes = sh_boxes(d.p);
    const ShMem<R> m(sh_smem, d.p, boxes, L2L ? 1 : 4);
    const int64_t first = (int64_t(blockIdx.x) - t.block0) * boxes;
    sh_tables(m, d.t_shift, d.p, L2L);  // (its loads overlap the parents')
    const int n = sh_parents(m, start + d.soff, d.L, t.level, first, boxes);
    if (n == 0) return;
    if (L2L) sh_l2l(m, d, t.level, n, ex);
    else sh_m2m(m, d, t.level, n, ex);
}

// Levels 2 .. kShiftTop of one instance per block, one after another.
template <typename R, bool L2L>
__global__ void __launch_bounds__(SH_TOP_THREADS) k_shift_top(const InstDesc *__restrict__ insts,
                                                              const uint32_t *__restrict__ start,
                                                              typename Cplx<R>::T *ex) {
    extern __shared__ __align__(16) unsigned char sh_smem[];
    const InstDesc &d = insts[blockIdx.x];
    if (d.L < 3 || d.n == 0) return;
    const int boxes = SH_TOP_BOXES;
    const ShMem<R> m(sh_smem, d.p, boxes, L2L ? 1 : 4);
    sh_tables(m, d.t_shift, d.p, L2L);
    const int last = min(d.L - 1, kShiftTop);  // parents' levels 2 .. last
    for (int i = 2; i <= last; ++i) {
        const int l = L2L ? i : last + 2 - i;
        __syncthreads();  // the previous level's results
        const int n = sh_parents(m, start + d.soff, d.L, l, 0, boxes);
        if (L2L) sh_l2l(m, d, l, n, ex);
        else sh_m2m(m, d, l, n, ex);
    }
}

}  // namespace

// The real matrices from the complex tables of turn 0 (class 3): T =
// B e_0^(difference).
void host_shift_table(int p, int kernel, std::vector<double> &out) {
    const int row = sh_row(p);
    std::vector<double> m2m, l2l;
    host_op_table(p, kernel, 0, m2m);  // [c][l][k]
    host_op_table(p, kernel, 1, l2l);  // [c][n][m]
    out.assign(size_t(2) * p * row + 4 * row, 0.0);
    double *ep = out.data() + size_t(2) * p * row, *em = ep + 2 * row;
    double re = 1.0, im = 0.0, rn = 1.0, in = 0.0;
    for (int k = 0; k < p; ++k) {
        ep[2 * k] = re;
        ep[2 * k + 1] = im;
        em[2 * k] = rn;
        em[2 * k + 1] = in;
        const double t = 0.5 * (re - im), u = rn + in;
        im = 0.5 * (re + im);
        re = t;
        in = in - rn;
        rn = u;
    }
    for (int l = 0; l < p; ++l)
        for (int k = 0; k <= l; ++k) {
            const double *t = &m2m[((size_t(3) * p + l) * p + k) * 2];
            const double *e = em + 2 * (l - k);
            out[size_t(l) * row + k] = t[0] * e[0] - t[1] * e[1];
            const double *u = &l2l[((size_t(3) * p + k) * p + l) * 2];
            out[size_t(p) * row + size_t(k) * row + l] = u[0] * e[0] - u[1] * e[1];
        }
}

int64_t shift_units(int p, int level) {
    const int64_t np = int64_t(1) << (2 * level);
    return (np + sh_boxes(p) - 1) / sh_boxes(p);
}

size_t shift_smem(int p, bool fp64, bool top) {
    const int boxes = top ? SH_TOP_BOXES : sh_boxes(p);
    return fp64 ? sh_bytes<double>(p, boxes, 4) : sh_bytes<float>(p, boxes, 4);
}

template <typename R>
cudaError_t launch_shift(bool l2l, const Task *tasks, int ntasks, int64_t nblocks, size_t smem,
                         const InstDesc *insts, const uint32_t *start, typename Cplx<R>::T *ex,
                         cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    auto *k = l2l ? k_shift<R, true> : k_shift<R, false>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    k<<<unsigned(nblocks), SH_THREADS, smem, st>>>(tasks, ntasks, insts, start, ex);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

cudaError_t launch_shift_top(bool l2l, int ninst, size_t smem, const InstDesc *insts,
                             const uint32_t *start, float2 *ex, cudaStream_t st,
                             uint64_t *launches) {
    if (ninst <= 0) return cudaSuccess;
    auto *k = l2l ? k_shift_top<float, true> : k_shift_top<float, false>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    k<<<unsigned(ninst), SH_TOP_THREADS, smem, st>>>(insts, start, ex);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

template cudaError_t launch_shift<float>(bool, const Task *, int, int64_t, size_t, const InstDesc *,
                                         const uint32_t *, float2 *, cudaStream_t, uint64_t *);
template cudaError_t launch_shift<double>(bool, const Task *, int, int64_t, size_t, const InstDesc *,
                                          const uint32_t *, double2 *, cudaStream_t, uint64_t *);

PF_DEFINE_CHECK_READER(shifts)

}  // namespace petfmm
