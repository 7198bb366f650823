// smooth.cu -- the mixed path's near field where the blob core is wide
// against a leaf (Eq. 8 with kappa = w^2 / 2 sigma^2 below kSmKappaMax).
//
// In leaf units the near field of Eq. 9 is u = c sum gamma (-d_eta, d_xi)
// g(kappa |d|^2), g(q) = (1 - e^-q) / q, the turned gradient of the radial
// function Phi(d) = Ein(kappa |d|^2) / (2 kappa), which is smooth when the
// core is no narrower than a leaf: between two given leaves,
//     Phi(D + tau - s) = sum_{alpha, beta} C^D[beta][alpha] m_alpha(tau) P_beta(s)
// to FP32 accuracy with few terms (tau, s: target and source offsets from
// their leaf centres, D the offset of the centres, P products of Legendre
// polynomials and m products of powers, total degree <= n each).  So the
// blobs of two leaves need not meet one by one (12 operations a pair): each
// leaf's blobs are summed into (n + 1)(n + 2) / 2 moments, a leaf adds its
// 9 neighbours' moments through the 9 fixed matrices C^D, and each blob
// evaluates one polynomial gradient.  The far field's expansions cannot do
// this: they hold the singular kernel 1 / |x|^2.
//
// Leaf pairs with few blobs on both sides (na nb below sm_direct_max) are
// cheaper summed directly, by the final pass with one thread per target.
//
// Measured on one GB300, the whole evaluation against the pairwise near field
// (p2p.cu): 16.8M clustered blobs, kappa = 0.12: 18.3 -> 2.4 ms; 4.2M with the
// copies from and to the host: 5.2 -> 1.15 ms; 765k blobs, one per leaf (direct
// pairs only, without their work lists, with the other steps): 2.89 -> 1.57 ms.
//
// kappa <= 1.95 (degree 14) is where the line lies: the degree needed grows
// with the core's steepness (a translation costs the square of (n + 1)(n + 2)
// / 2), and at the next density in use, kappa near 3.6 at 16 blobs per leaf, a
// leaf pair has 256 blob pairs against 14,400 multiply-adds at degree 14.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "kernels.cuh"
#include "near_direct.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

namespace {

// terms of total degree <= n, ordered by the power b of y, then a of x
__host__ __device__ constexpr int sm_terms(int n) { return (n + 1) * (n + 2) / 2; }
__host__ __device__ constexpr int sm_stride(int n) { return (sm_terms(n) + 3) / 4 * 4; }
__host__ __device__ constexpr int sm_idx(int n, int a, int b) {
    return b * (n + 1) - b * (b - 1) / 2 + a;
}

// A leaf pair with fewer blob pairs than this is summed directly: about the
// cost of one translation (terms^2 multiply-adds of a tiled product) plus
// its share of moments and evaluation.
__host__ __device__ constexpr uint32_t sm_direct_max(int n) {
    return uint32_t(sm_terms(n) * sm_terms(n) / 8);
}

constexpr int SM_TGT = 64;        // target leaves per block of the translation
constexpr uint32_t LM_EXP = 16;   // lmask: bits 0..8 direct neighbours, 16..24 by expansion

}  // namespace

// ----------------------------------------------------------------------------
// Host: degree and operators
// ----------------------------------------------------------------------------
// Largest error of the gradient over the near domain, against its largest
// value there, of the projection below: at most 1.2e-7 up to each bound, and
// another 3e-7 by the FP32 rounding of the operators' entries
// (tests/test_smooth_operator.py).  A caller who asks for less gets pair sums.
constexpr double kSmTol = 4.2e-7;

int sm_degree(double kappa, double near_tol) {
    if (!(near_tol >= kSmTol)) return 0;
    static const struct { double kappa; int n; } kBound[] = {
        {0.17, 8}, {0.50, 10}, {1.04, 12}, {1.95, 14}};
    for (const auto &b : kBound)
        if (kappa <= b.kappa) return b.n;
    return 0;
}

size_t sm_row_floats(int n) { return size_t(sm_stride(n)); }

// Leaves of an instance that can need expansions: one of the two leaves of a
// pair of at least sm_direct_max blob pairs holds at least its square root,
// and each such leaf has 9 neighbours.
int64_t sm_max_rows(int n, int64_t blobs, int64_t leaves) {
    int64_t s = 1;
    while ((s + 1) * (s + 1) <= int64_t(sm_direct_max(n))) ++s;
    return std::min(std::min(blobs, leaves), 9 * (blobs / s));
}

// Chebyshev terms per axis of Phi in d (the interpolation error is below
// 1e-12 for kappa < 2).
constexpr int kSmCheb = 26;

// What the operators of a degree have in common, FP64, built once per process
// (one copy per context on the device): U[a][b][i], i < kSmCheb, with which
// sum_ij U[a1][b1][i] f[i][j] U[a2][b2][j] is the coefficient of P_a1(2 tau_x)
// P_b1(2 s_x) P_a2(2 tau_y) P_b2(2 s_y) in the function of tau - s that has the
// values f at the Chebyshev nodes; the powers pw[a][e] of x in P_a(x); the nodes
// cos(pi (i + 1/2) / kSmCheb); 1 / k for the series of Ein.
constexpr int kSmSeries = 160;
struct SmFixed {
    const double *u, *pw, *node, *inv;
    __host__ __device__ SmFixed(const double *t, int n) {
        const int n1 = n + 1;
        u = t;
        pw = u + n1 * n1 * kSmCheb;
        node = pw + n1 * n1;
        inv = node + kSmCheb;
    }
};
static size_t sm_fixed_words(int n) {
    return size_t(n + 1) * (n + 1) * (kSmCheb + 1) + kSmCheb + kSmSeries;
}

const std::vector<double> &host_sm_fixed(int n) {
    static std::mutex mu;
    static std::map<int, std::vector<double>> tables;
    std::lock_guard<std::mutex> lk(mu);
    std::vector<double> &out = tables[n];
    if (!out.empty()) return out;
    // V[a][b][k]: T_k(tau - s), tau, s in [-1/2, 1/2], projected onto
    // P_a(2 tau) P_b(2 s), a, b <= n
    std::vector<double> V;
    const int n1 = n + 1, q = n + 12;  // Gauss nodes: exact for T_k P_a products
    // Gauss-Legendre nodes by Newton's method on P_q
    std::vector<double> xg(q), wg(q);
    for (int i = 0; i < q; ++i) {
        double x = std::cos(M_PI * (i + 0.75) / (q + 0.5)), dp = 1.0;
        for (int it = 0; it < 60; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= q; ++k) {
                const double p2 = ((2 * k - 1) * x * p1 - (k - 1) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = q * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-15) break;
        }
        xg[i] = x;
        wg[i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
    // proj[a][i]: coefficient a of the Legendre projection from node values
    std::vector<double> proj(size_t(n1) * q), t(size_t(q) * q), tmp(size_t(n1) * q);
    for (int i = 0; i < q; ++i) {
        double p0 = 1.0, p1 = xg[i];
        for (int a = 0; a <= n; ++a) {
            proj[size_t(a) * q + i] = p0 * wg[i] * (2 * a + 1) * 0.5;
            const double p2 = ((2 * a + 3) * xg[i] * p1 - (a + 1) * p0) / (a + 2);
            p0 = p1;
            p1 = p2;
        }
    }
    V.assign(size_t(n1) * n1 * kSmCheb, 0.0);
    std::vector<double> t0(size_t(q) * q), t1(size_t(q) * q);  // T_{k-2}, T_{k-1}
    for (int k = 0; k < kSmCheb; ++k) {
        for (int i = 0; i < q; ++i)
            for (int j = 0; j < q; ++j) {
                const size_t e = size_t(i) * q + j;
                const double x = 0.5 * (xg[i] - xg[j]);
                t[e] = k == 0 ? 1.0 : k == 1 ? x : 2.0 * x * t1[e] - t0[e];
                t0[e] = t1[e];
                t1[e] = t[e];
            }
        for (int a = 0; a < n1; ++a)
            for (int j = 0; j < q; ++j) {
                double s = 0.0;
                for (int i = 0; i < q; ++i) s += proj[size_t(a) * q + i] * t[size_t(i) * q + j];
                tmp[size_t(a) * q + j] = s;
            }
        for (int a = 0; a < n1; ++a)
            for (int b = 0; b < n1; ++b) {
                double s = 0.0;
                for (int j = 0; j < q; ++j) s += proj[size_t(b) * q + j] * tmp[size_t(a) * q + j];
                V[size_t(a * n1 + b) * kSmCheb + k] = s;
            }
    }
    out.assign(sm_fixed_words(n), 0.0);
    double *U = out.data(), *pw = U + size_t(n1) * n1 * kSmCheb, *node = pw + n1 * n1,
           *inv = node + kSmCheb;
    for (int i = 0; i < kSmCheb; ++i) node[i] = std::cos(M_PI * (i + 0.5) / kSmCheb);
    for (int k = 1; k < kSmSeries; ++k) inv[k] = 1.0 / k;
    // Chebyshev coefficients from the values at the nodes
    std::vector<double> cs(size_t(kSmCheb) * kSmCheb);
    for (int k = 0; k < kSmCheb; ++k)
        for (int i = 0; i < kSmCheb; ++i)
            cs[size_t(k) * kSmCheb + i] =
                std::cos(M_PI * k * (i + 0.5) / kSmCheb) * (k ? 2.0 : 1.0) / kSmCheb;
    for (int e = 0; e < n1 * n1; ++e)
        for (int i = 0; i < kSmCheb; ++i) {
            double v = 0.0;
            // (T_k has the parity of k)
            for (int k = (e / n1 + e % n1) & 1; k < kSmCheb; k += 2)
                v += V[size_t(e) * kSmCheb + k] * cs[size_t(k) * kSmCheb + i];
            U[size_t(e) * kSmCheb + i] = v;
        }
    pw[0] = 1.0;
    if (n >= 1) pw[n1 + 1] = 1.0;
    for (int a = 2; a <= n; ++a)
        for (int k = 0; k <= a; ++k)
            pw[a * n1 + k] = ((k ? (2 * a - 1) * pw[(a - 1) * n1 + k - 1] : 0.0) -
                              (a - 1) * pw[(a - 2) * n1 + k]) / a;
    return out;
}

// The operators C^D of the 9 neighbour offsets, source = target + (ox, oy), block
// (oy + 1) 3 + ox + 1, as [beta][alpha] with rows of sm_stride(n) floats; beta:
// Legendre products of twice the source offset, alpha: powers of twice the
// target offset.  Phi is interpolated in d by Chebyshev polynomials, T_k(tau -
// s) projected onto Legendre products (both in U), the total degrees cut at n,
// and the target side turned into powers; FP64 throughout.  Three of the nine
// are computed, D = (0, 0), (1, 0), (1, 1); the others mirror or swap them.  The
// steps below make them on the device (k_sm_values, k_sm_half, k_sm_finish: an
// evaluation meets a new kappa without the host's 0.6 to 1.6 ms) and on the host.

// Phi = Ein(kappa s) / (2 kappa), s = |d|^2
__host__ __device__ inline double sm_phi(const SmFixed &t, double kappa, double s) {
    const double z = kappa * s;
    double term = 1.0, sum = 0.0;  // sum_k (-z)^(k-1) / (k k!)
    for (int k = 1; k < kSmSeries - 1; ++k) {
        sum += term * t.inv[k];
        term *= -z * t.inv[k + 1];
        if (fabs(term) < 1e-18 && k > z) break;
    }
    return 0.5 * s * sum;
}
// value e = (i, j) of offset D (0: (0, 0), 1: (1, 0), 2: (1, 1))
__host__ __device__ inline double sm_value(const SmFixed &t, double kappa, int D, int e) {
    const double dx = (D > 0) + t.node[e / kSmCheb], dy = (D > 1) + t.node[e % kSmCheb];
    return sm_phi(t, kappa, dx * dx + dy * dy);
}
// w[a2][b2][i] = sum_j f[i][j] U[a2][b2][j], e = (a2, b2, i)
__host__ __device__ inline double sm_half(const SmFixed &t, const double *f, int e) {
    const double *u = t.u + e / kSmCheb * kSmCheb, *g = f + e % kSmCheb * kSmCheb;
    double v = 0.0;
    for (int j = 0; j < kSmCheb; ++j) v += g[j] * u[j];
    return v;
}
// A term's degrees (a of x, b of y).
__host__ __device__ inline void sm_degrees(int n, int t, int *a, int *b) {
    int y = 0;
    while (sm_idx(n, 0, y + 1) <= t && y < n) ++y;
    *b = y;
    *a = t - sm_idx(n, 0, y);
}
// Row (b1, b2) of C^D, term (a1, a2): Legendre coefficient ...
__host__ __device__ inline double sm_legendre(const SmFixed &t, int n, const double *w, int b1,
                                              int b2, int a1, int a2) {
    const double *u = t.u + (a1 * (n + 1) + b1) * kSmCheb;
    const double *v = w + (a2 * (n + 1) + b2) * kSmCheb;
    double c = 0.0;
    for (int i = 0; i < kSmCheb; ++i) c += u[i] * v[i];
    return c;
}
// ... then powers of x (cl: the row's terms) ...
__host__ __device__ inline double sm_power_x(const SmFixed &t, int n, const double *cl, int e1, int a2) {
    double v = 0.0;
    for (int a1 = e1; a1 + a2 <= n; a1 += 2) v += cl[sm_idx(n, a1, a2)] * t.pw[a1 * (n + 1) + e1];
    return v;
}
// ... and of y.
__host__ __device__ inline double sm_power_y(const SmFixed &t, int n, const double *cx, int e1, int e2) {
    double v = 0.0;
    for (int a2 = e2; e1 + a2 <= n; a2 += 2) v += cx[sm_idx(n, e1, a2)] * t.pw[a2 * (n + 1) + e2];
    return v;
}
// Entry (b1, b2), (e1, e2) of C^D into the offsets that mirror or swap D; pad >=
// 0: column pad of the row instead, which has no term, zero.
__host__ __device__ inline void sm_store(int n, int D, int b1, int b2, int e1, int e2, int pad,
                                         double v, float *out) {
    const int M = sm_terms(n), S = sm_stride(n);
    for (int o = 0; o < 9; ++o) {
        const int ox = o % 3 - 1, oy = o / 3 - 1, ax = ox < 0 ? -ox : ox, ay = oy < 0 ? -oy : oy;
        if (ax + ay != D) continue;
        const bool swap = ay > ax;
        const int p1 = swap ? b2 : b1, p2 = swap ? b1 : b2, q1 = swap ? e2 : e1, q2 = swap ? e1 : e2;
        const int par = (ox > 0 ? p1 + q1 : 0) + (oy > 0 ? p2 + q2 : 0);
        float *row = out + (size_t(o) * M + sm_idx(n, p1, p2)) * S;
        if (pad >= 0) row[pad] = 0.0f;
        else row[sm_idx(n, q1, q2)] = float(par & 1 ? -v : v);
    }
}

void host_sm_operators(double kappa, int n, std::vector<float> &out) {
    const int n1 = n + 1, M = sm_terms(n), S = sm_stride(n);
    const SmFixed t(host_sm_fixed(n).data(), n);
    out.assign(size_t(9) * M * S, 0.0f);
    std::vector<double> f(size_t(kSmCheb) * kSmCheb), w(size_t(n1) * n1 * kSmCheb);
    std::vector<double> cl(static_cast<size_t>(M)), cx(static_cast<size_t>(M));
    for (int D = 0; D < 3; ++D) {
        for (size_t e = 0; e < f.size(); ++e) f[e] = sm_value(t, kappa, D, int(e));
        for (size_t e = 0; e < w.size(); ++e) w[e] = sm_half(t, f.data(), int(e));
        for (int beta = 0; beta < M; ++beta) {
            int b1, b2, x, y;
            sm_degrees(n, beta, &b1, &b2);
            for (int k = 0; k < M; ++k) {
                sm_degrees(n, k, &x, &y);
                cl[size_t(k)] = sm_legendre(t, n, w.data(), b1, b2, x, y);
            }
            for (int k = 0; k < M; ++k) {
                sm_degrees(n, k, &x, &y);
                cx[size_t(k)] = sm_power_x(t, n, cl.data(), x, y);
            }
            for (int k = 0; k < M; ++k) {
                sm_degrees(n, k, &x, &y);
                sm_store(n, D, b1, b2, x, y, -1, sm_power_y(t, n, cx.data(), x, y), out.data());
            }
        }
    }
}

// ----------------------------------------------------------------------------
// The same on the device: grid (entries, D, operator)
// ----------------------------------------------------------------------------
namespace {

constexpr int SM_OPS = 64;  // operators per launch
struct SmOps {
    const double *fixed[SM_OPS];
    float *out[SM_OPS];
    double kappa[SM_OPS];
    int n[SM_OPS];
    double *work;   // per operator and D: values, then w
    size_t stride;  // of one (operator, D)
};

__device__ __forceinline__ double *sm_work(const SmOps &o, int op, int D) {
    return o.work + size_t(op * 3 + D) * o.stride;
}

__global__ void __launch_bounds__(128) k_sm_values(const __grid_constant__ SmOps o) {
    const int op = int(blockIdx.z), D = int(blockIdx.y), e = int(blockIdx.x * 128 + threadIdx.x);
    if (e >= kSmCheb * kSmCheb) return;
    sm_work(o, op, D)[e] = sm_value(SmFixed(o.fixed[op], o.n[op]), o.kappa[op], D, e);
}

__global__ void __launch_bounds__(128) k_sm_half(const __grid_constant__ SmOps o) {
    const int op = int(blockIdx.z), D = int(blockIdx.y), e = int(blockIdx.x * 128 + threadIdx.x);
    const int n = o.n[op];
    if (e >= (n + 1) * (n + 1) * kSmCheb) return;
    double *f = sm_work(o, op, D);
    f[kSmCheb * kSmCheb + e] = sm_half(SmFixed(o.fixed[op], n), f, e);
}

// A block per row of C^D, a thread per term.
constexpr int SM_TERMS_MAX = sm_terms(14);
static_assert(SM_TERMS_MAX <= 128 && sm_stride(14) <= 128, "a thread per term");
__global__ void __launch_bounds__(128) k_sm_finish(const __grid_constant__ SmOps o) {
    __shared__ double cl[SM_TERMS_MAX], cx[SM_TERMS_MAX];
    const int op = int(blockIdx.z), D = int(blockIdx.y), beta = int(blockIdx.x);
    const int n = o.n[op], M = sm_terms(n), k = int(threadIdx.x);
    if (beta >= M) return;
    const SmFixed t(o.fixed[op], n);
    const double *w = sm_work(o, op, D) + kSmCheb * kSmCheb;
    int b1, b2, x = 0, y = 0;
    sm_degrees(n, beta, &b1, &b2);
    if (k < M) {
        sm_degrees(n, k, &x, &y);
        cl[k] = sm_legendre(t, n, w, b1, b2, x, y);
    }
    __syncthreads();
    if (k < M) cx[k] = sm_power_x(t, n, cl, x, y);
    __syncthreads();
    if (k < M) sm_store(n, D, b1, b2, x, y, -1, sm_power_y(t, n, cx, x, y), o.out[op]);
    else if (k < sm_stride(n)) sm_store(n, D, b1, b2, 0, 0, k, 0.0, o.out[op]);
}

}  // namespace

size_t sm_operator_floats(int n) { return size_t(9) * sm_terms(n) * sm_stride(n); }

static size_t sm_work_stride(int n) {
    return size_t(kSmCheb) * kSmCheb + size_t(n + 1) * (n + 1) * kSmCheb;
}
size_t sm_work_bytes(int n, size_t ops) {
    return std::min(ops, size_t(SM_OPS)) * 3 * sm_work_stride(n) * sizeof(double);
}

cudaError_t launch_sm_operators(const std::vector<SmOperator> &ops, int nmax, double *work,
                                cudaStream_t st, uint64_t *launches) {
    for (size_t i0 = 0; i0 < ops.size(); i0 += SM_OPS) {
        SmOps o{};
        const size_t m = std::min(ops.size() - i0, size_t(SM_OPS));
        for (size_t i = 0; i < m; ++i) {
            o.fixed[i] = ops[i0 + i].fixed;
            o.out[i] = ops[i0 + i].out;
            o.kappa[i] = ops[i0 + i].kappa;
            o.n[i] = ops[i0 + i].n;
        }
        o.work = work;
        o.stride = sm_work_stride(nmax);
        const unsigned z = unsigned(m);
        k_sm_values<<<dim3((kSmCheb * kSmCheb + 127) / 128, 3, z), 128, 0, st>>>(o);
        k_sm_half<<<dim3(unsigned((nmax + 1) * (nmax + 1) * kSmCheb + 127) / 128, 3, z), 128, 0, st>>>(o);
        k_sm_finish<<<dim3(unsigned(sm_terms(nmax)), 3, z), 128, 0, st>>>(o);
        PF_LAUNCHED(3);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ----------------------------------------------------------------------------
// Lists: a thread per leaf
// ----------------------------------------------------------------------------
// The occupied leaves (as k_occ_list of expansions.cu, which this replaces in
// plans with smooth instances) and, for those of a smooth instance, which of
// the nine neighbours are summed directly and which by expansions, the leaves
// that need a row of the expansion buffers, and the ordered near pairs for the
// statistics.  One atomic per block and list: a block's leaves, neighbours on
// the Morton curve, get consecutive rows.  With the classification in
// k_sm_moments (a warp per occupied leaf) 765k blobs, one per leaf, spent
// 234 us there, now 25 us here with the occupied list.
__global__ void __launch_bounds__(256) k_sm_lists(const Task *__restrict__ tasks, int ntasks,
                                                  const InstDesc *__restrict__ insts,
                                                  const uint32_t *__restrict__ start,
                                                  uint2 *__restrict__ occ, uint32_t *ctrl,
                                                  const SmBufs sb) {
    __shared__ uint32_t wcnt[2][8], base[2];
    __shared__ unsigned long long wpairs[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    const InstDesc &d = insts[t.inst];
    const uint32_t *st = start + d.soff;
    const uint32_t n = m < t.count ? st[m + 1] - st[m] : 0u;
    unsigned long long pairs = 0;
    uint32_t em = 0;
    if (n && d.smdeg) {
        const int nside = 1 << d.L;
        const uint32_t least = sm_direct_max(d.smdeg);
        const int ix = int(compact_bits(uint32_t(m))), iy = int(compact_bits(uint32_t(m) >> 1));
        uint32_t dm = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int x = ix + k % 3 - 1, y = iy + k / 3 - 1;
            if (x < 0 || y < 0 || x >= nside || y >= nside) continue;
            const uint32_t nm = morton_key(uint32_t(x), uint32_t(y));
            const uint32_t cnt = st[nm + 1] - st[nm];
            const bool byexp = uint64_t(n) * cnt >= least;
            em |= uint32_t(byexp) << k;
            dm |= uint32_t(cnt > 0 && !byexp) << k;
            pairs += (unsigned long long)n * (k == 4 ? cnt - 1 : cnt);
        }
        sb.lmask[d.loff + m] = dm | (em << LM_EXP);
    }
    const uint32_t bo = __ballot_sync(0xffffffffu, n > 0), be = __ballot_sync(0xffffffffu, em != 0);
#pragma unroll
    for (int o = 16; o; o >>= 1) pairs += __shfl_down_sync(0xffffffffu, pairs, o);
    if (lane == 0) {
        wcnt[0][wid] = __popc(bo);
        wcnt[1][wid] = __popc(be);
        wpairs[wid] = pairs;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        uint32_t s = 0;
        for (int w = 0; w < 8; ++w) {
            const uint32_t v = wcnt[threadIdx.x][w];
            wcnt[threadIdx.x][w] = s;
            s += v;
        }
        base[threadIdx.x] = s ? atomicAdd(ctrl + (threadIdx.x ? CTRL_NSMOOTH : CTRL_NOCC), s) : 0u;
    } else if (threadIdx.x == 32) {
        unsigned long long s = 0;
        for (int w = 0; w < 8; ++w) s += wpairs[w];
        if (s) atomicAdd(reinterpret_cast<unsigned long long *>(ctrl + CTRL_PAIRS_LO), s);
    }
    __syncthreads();
    const uint32_t below = (1u << lane) - 1u;
    const uint2 e = make_uint2(uint32_t(t.inst), uint32_t(m));
    if (n) occ[base[0] + wcnt[0][wid] + __popc(bo & below)] = e;
    if (em) {
        const uint32_t rank = base[1] + wcnt[1][wid] + __popc(be & below);
        sb.lrank[d.loff + m] = rank;
        if (PF_IN(rank, sb.rows)) sb.list[rank] = e;
    }
}

cudaError_t launch_sm_lists(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, uint2 *occ, uint32_t *ctrl, const SmBufs &sb,
                            cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_sm_lists<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, occ, ctrl, sb);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Moments: a warp per leaf of the list
// ----------------------------------------------------------------------------
// Each lane sums all the moments of its blobs in registers (one multiply-add per
// blob and term), then 32 values at a time are reduced and scattered over the
// lanes by halving exchanges (31 shuffles per 32 values instead of 160).  Waits on
// its records (2M clustered blobs: FMA pipe 30 %, DRAM 15 %, a third of the warps
// resident).
template <int N>
__global__ void __launch_bounds__(128) k_sm_moments(const uint32_t *ctrl,
                                                    const InstDesc *__restrict__ insts,
                                                    const uint32_t *__restrict__ start,
                                                    const float4 *__restrict__ rec,
                                                    const SmBufs sb) {
    constexpr int M = sm_terms(N), G = (M + 31) / 32;
    const int lane = threadIdx.x & 31;
    const uint32_t nlist = ctrl[CTRL_NSMOOTH];
    const uint32_t nwarps = gridDim.x * 4;
    for (uint32_t i = blockIdx.x * 4 + (threadIdx.x >> 5); i < nlist; i += nwarps) {
        if (!PF_IN(i, sb.rows)) break;
        const uint2 e = sb.list[i];
        const InstDesc &d = insts[e.x];
        if (d.smdeg != N) continue;
        const uint32_t s0 = start[d.soff + e.y], s1 = start[d.soff + e.y + 1];
        if (!(PF_IN(int64_t(s0) - d.poff, d.n + 1) && PF_IN(int64_t(s1) - d.poff, d.n + 1)))
            continue;
        float acc[G * 32];
#pragma unroll
        for (int k = 0; k < G * 32; ++k) acc[k] = 0.f;
        for (uint32_t j = s0 + lane; j < s1; j += 32) {
            const float4 r = rec[j];
            const float sx = 2.f * r.x, sy = 2.f * r.y;
            float px[N + 1], py[N + 1];
            px[0] = 1.f;
            px[1] = sx;
            py[0] = r.z;
            py[1] = r.z * sy;
#pragma unroll
            for (int k = 1; k < N; ++k) {
                const float ca = float(2 * k + 1) / float(k + 1), cb = -float(k) / float(k + 1);
                px[k + 1] = fmaf(ca * sx, px[k], cb * px[k - 1]);
                py[k + 1] = fmaf(ca * sy, py[k], cb * py[k - 1]);
            }
#pragma unroll
            for (int b = 0; b <= N; ++b)
#pragma unroll
                for (int a = 0; a <= N - b; ++a)
                    acc[sm_idx(N, a, b)] = fmaf(px[a], py[b], acc[sm_idx(N, a, b)]);
        }
        float *out = sb.mom + size_t(i) * sb.row;
#pragma unroll
        for (int g = 0; g < G; ++g) {
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int k = 0; k < o; ++k) {
                    const float lo = acc[g * 32 + k], hi = acc[g * 32 + k + o];
                    acc[g * 32 + k] = (up ? hi : lo) +
                                      __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
                }
            }
            if (g * 32 + lane < M) out[g * 32 + lane] = acc[g * 32];
        }
    }
}

// ----------------------------------------------------------------------------
// Translation: loc[target] = sum over its neighbours of C^D moments
// ----------------------------------------------------------------------------
// A tiled FP32 product per block: 64 target leaves (consecutive in the
// occupied list, so mostly neighbours that share sources in L1) x all terms,
// 4 x 4 outputs per thread, the source moments of one neighbour offset and
// its operator staged in shared memory at a time.  Bound by the wait for the
// staged operands and the shared loads (two 16-byte loads per 16 multiply-adds):
// 2M clustered blobs, L1 46 %, FMA pipe 22 %.
template <int N>
struct SmTile {
    static constexpr int M = sm_terms(N), S = sm_stride(N), CG = S / 4;
    static constexpr int THREADS = (CG * (SM_TGT / 4) + 31) / 32 * 32;
    static constexpr int KT = N <= 8 ? 48 : N == 10 ? 36 : N == 12 ? 48 : 40;  // multiple of 4
};

template <int N>
__global__ void __launch_bounds__(SmTile<N>::THREADS) k_sm_translate(
    const uint32_t *__restrict__ ctrl, const InstDesc *__restrict__ insts, const SmBufs sbuf) {
    using T = SmTile<N>;
    constexpr int M = T::M, S = T::S, KT = T::KT;
    __shared__ __align__(16) float sa[KT][SM_TGT + 4];
    __shared__ __align__(16) float sb[KT * S];
    __shared__ uint2 se[SM_TGT];         // (instance, leaf)
    __shared__ uint32_t sm[SM_TGT];      // expansion neighbours
    __shared__ int ssrc[SM_TGT];         // rank of the source leaf of this offset, or -1
    const int tid = threadIdx.x;
    const int tg = tid & 15, cg = tid >> 4;
    const bool active = cg < T::CG;
    const uint32_t nrows = min(ctrl[CTRL_NSMOOTH], uint32_t(sbuf.rows));
    const uint32_t *__restrict__ lmask = sbuf.lmask;
    const uint32_t *__restrict__ lrank = sbuf.lrank;
    const float *__restrict__ mom = sbuf.mom;
    const int row = sbuf.row;
    for (uint32_t base = blockIdx.x * SM_TGT; base < nrows; base += gridDim.x * SM_TGT) {
        __syncthreads();  // the previous group's readers are done
        uint32_t mine = 0;
        if (tid < SM_TGT) {
            uint2 e = make_uint2(0xffffffffu, 0);
            if (base + tid < nrows) {
                e = sbuf.list[base + tid];
                const InstDesc &d = insts[e.x];
                if (d.smdeg == N) mine = lmask[d.loff + e.y] >> LM_EXP;
            }
            se[tid] = e;
            sm[tid] = mine;
        }
        if (!__syncthreads_or(int(mine))) continue;
        // one instance at a time (its operators); nearly always only one
        uint32_t done = 0xffffffffu;  // instances are taken in ascending order
        for (;;) {
            uint32_t inst = 0xffffffffu;
            for (int t = 0; t < SM_TGT; ++t)
                if (sm[t] && (done == 0xffffffffu || se[t].x > done)) inst = min(inst, se[t].x);
            if (inst == 0xffffffffu) break;
            done = inst;
            const InstDesc &d = insts[inst];
            const float *op = static_cast<const float *>(d.t_sm);
            float acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
            for (int o = 0; o < 9; ++o) {
                __syncthreads();
                int src = -1;
                if (tid < SM_TGT) {
                    if (se[tid].x == inst && ((sm[tid] >> o) & 1u)) {
                        const uint32_t m = se[tid].y;
                        const uint32_t nm = morton_key(compact_bits(m) + uint32_t(o % 3 - 1),
                                                       compact_bits(m >> 1) + uint32_t(o / 3 - 1));
                        if (PF_IN(nm, int64_t(1) << (2 * d.L)) &&
                            PF_IN(lrank[d.loff + nm], int64_t(nrows)))
                            src = int(lrank[d.loff + nm]);
                    }
                    ssrc[tid] = src;
                }
                if (!__syncthreads_or(src >= 0)) continue;
                for (int k0 = 0; k0 < M; k0 += KT) {
                    const int kt = min(KT, M - k0);
                    if (k0) __syncthreads();
                    for (int e = tid; e < SM_TGT * (KT / 4); e += T::THREADS) {
                        const int t = e & (SM_TGT - 1), k = (e / SM_TGT) * 4;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (k < kt && ssrc[t] >= 0)
                            v = *reinterpret_cast<const float4 *>(mom + size_t(ssrc[t]) * row + k0 +
                                                                  k);
                        sa[k][t] = v.x;
                        sa[k + 1][t] = v.y;
                        sa[k + 2][t] = v.z;
                        sa[k + 3][t] = v.w;
                    }
                    const float4 *ob =
                        reinterpret_cast<const float4 *>(op + (size_t(o) * M + k0) * S);
                    for (int e = tid; e < kt * (S / 4); e += T::THREADS)
                        reinterpret_cast<float4 *>(sb)[e] = __ldg(ob + e);
                    __syncthreads();
                    if (active)
#pragma unroll 4
                        for (int k = 0; k < kt; ++k) {
                            const float4 a = *reinterpret_cast<const float4 *>(&sa[k][tg * 4]);
                            const float4 b = *reinterpret_cast<const float4 *>(&sb[k * S + cg * 4]);
                            const float av[4] = {a.x, a.y, a.z, a.w};
                            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                            for (int p = 0; p < 4; ++p)
#pragma unroll
                                for (int c = 0; c < 4; ++c)
                                    acc[p][c] = fmaf(av[p], bv[c], acc[p][c]);
                        }
                }
            }
            if (active)
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int t = tg * 4 + p;
                    if (sm[t] && se[t].x == inst)
                        *reinterpret_cast<float4 *>(sbuf.loc + size_t(base + t) * row + cg * 4) =
                            make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
                }
        }
    }
}

// ----------------------------------------------------------------------------
// Final pass of these instances, one thread per blob
// ----------------------------------------------------------------------------
// Gradient of sum c[a, b] s^a t^b by nested Horner schemes.
template <int N>
__device__ __forceinline__ float2 sm_gradient(const float *__restrict__ loc, float s, float t) {
    constexpr int S4 = sm_stride(N) / 4;
    float c[sm_stride(N)];
#pragma unroll
    for (int k = 0; k < S4; ++k) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(loc) + k);
        c[4 * k] = v.x;
        c[4 * k + 1] = v.y;
        c[4 * k + 2] = v.z;
        c[4 * k + 3] = v.w;
    }
    float f = 0.f, fs = 0.f, ft = 0.f;
#pragma unroll
    for (int b = N; b >= 0; --b) {
        float h = c[sm_idx(N, N - b, b)], hd = 0.f;
#pragma unroll
        for (int a = N - b - 1; a >= 0; --a) {
            hd = fmaf(hd, s, h);
            h = fmaf(h, s, c[sm_idx(N, a, b)]);
        }
        ft = fmaf(ft, t, f);
        f = fmaf(f, t, h);
        fs = fmaf(fs, t, hd);
    }
    return make_float2(fs, ft);
}

// Bound by load latency: the coefficients are mostly one address per warp, the
// row number is looked up before the far field, and registers are capped for
// four blocks an SM.  16.8M clustered blobs, with the two scatters: 806 ->
// 688 us (three blocks 738; five 658, but 216 bytes of spills and the small
// cases a little slower).
__global__ void __launch_bounds__(256, 4) k_sm_final(
    const Task *__restrict__ tasks, int ntasks, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const uint32_t *__restrict__ skeys,
    const float4 *__restrict__ rec, const float2 *__restrict__ le,
    const SmBufs sb, int dtype_f32, float *__restrict__ stage, int64_t nstage) {
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t j = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    if (j >= t.count) return;
    const InstDesc &d = insts[t.inst];
    if (!d.smdeg) return;
    const int64_t r = d.poff + j;
    const uint32_t m = skeys[r] & ((1u << (2 * d.L)) - 1u);
    const float4 rr = rec[r];
    const uint32_t mask = sb.lmask[d.loff + m], rank = sb.lrank[d.loff + m];  // (if by expansions)
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    float2 w = make_float2(0.f, 0.f);
    if (d.L >= 2) {
        // far field: w = (1/r) sum c_m zeta^m, u - i v = cfar w
        const int p = d.p;
        const float2 *c =
            le + d.eoff + (lvl_off(d.L) + box_index(d.L, uint32_t(ix), uint32_t(iy))) * p;
        const float2 z = far_series(c, p, rr.x, rr.y);
        w = make_float2(d.cfar * z.y, d.cfar * z.x);
    }
    if ((mask >> LM_EXP) && PF_IN(rank, sb.rows)) {
        const float *l = sb.loc + size_t(rank) * sb.row;
        const float s = 2.f * rr.x, q = 2.f * rr.y;
        float2 g;
        switch (d.smdeg) {
            case 8: g = sm_gradient<8>(l, s, q); break;
            case 10: g = sm_gradient<10>(l, s, q); break;
            case 12: g = sm_gradient<12>(l, s, q); break;
            default: g = sm_gradient<14>(l, s, q); break;
        }
        const float c2 = 2.f * d.cnear;  // d/dxi = 2 d/ds
        w.x = fmaf(-c2, g.y, w.x);
        w.y = fmaf(c2, g.x, w.y);
    }
    const uint32_t dm = mask & 0x1ffu;
    if (dm) {
        uint32_t total;
        const NearLeaves q{&d, start + d.soff, ix, iy, dm, 0u, ~0u};
        const float2 n = near_vortex_of(q, rec, rr.x, rr.y, total);
        w.x = fmaf(d.cfar, n.x, w.x);  // cnear / kappa = cfar
        w.y = fmaf(d.cfar, n.y, w.y);
    }
    if (stage) {
        stage[r] = w.x;
        stage[nstage + r] = w.y;
        return;
    }
    const int64_t q = int64_t(__float_as_uint(rr.w)) - d.poff;
    if (!PF_IN(q, d.n)) return;  // checked build: the caller's index of the blob
    if (dtype_f32) {
        static_cast<float *>(d.u)[q] = w.x;
        static_cast<float *>(d.v)[q] = w.y;
    } else {
        static_cast<double *>(d.u)[q] = double(w.x);
        static_cast<double *>(d.v)[q] = double(w.y);
    }
}

// ----------------------------------------------------------------------------
// Launches
// ----------------------------------------------------------------------------
template <int N>
static cudaError_t sm_near(const uint32_t *ctrl, const InstDesc *insts, const uint32_t *start,
                           const float4 *rec, const SmBufs &sb, cudaStream_t st,
                           uint64_t *launches) {
    // (found once, by whichever thread comes first; the others wait for it)
    static const int2 per_sm = [] {
        int2 n = make_int2(0, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n.x, k_sm_moments<N>, 128, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n.y, k_sm_translate<N>, SmTile<N>::THREADS, 0);
        return make_int2(std::max(n.x, 1), std::max(n.y, 1));
    }();
    const int64_t sms = device_sm_count();
    if (sb.rows <= 0) return cudaSuccess;
    const int64_t gm = std::min<int64_t>(sms * per_sm.x, (sb.rows + 3) / 4);
    k_sm_moments<N><<<unsigned(gm), 128, 0, st>>>(ctrl, insts, start, rec, sb);
    PF_LAUNCHED(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t gt = std::min<int64_t>(sms * per_sm.y, (sb.rows + SM_TGT - 1) / SM_TGT);
    k_sm_translate<N><<<unsigned(gt), SmTile<N>::THREADS, 0, st>>>(ctrl, insts, sb);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

cudaError_t launch_sm_near(uint32_t degrees, const uint32_t *ctrl, const InstDesc *insts,
                           const uint32_t *start, const float4 *rec, const SmBufs &sb,
                           cudaStream_t st, uint64_t *launches) {
    cudaError_t e = cudaSuccess;
    if (degrees & (1u << 8)) e = sm_near<8>(ctrl, insts, start, rec, sb, st, launches);
    if (e == cudaSuccess && (degrees & (1u << 10)))
        e = sm_near<10>(ctrl, insts, start, rec, sb, st, launches);
    if (e == cudaSuccess && (degrees & (1u << 12)))
        e = sm_near<12>(ctrl, insts, start, rec, sb, st, launches);
    if (e == cudaSuccess && (degrees & (1u << 14)))
        e = sm_near<14>(ctrl, insts, start, rec, sb, st, launches);
    return e;
}

cudaError_t launch_sm_final(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, const uint32_t *skeys, const float4 *rec,
                            const float2 *le, const SmBufs &sb, int dtype_f32, float *stage,
                            int64_t nstage, cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_sm_final<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, skeys, rec, le, sb,
                                                  dtype_f32, stage, nstage);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

PF_DEFINE_CHECK_READER(smooth)

}  // namespace petfmm
