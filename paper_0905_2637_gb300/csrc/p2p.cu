// p2p.cu -- evaluation step of Sec. 2.2: the direct near-field sum over the
// leaf and its 8 neighbours with the regularised kernel of Eq. 8, fused with
// L2P of the leaf's local expansion, written back in the caller's order.
//
// Mixed path: a thread per target (k_near_direct) unless the core is wide
// against the leaf (smooth.cu) or PETFMM_OPT_P2P_PAIRS asks for items (0) or
// for leaf pairs (1).
//
// Work list (FP64, and option 0).  Every occupied leaf is cut into items
// of at most TPI targets (one warp per item); an item's cost is (targets) x (sources in the 9
// leaves), the n_nd N_i^2 term of the work estimate of Eq. 14.  Warps of a
// persistent grid take items from a queue, so equal-cost items of one leaf
// spread across SMs and the heavy leaves of clustered inputs do not pin one
// SM.  An item with few targets (small leaves: a uniform layout holds about
// 16 blobs per leaf) would leave most lanes idle, so its warp splits into S
// groups of lanes: each group holds all the item's targets and takes every
// S-th source, and the S partial sums of a target are added by a fixed
// butterfly of warp shuffles.  The order of every sum depends only on the
// item's target count: results do not depend on which warp ran the item.
//
// Mixed path (FP32).  Coordinates are leaf-relative in leaf units; with
// rho^2 = |dx|^2 in leaf units and q = kappa rho^2, kappa = w^2 / 2 sigma^2,
//     u_i = w / (4 pi sigma^2) sum_j gamma_j (-d_eta, d_xi) g(q),
//     g(q) = (1 - exp(-q)) / q,
// which is Eq. 8 rearranged (no division, no cancellation at small q).  g is
// evaluated as a polynomial in rho^2 fitted on the host (Chebyshev
// interpolation of g on the range the near field can reach), i.e. on the FMA
// pipe only; if the near field reaches beyond the fitted range the "general"
// variant switches to (1 - exp(-q)) / q from the special-function unit above
// the split.  The self pair has d = 0 and adds exactly zero.
//
// FP64 path: the same loop in FP64, g from a table (see k_p2p_f64).
#include <cmath>
#include <type_traits>
#include <vector>

#include "kernels.cuh"
#include "near_direct.cuh"

namespace petfmm {

#define PF_LAUNCHED(n) do { if (launches) *launches += (n); } while (0)

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ----------------------------------------------------------------------------
// Work list
// ----------------------------------------------------------------------------
// log2 of the lanes that hold the targets of an item with nt targets, r per
// lane: the smallest power of two >= ceil(nt / r), at most 32.  The other
// 32 / 2^lw lane groups split the item's sources.
__host__ __device__ __forceinline__ int p2p_group_log2(uint32_t nt, int r) {
    const uint32_t h = (nt + uint32_t(r) - 1) / uint32_t(r);
    int lw = 0;
    while (lw < 5 && (1u << lw) < h) ++lw;
    return lw;
}

// Forward neighbours of a leaf in the pairwise near field (see below).
__constant__ int8_t c_fwd[4][2] = {{1, 0}, {-1, 1}, {0, 1}, {1, 1}};

// A pair of neighbouring leaves is evaluated pairwise when both hold at least
// pmin (InstDesc::pair_min) blobs; the others are summed directly, one thread
// per target (k_near_direct).  Both leaves of a pair decide from the same two
// counts.  PETFMM_OPT_P2P_PAIRS = 1 sets pmin to a warp's worth, 32.  The
// automatic choice never does: wide cores (kappa <= 1.95) go by expansions, and
// beyond them neither kernel is always the better one.  Whole evaluations,
// direct / pairs, ms: where few heavy items decide, 349,185 clustered blobs, 530
// per leaf, kappa = 6: 1.38 / 2.65; 131,072 even blobs, 512 per leaf, kappa = 3.9:
// 0.51 / 0.81; 64 per leaf, kappa = 12: 0.60 / 0.63.  In dense trees with many
// leaves pairs win: 1,048,576 even blobs, 256 per leaf, kappa = 3.9: 1.66 / 1.39;
// 4,000,000 clustered ones, 560 per leaf: 8.96 / 7.28.  Which it is depends on how
// the blobs lie, which the plan does not know; the option is there for dense
// trees.
__host__ __device__ __forceinline__ bool pairwise(uint32_t na, uint32_t nb, uint32_t pmin) {
    return na >= pmin && nb >= pmin;
}

// A heavy pair is cut into pieces along A, each piece a run of whole
// 128-target chunks holding at most P2P_PAIR_CAPU tiles of 128 targets x 32
// sources, so that no single warp's item outlasts the average share of the
// launch.  Piece 0 writes B's reaction to the pair's slot, piece i >= 1 to a
// scratch run of nb entries; the final pass adds them in piece order.
// Returns the number of pieces; *pc = targets per piece (a multiple of 128).
constexpr uint64_t P2P_PAIR_CAPU = 256;
__host__ __device__ __forceinline__ uint32_t pair_pieces(uint32_t na, uint32_t nb, uint32_t *pc) {
    const uint32_t ca = (na + 127) / 128, cb = (nb + 31) / 32;
    uint64_t np = (uint64_t(ca) * cb + P2P_PAIR_CAPU - 1) / P2P_PAIR_CAPU;
    if (np > ca) np = ca;
    if (np < 1) np = 1;
    const uint32_t per = uint32_t((ca + np - 1) / np);
    *pc = per * 128;
    return (ca + per - 1) / per;
}

// count of the leaf (x, y), 0 outside the domain
__device__ __forceinline__ uint32_t leaf_count(const uint32_t *st, int nside, int x, int y) {
    if (x < 0 || y < 0 || x >= nside || y >= nside) return 0;
    const uint32_t m = morton_key(uint32_t(x), uint32_t(y));
    return st[m + 1] - st[m];
}

// Per-leaf flags of the pairwise mode, read by the final pass: which result
// slots hold this leaf's blobs' sums.
enum : uint32_t {
    LF_FWD = 1u,        // << k: pairs with forward neighbour k (slot k)
    LF_BWD = 16u,       // << k: pairs with backward neighbour k (slot 4 + k)
    LF_SPLIT = 256u,    // << k: ... cut into pieces, partial sums in the scratch
    LF_SELF = 4096u     // the leaf's own pairs (slot 8)
};

// The work list takes two launches, both walking every leaf's items in the same
// way: the first counts the items of each work class, the second puts the
// items down class after class, heaviest first, their places within a class by
// atomics (the order of items changes no result).  ordered = 0
// (PETFMM_OPT_P2P_MODE = 1): one class, about leaf order.  Launches bound it:
// 10,000 blobs 35 us with a scan and a radix pass, 16 us now.
constexpr int WORK_CLASSES = 128;

// log2(cost) in quarter steps, heaviest = smallest class
__device__ __forceinline__ uint32_t work_class(uint32_t cost) {
    if (cost < 1) cost = 1;
    const int e = 31 - __clz(int(cost));
    const uint32_t frac = e >= 2 ? (cost >> (e - 2)) & 3u : (cost << (2 - e)) & 3u;
    return 127u - (uint32_t(e) * 4u + frac);
}

// Calls emit(class, first item, count) for every run of alike items of leaf m (its
// whole ones, then the rest: warps that take them together share its sources in
// L1); the leaf's ordered pairs.
// The class is that of the n_nd N_i^2 term of Eq. 14 (targets x sources):
// every lane of the warp runs the source loop of its group, target slot filled
// or not, so the cost is the sources per lane group, ceil(src / S) with S
// groups.
template <typename F>
__device__ __forceinline__ unsigned long long leaf_items(const InstDesc &d, const uint32_t *st,
                                                         uint32_t m, uint32_t inst, uint32_t tpi,
                                                         int ordered, F &&emit) {
    const uint32_t s0 = st[m], n = st[m + 1] - s0;
    if (!n || d.direct) return 0;
    const int nside = 1 << d.L;
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    uint32_t src = 0;  // the blobs of the leaf and its neighbours
    for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) src += leaf_count(st, nside, ix + dx, iy + dy);
    const uint32_t whole = n / tpi, rest = n - whole * tpi;
    auto run = [&](uint32_t f, uint32_t nt, uint32_t count) {
        const int ns = 5 - p2p_group_log2(nt, int(tpi) / 32);  // log2 S
        emit(ordered ? work_class((src + (1u << ns) - 1) >> ns) : 0u,
             make_uint4(inst, m, s0 + f, nt), count);
    };
    if (whole) run(0, tpi, whole);
    if (rest) run(whole * tpi, rest, 1);
    return (unsigned long long)n * (src - 1);
}

__global__ void __launch_bounds__(256) k_item_count(const Task *__restrict__ tasks, int ntasks,
                                                    const InstDesc *__restrict__ insts,
                                                    const uint32_t *__restrict__ start,
                                                    uint32_t tpi, int ordered, uint32_t *ctrl) {
    __shared__ uint32_t hist[WORK_CLASSES];
    __shared__ unsigned long long sums;
    for (int i = threadIdx.x; i < WORK_CLASSES; i += 256) hist[i] = 0;
    if (threadIdx.x == 0) sums = 0;
    __syncthreads();
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    unsigned long long pairs = 0;
    if (m < t.count) {
        const InstDesc &d = insts[t.inst];
        pairs = leaf_items(d, start + d.soff, uint32_t(m), uint32_t(t.inst), tpi, ordered,
                           [&](uint32_t c, const uint4 &, uint32_t k) { atomicAdd(&hist[c], k); });
    }
    // the ordered pair count, for the statistics
#pragma unroll
    for (int o = 16; o; o >>= 1) pairs += __shfl_down_sync(0xffffffffu, pairs, o);
    if ((threadIdx.x & 31) == 0 && pairs) atomicAdd(&sums, pairs);
    __syncthreads();
    if (threadIdx.x < WORK_CLASSES && hist[threadIdx.x]) {
        atomicAdd(ctrl + CTRL_CLASSES + threadIdx.x, hist[threadIdx.x]);
        atomicAdd(ctrl + CTRL_NITEMS, hist[threadIdx.x]);
    }
    if (threadIdx.x == 0 && sums)
        atomicAdd(reinterpret_cast<unsigned long long *>(ctrl + CTRL_PAIRS_LO), sums);
}

__global__ void __launch_bounds__(256) k_item_emit(const Task *__restrict__ tasks, int ntasks,
                                                   const InstDesc *__restrict__ insts,
                                                   const uint32_t *__restrict__ start,
                                                   uint32_t tpi, int ordered, uint32_t *ctrl,
                                                   uint4 *__restrict__ items, int64_t cap) {
    __shared__ uint32_t hist[WORK_CLASSES], first[WORK_CLASSES];
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    const InstDesc &d = insts[t.inst];
    const uint32_t *st = start + d.soff;
    if (threadIdx.x < WORK_CLASSES) {
        hist[threadIdx.x] = 0;
        first[threadIdx.x] = ctrl[CTRL_CLASSES + threadIdx.x];
    }
    __syncthreads();
    if (m < t.count)
        leaf_items(d, st, uint32_t(m), uint32_t(t.inst), tpi, ordered,
                   [&](uint32_t c, const uint4 &, uint32_t k) { atomicAdd(&hist[c], k); });
    __syncthreads();
    // this block's run within each class
    uint32_t base = 0, n = 0;
    if (threadIdx.x < WORK_CLASSES && (n = hist[threadIdx.x])) {
        for (int i = 0; i < int(threadIdx.x); ++i) base += first[i];
        base += atomicAdd(ctrl + CTRL_CLASSES + WORK_CLASSES + threadIdx.x, n);
    }
    __syncthreads();
    if (threadIdx.x < WORK_CLASSES) {
        first[threadIdx.x] = base;
        hist[threadIdx.x] = 0;
    }
    __syncthreads();
    if (m < t.count)
        leaf_items(d, st, uint32_t(m), uint32_t(t.inst), tpi, ordered,
                   [&](uint32_t c, uint4 item, uint32_t k) {
                       const uint32_t o = first[c] + atomicAdd(&hist[c], k);
                       for (uint32_t i = 0; i < k; ++i, item.z += tpi)
                           if (PF_IN(o + i, cap)) items[o + i] = item;
                   });
}

cudaError_t launch_p2p_worklist(const Task *tasks, int ntasks, int64_t nblocks,
                                const InstDesc *insts, const uint32_t *start, int tpi, int ordered,
                                uint4 *items, int64_t cap, uint32_t *ctrl, cudaStream_t st,
                                uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_item_count<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, uint32_t(tpi),
                                                    ordered, ctrl);
    PF_LAUNCHED(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_item_emit<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, uint32_t(tpi),
                                                   ordered, ctrl, items, cap);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Mixed-precision P2P + L2P
// ----------------------------------------------------------------------------
constexpr int P2P_THREADS = 256;

template <int DEG>
__device__ __forceinline__ float poly_eval(const float (&a)[DEG + 1], float s) {
    float g = a[DEG];
#pragma unroll
    for (int k = DEG - 1; k >= 0; --k) g = fmaf(g, s, a[k]);
    return g;
}

template <int DEG, bool GENERAL>
__device__ __forceinline__ float g_of(const float (&a)[DEG + 1], float r2, float kappa, float split) {
    float g = poly_eval<DEG>(a, r2);
    if (GENERAL) {
        const float q = kappa * r2;
        const float ge = __fdividef(1.0f - __expf(-q), q);
        g = r2 < split ? g : ge;
    }
    return g;
}

// One source against the lane's two targets (a, b), both in the source
// leaf's frame.
template <int DEG, bool GENERAL>
__device__ __forceinline__ void pair2(const float4 s, float xa, float ya, float xb, float yb,
                                      const float (&a)[DEG + 1], float kappa, float split,
                                      float &ua, float &va, float &ub, float &vb) {
    const float dxa = xa - s.x, dya = ya - s.y;
    const float dxb = xb - s.x, dyb = yb - s.y;
    const float r2a = fmaf(dxa, dxa, dya * dya);
    const float r2b = fmaf(dxb, dxb, dyb * dyb);
    const float fa = s.z * g_of<DEG, GENERAL>(a, r2a, kappa, split);
    const float fb = s.z * g_of<DEG, GENERAL>(a, r2b, kappa, split);
    ua = fmaf(-dya, fa, ua);
    va = fmaf(dxa, fa, va);
    ub = fmaf(-dyb, fb, ub);
    vb = fmaf(dxb, fb, vb);
}

// One work item of the directed near field: up to 64 targets of a leaf
// against the leaf and its neighbours; the near sum goes to own[] in sorted
// order, the final pass
// adds the far field.  No L2P here: with few targets per item the lanes of
// all source groups would repeat it.
// Laplace kernel: one source against the lane's two targets, both in the
// source leaf's frame (leaf units): u += q (log rho + log w), i.e. q log r in
// global units; coincident pairs add nothing.
__device__ __forceinline__ void pair2_lap(const float4 s, float xa, float ya, float xb, float yb,
                                          float logw, float &ua, float &ub) {
    const float dxa = xa - s.x, dya = ya - s.y;
    const float dxb = xb - s.x, dyb = yb - s.y;
    const float r2a = fmaf(dxa, dxa, dya * dya);
    const float r2b = fmaf(dxb, dxb, dyb * dyb);
    const float la = r2a > 0.f ? fmaf(0.5f, __logf(r2a), logw) : 0.f;
    const float lb = r2b > 0.f ? fmaf(0.5f, __logf(r2b), logw) : 0.f;
    ua = fmaf(s.z, la, ua);
    ub = fmaf(s.z, lb, ub);
}

template <int DEG, bool GENERAL, bool LAP>
__device__ __forceinline__ void directed_item(const uint4 item, const InstDesc *__restrict__ insts,
                                              const uint32_t *__restrict__ start,
                                              const float4 *__restrict__ rec,
                                              float2 *__restrict__ own, int lane) {
    const InstDesc &d = insts[item.x];
    const int L = d.L;
    float a[DEG + 1];
#pragma unroll
    for (int k = 0; k <= DEG; ++k) a[k] = d.poly[k];
    const float kappa = d.kappa, split = d.qsplit_rho2;
    const uint32_t m = item.y;
    // checked build: the item's leaf and target range lie inside the instance
    if (!(PF_IN(m, int64_t(1) << (2 * L)) && PF_IN(int64_t(item.z) - d.poff, d.n + 1) &&
          PF_IN(int64_t(item.z) + item.w - d.poff, d.n + 1)))
        return;
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    // lane = (source group grp, target slot k); targets k and k + W
    const int lw = p2p_group_log2(item.w, 2);
    const uint32_t W = 1u << lw, S = 32u >> lw;
    const uint32_t grp = uint32_t(lane) >> lw, k = uint32_t(lane) & (W - 1u);
    const uint32_t ta = item.z + k, tb = item.z + k + W;
    const bool has_a = k < item.w, has_b = k + W < item.w;
    const float4 ra = has_a ? rec[ta] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 rb = has_b ? rec[tb] : make_float4(0.f, 0.f, 0.f, 0.f);
    float ua = 0.f, va = 0.f, ub = 0.f, vb = 0.f;
    const uint32_t *st = start + d.soff;
    const int nside = 1 << L;
    const float logw = LAP ? float(d.logw0 - double(L) * 0.69314718055994530942) : 0.f;
    // The Laplace kernel's lanes 0..8 fetch the 9 leaves' source ranges at
    // once (lane q: offset (q % 3 - 1, q / 3 - 1)), so an item pays one load
    // latency, not nine; the vortex kernel keeps the plain loop, which
    // measured faster there.
    constexpr bool FETCH9 = LAP;
    uint32_t lj0 = 0, lj1 = 0;
    if (FETCH9 && lane < 9) {
        const int sx = ix + lane % 3 - 1, sy = iy + lane / 3 - 1;
        if (sx >= 0 && sy >= 0 && sx < nside && sy < nside) {
            const uint32_t nm = morton_key(uint32_t(sx), uint32_t(sy));
            lj0 = st[nm];
            lj1 = st[nm + 1];
        }
    }
    for (int q = 0; q < 9; ++q) {
        const int dx = q % 3 - 1, dy = q / 3 - 1;
        uint32_t j0, j1;
        if (FETCH9) {
            j0 = __shfl_sync(0xffffffffu, lj0, q);
            j1 = __shfl_sync(0xffffffffu, lj1, q);
        } else {
            const int sx = ix + dx, sy = iy + dy;
            if (sx < 0 || sy < 0 || sx >= nside || sy >= nside) continue;
            const uint32_t nm = morton_key(uint32_t(sx), uint32_t(sy));
            j0 = st[nm];
            j1 = st[nm + 1];
        }
        if (j0 == j1) continue;
        {
            const float xa = ra.x - float(dx), ya = ra.y - float(dy);
            const float xb = rb.x - float(dx), yb = rb.y - float(dy);
            // the stride-1 loop keeps constant load offsets after unrolling
            if (S == 1) {
#pragma unroll 4
                for (uint32_t j = j0; j < j1; ++j) {
                    if constexpr (LAP)
                        pair2_lap(__ldg(rec + j), xa, ya, xb, yb, logw, ua, ub);
                    else
                        pair2<DEG, GENERAL>(__ldg(rec + j), xa, ya, xb, yb, a, kappa, split, ua,
                                            va, ub, vb);
                }
            } else {
#pragma unroll 4
                for (uint32_t j = j0 + grp; j < j1; j += S) {
                    if constexpr (LAP)
                        pair2_lap(__ldg(rec + j), xa, ya, xb, yb, logw, ua, ub);
                    else
                        pair2<DEG, GENERAL>(__ldg(rec + j), xa, ya, xb, yb, a, kappa, split, ua,
                                            va, ub, vb);
                }
            }
        }
    }
    // add the partial sums of the source groups (fixed butterfly)
    for (uint32_t o = W; o < 32u; o <<= 1) {
        ua += __shfl_xor_sync(0xffffffffu, ua, int(o));
        va += __shfl_xor_sync(0xffffffffu, va, int(o));
        ub += __shfl_xor_sync(0xffffffffu, ub, int(o));
        vb += __shfl_xor_sync(0xffffffffu, vb, int(o));
    }
    const float cn = LAP ? 1.f : d.cnear;
    if (has_a && grp == 0) own[ta] = make_float2(cn * ua, cn * va);
    if (has_b && grp == 0) own[tb] = make_float2(cn * ub, cn * vb);
}

template <int DEG, bool GENERAL, bool LAP>
__global__ void __launch_bounds__(P2P_THREADS, 5) k_p2p_mixed(
    const uint4 *__restrict__ items, uint32_t *ctrl, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const float4 *__restrict__ rec,
    float2 *__restrict__ own, unsigned long long *busy) {
    const int lane = threadIdx.x & 31;
    const uint32_t nitems = *reinterpret_cast<volatile uint32_t *>(ctrl + CTRL_NITEMS);
    const uint64_t t_begin = busy ? global_ns() : 0;
    // a warp's first item by its position, block by block (few items then spread
    // over the SMs), the others from the queue
    const uint32_t nwarps = gridDim.x * (P2P_THREADS / 32);
    uint32_t it = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (it < nitems) {
        directed_item<DEG, GENERAL, LAP>(items[it], insts, start, rec, own, lane);
        if (lane == 0) it = nwarps + atomicAdd(ctrl + CTRL_QUEUE, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
    }
    if (busy && lane == 0) {
        const uint64_t t_end = global_ns();
        const size_t gw = size_t(blockIdx.x) * (P2P_THREADS / 32) + (threadIdx.x >> 5);
        busy[2 * gw] = t_begin;
        busy[2 * gw + 1] = t_end;
    }
}

// ----------------------------------------------------------------------------
// FP64 P2P + L2P (one target per lane).
// ----------------------------------------------------------------------------
// Bound by the FP64 pipe (two lanes a cycle and SM on this part; every other
// instruction is nearly free beside it), so a pair's factor g(q) = (1 - e^-q)
// / q comes without division or exponential: below q = 40 a polynomial of
// degree 6 in q on 640 cells of width 1/16, read from shared memory (within 2
// ulp, tests/test_gpu_factors.py), above it 1 / q (e^-40 is below the rounding)
// from the hardware's approximate reciprocal y and the series step
// y (1 + e + e^2), e = 1 - q y.  15 operations a pair where expm1 and a
// division took about 45.  Items hold 16 targets: two lanes a target, so that
// leaves of 16 fill their warps and small problems have warps for every SM.
// Measured on one GB300: 1,048,576 blobs, 16 per leaf: 10.6 -> 4.2 ms; 10,000
// blobs, 39 per leaf: 3.14 -> 0.16 ms.
__device__ __forceinline__ double g_f64(double q, const double *__restrict__ tab) {
    const uint32_t h = uint32_t(__double2hiint(q));
    if (h < 0x40440000u) {  // q < 40: floor(16 q) from the bits
        const uint32_t sh = 1039u - (h >> 20);
        const int c = int(sh < 32u ? ((h & 0xfffffu) | 0x100000u) >> sh : 0u);
        const double t = q - tab[G64_TERMS * G64_CELLS + c];
        double g = tab[(G64_TERMS - 1) * G64_CELLS + c];
#pragma unroll
        for (int k = G64_TERMS - 2; k >= 0; --k) g = fma(g, t, tab[k * G64_CELLS + c]);
        return g;
    }
    if (h >= 0x7fd00000u) return 1.0 / q;  // the approximation flushes there
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(q));
    const double e = fma(-q, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// Taylor coefficients of g about each cell's middle from E_n = int_0^1 s^n
// e^(-q s) ds: E_top = e^-q sum_k q^k / ((top+1) .. (top+1+k)) and downwards
// E_(n-1) = (q E_n + e^-q) / n (positive terms only); to degree 12, the terms
// above degree 6 folded down by Chebyshev economisation (|t| <= 1/32).
// Layout: coefficient k of every cell, then the middles.  Built once.
const double *host_g64_table() {
    static const std::vector<double> table = [] {
        constexpr int top = 12;
        long double cheb[top + 1][top + 1] = {};  // T_n's powers
        cheb[0][0] = cheb[1][1] = 1.0L;
        for (int n = 2; n <= top; ++n)
            for (int i = 0; i <= n; ++i)
                cheb[n][i] = (i ? 2.0L * cheb[n - 1][i - 1] : 0.0L) - cheb[n - 2][i];
        std::vector<double> out(G64_WORDS);
        for (int c = 0; c < G64_CELLS; ++c) {
            const long double q = (c + 0.5L) / 16.0L, ex = std::exp(-q);
            long double term = 1.0L / (top + 1), en = 0.0L;
            for (int k = 1; term > 1e-21L * en; ++k) {
                en += term;
                term *= q / (top + 1 + k);
            }
            en *= ex;
            long double e[top + 1], a[top + 1], fact = 1.0L;
            for (int n = top; n >= 0; --n) {
                e[n] = en;
                if (n) en = (q * en + ex) / n;
            }
            for (int n = 0; n <= top; ++n) {  // in t 32, |t 32| <= 1
                if (n) fact *= -n;
                a[n] = std::ldexp(e[n] / fact, -5 * n);
            }
            for (int n = top; n >= G64_TERMS; --n) {
                const long double f = a[n] / cheb[n][n];
                for (int i = 0; i <= n; ++i) a[i] -= f * cheb[n][i];
            }
            for (int k = 0; k < G64_TERMS; ++k)
                out[size_t(k) * G64_CELLS + c] = double(std::ldexp(a[k], 5 * k));
            out[size_t(G64_TERMS) * G64_CELLS + c] = double(q);
        }
        return out;
    }();
    return table.data();
}

__global__ void __launch_bounds__(256) k_g64(const double *__restrict__ q, double *__restrict__ g,
                                             int64_t n, const double *__restrict__ tab) {
    const int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x;
    if (i < n) g[i] = g_f64(q[i], tab);
}

cudaError_t launch_g64(const double *q, double *g, int64_t n, const double *gtab, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_g64<<<unsigned((n + 255) / 256), 256, 0, st>>>(q, g, n, gtab);
    return cudaGetLastError();
}

template <bool LAP>
__global__ void __launch_bounds__(P2P_THREADS) k_p2p_f64(
    const uint4 *__restrict__ items, uint32_t *ctrl, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const double *__restrict__ xs,
    const double *__restrict__ ys, const double *__restrict__ gs, const uint32_t *__restrict__ perm,
    const double2 *__restrict__ le, const double *__restrict__ gtab, int dtype_f32,
    unsigned long long *busy) {
    __shared__ double tab[LAP ? 1 : G64_WORDS];
    const int lane = threadIdx.x & 31;
    const uint32_t nitems = *reinterpret_cast<volatile uint32_t *>(ctrl + CTRL_NITEMS);
    const uint64_t t_begin = busy ? global_ns() : 0;
    if (!LAP && blockIdx.x < nitems) {  // (a block past the first items' has no work)
        for (int i = threadIdx.x; i < G64_WORDS; i += P2P_THREADS) tab[i] = __ldg(gtab + i);
        __syncthreads();
    }
    // a warp's first item by its position, block by block (few items then
    // spread over the SMs), the others from the queue
    const uint32_t nwarps = gridDim.x * (P2P_THREADS / 32);
    uint32_t it = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (; it < nitems;) {
        const uint4 item = items[it];
        const InstDesc &d = insts[item.x];
        const int L = d.L;
        const uint32_t m = item.y;
        const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
        const int lw = p2p_group_log2(item.w, 1);
        const uint32_t W = 1u << lw, S = 32u >> lw;
        const uint32_t grp = uint32_t(lane) >> lw, k = uint32_t(lane) & (W - 1u);
        const bool has = k < item.w;
        const uint32_t ti = item.z + (has ? k : 0u);
        const double x = xs[ti], y = ys[ti];
        const double inv2s2 = d.inv2s2;
        // Laplace kernel: su = sum q_j log|x - x_j| (coincident pairs excluded)
        double su = 0.0, sv = 0.0;
        const uint32_t *st = start + d.soff;
        const int nside = 1 << L;
        auto sum = [&](auto guard) {
            su = sv = 0.0;
            for (int dy = -1; dy <= 1; ++dy) {
                const int sy = iy + dy;
                if (sy < 0 || sy >= nside) continue;
                for (int dx = -1; dx <= 1; ++dx) {
                    const int sx = ix + dx;
                    if (sx < 0 || sx >= nside) continue;
                    const uint32_t nm = morton_key(uint32_t(sx), uint32_t(sy));
                    const uint32_t j0 = st[nm], j1 = st[nm + 1];
#pragma unroll 2
                    for (uint32_t j = j0 + grp; j < j1; j += S) {
                        const double ddx = x - __ldg(xs + j), ddy = y - __ldg(ys + j);
                        const double r2 = fma(ddx, ddx, ddy * ddy);
                        if (LAP) {
                            if (r2 > 0.0) su += __ldg(gs + j) * (0.5 * log(r2));
                        } else {
                            // (the self pair and coincident blobs have ddx = ddy =
                            // 0 and add zero, unless the strength is infinite)
                            if (decltype(guard)::value && !(r2 > 0.0)) continue;
                            const double f = __ldg(gs + j) * g_f64(r2 * inv2s2, tab);
                            su = fma(-ddy, f, su);
                            sv = fma(ddx, f, sv);
                        }
                    }
                }
            }
        };
        sum(std::false_type());
        if (!LAP && (isnan(su) || isnan(sv))) sum(std::true_type());
        for (uint32_t o = W; o < 32u; o <<= 1) {
            su += __shfl_xor_sync(0xffffffffu, su, int(o));
            sv += __shfl_xor_sync(0xffffffffu, sv, int(o));
        }
        double fu = 0.0, fv = 0.0;
        if (L >= 2) {
            const int p = d.p;
            const double cx = d.x0 + (double(ix) + 0.5) * d.wleaf;
            const double cy = d.y0 + (double(iy) + 0.5) * d.wleaf;
            double zx = (x - cx) * d.scale, zy = (y - cy) * d.scale;
            const double2 *c = le + d.eoff + (lvl_off(L) + box_index(L, uint32_t(ix), uint32_t(iy))) * p;
            // with two lane groups or more, the groups take the even and the
            // odd coefficients, in zeta^2
            const int h = S > 1 ? 2 : 1, g = h == 2 ? int(grp & 1u) : 0;
            const double ox = zx, oy = zy;
            if (h == 2) {
                zx = fma(ox, ox, -(oy * oy));
                zy = 2.0 * ox * oy;
            }
            double2 w = make_double2(0.0, 0.0);
            int q = p - 1;
            if (h == 2 && (q & 1) != g) --q;
            if (q >= 0) w = c[q];
            for (q -= h; q >= 0; q -= h) {
                const double2 ck = c[q];
                w = make_double2(fma(w.x, zx, fma(-w.y, zy, ck.x)),
                                 fma(w.x, zy, fma(w.y, zx, ck.y)));
            }
            if (h == 2) {
                if (g) w = make_double2(fma(w.x, ox, -(w.y * oy)), fma(w.x, oy, w.y * ox));
                w.x += __shfl_xor_sync(0xffffffffu, w.x, int(W));
                w.y += __shfl_xor_sync(0xffffffffu, w.y, int(W));
            }
            if (LAP) {
                fu = w.x;  // the potential is Re of the local expansion
            } else {
                fu = d.cfar64 * w.y;
                fv = d.cfar64 * w.x;
            }
        }
        if (has && grp == 0) {
            const int64_t q = int64_t(perm[ti]) - d.poff;
            const double cn = d.cnear64 * inv2s2;
            const double uo = LAP ? su + fu : fma(su, cn, fu);
            const double vo = LAP ? 0.0 : fma(sv, cn, fv);
            if (dtype_f32) {
                static_cast<float *>(d.u)[q] = float(uo);
                static_cast<float *>(d.v)[q] = float(vo);
            } else {
                static_cast<double *>(d.u)[q] = uo;
                static_cast<double *>(d.v)[q] = vo;
            }
        }
        if (lane == 0) it = nwarps + atomicAdd(ctrl + CTRL_QUEUE, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
    }
    if (busy && lane == 0) {
        const uint64_t t_end = global_ns();
        const size_t gw = size_t(blockIdx.x) * (P2P_THREADS / 32) + (threadIdx.x >> 5);
        busy[2 * gw] = t_begin;
        busy[2 * gw + 1] = t_end;
    }
}

// ----------------------------------------------------------------------------
// Pairwise near field between neighbouring leaves (mixed path).
//
// Each unordered pair {A, B} of neighbouring occupied leaves is evaluated
// once, by the item (A, d) with B = A + off[d] one of A's four forward
// neighbours.  One warp holds up to 64 targets of A (two per lane) and 32
// sources of B (one per lane); in 32 steps the sources travel once around
// the warp (shuffles), and for every (target, source) pair the kernel factor
// K(x_a - x_s) is computed once and used twice: gamma_s K for the target and
// -gamma_a K for the source (K is odd, Eq. 8), the latter summed in a register
// that travels with the source.  The sums go to single-owner slots of the
// receiving particle: part[d][a] (from the forward neighbour d) and
// part[4 + d][b] (from the backward neighbour); the 64-target chunks of A
// add to a source's slot one after another in the same warp.  A final pass
// adds, per particle, its own leaf's sum and far field and the slots of its
// occupied neighbours in a fixed order: the result does not depend on which
// warp ran which item.
// ----------------------------------------------------------------------------

// Estimated time of nt targets against ns sources in the pair kernel: the
// target chunks it cuts (320/256/128/64/32, see pair_leaves) weighted by
// their measured time per source step (10 and 8 packed, 4 packed, 2 and 1
// targets per lane: 12.1, 10.3, 5.6, 3.4 and 2.5 relative units), times the
// source steps (32 per chunk of 32, 16 for a last chunk of at most 16).
__device__ __forceinline__ uint32_t pair_cost(uint32_t nt, uint32_t ns) {
    uint32_t c = 0;
    for (uint32_t r = nt; r > 0;) {
        if (r >= 257) { c += 121; r = r > 320 ? r - 320 : 0; }
        else if (r >= 192) { c += 103; r = r > 256 ? r - 256 : 0; }
        else if (r >= 96) { c += 56; r = r > 128 ? r - 128 : 0; }
        else if (r >= 33) { c += 34; r = r > 64 ? r - 64 : 0; }
        else { c += 25; r = r > 32 ? r - 32 : 0; }
    }
    const uint32_t tail = ns & 31u;
    return c * ((ns & ~31u) + (tail == 0 ? 0u : tail <= 16 ? 16u : 32u));
}

constexpr int PAIR_CLASSES = WORK_CLASSES;

// The work list takes two launches, both walking every leaf's items in the
// same way: the first counts the items of each work class (and the scratch
// entries and blob pairs), the second puts the items down class after class,
// heaviest first, their places within a class by atomics (the order of items
// changes no result).  ordered = 0 (PETFMM_OPT_P2P_MODE = 1): one class.
//
// Calls emit(class, item, scratch entries) for every item of leaf m.
template <typename F>
__device__ __forceinline__ void leaf_pair_items(const InstDesc &d, const uint32_t *st, uint32_t m,
                                                uint32_t inst, int ordered, F &&emit) {
    const uint32_t na = st[m + 1] - st[m];
    if (d.smdeg || na < d.pair_min) return;
    const int nside = 1 << d.L;
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    for (int k = 0; k < 4; ++k) {
        const uint32_t nb = leaf_count(st, nside, ix + c_fwd[k][0], iy + c_fwd[k][1]);
        if (!pairwise(na, nb, d.pair_min)) continue;
        uint32_t pc;
        const uint32_t np = pair_pieces(na, nb, &pc);
        // a pair in one piece runs with the leaf that pads less as targets
        const uint32_t swap = np == 1 && pair_cost(nb, na) < pair_cost(na, nb) ? 1u : 0u;
        for (uint32_t i = 0; i < np; ++i) {
            // a warp spends 32 steps per (64-target chunk, 32-source chunk)
            const uint32_t nt = min(pc, na - i * pc);
            const uint32_t cls =
                ordered ? work_class(((nt + 63) / 64) * ((nb + 31) / 32)) : 0u;
            emit(cls, make_uint4(inst, m, uint32_t(k) | (swap << 3) | (i << 4), 0u),
                 i ? 0u : (np - 1) * nb, (unsigned long long)(i ? 0u : na) * nb);
        }
    }
    // the leaf's own pairs (direction 4): half the tiles of the leaf with itself
    const uint32_t cls = ordered ? work_class(((na + 63) / 64) * ((na + 31) / 32) / 2) : 0u;
    emit(cls, make_uint4(inst, m, 4u, 0u), 0u, (unsigned long long)na * (na - 1) / 2);
}

__global__ void __launch_bounds__(256) k_pair_count(const Task *__restrict__ tasks, int ntasks,
                                                    const InstDesc *__restrict__ insts,
                                                    const uint32_t *__restrict__ start,
                                                    int ordered, uint32_t *ctrl,
                                                    uint32_t *__restrict__ ccount) {
    __shared__ uint32_t hist[PAIR_CLASSES];
    __shared__ unsigned long long sums;
    __shared__ uint32_t extra;
    for (int i = threadIdx.x; i < PAIR_CLASSES; i += 256) hist[i] = 0;
    if (threadIdx.x == 0) {
        sums = 0;
        extra = 0;
    }
    __syncthreads();
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    unsigned long long sym = 0;
    uint32_t x = 0;
    if (m < t.count) {
        const InstDesc &d = insts[t.inst];
        const uint32_t *st = start + d.soff;
        const uint32_t n = st[m + 1] - st[m];
        if (n && !d.smdeg)
            leaf_pair_items(d, st, uint32_t(m), uint32_t(t.inst), ordered,
                            [&](uint32_t cls, const uint4 &, uint32_t xtra, unsigned long long bp) {
                                atomicAdd(&hist[cls], 1u);
                                x += xtra;
                                sym += bp;
                            });
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        sym += __shfl_down_sync(0xffffffffu, sym, o);
        x += __shfl_down_sync(0xffffffffu, x, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (sym) atomicAdd(&sums, sym);
        if (x) atomicAdd(&extra, x);
    }
    __syncthreads();
    uint32_t items = 0;
    for (int i = threadIdx.x; i < PAIR_CLASSES; i += 256)
        if (hist[i]) {
            atomicAdd(ccount + i, hist[i]);
            items += hist[i];
        }
    if (items) atomicAdd(ctrl + CTRL_NPAIRS, items);
    if (threadIdx.x == 0) {
        if (sums) atomicAdd(reinterpret_cast<unsigned long long *>(ctrl + CTRL_SYM_LO), sums);
        if (extra) atomicAdd(ctrl + CTRL_NXTRA, extra);
    }
}

// ccount: the class counts; cplace: the items placed so far in each class
// (zeroed before), and one more word for the scratch entries handed out.
__global__ void __launch_bounds__(256) k_pair_emit(const Task *__restrict__ tasks, int ntasks,
                                                   const InstDesc *__restrict__ insts,
                                                   const uint32_t *__restrict__ start, int ordered,
                                                   const uint32_t *__restrict__ ctrl,
                                                   const uint32_t *__restrict__ ccount,
                                                   uint32_t *__restrict__ cplace, int64_t xcap,
                                                   int64_t cap, uint32_t *__restrict__ xtab,
                                                   uint32_t *__restrict__ lflags,
                                                   uint4 *__restrict__ items) {
    __shared__ uint32_t hist[PAIR_CLASSES], base[PAIR_CLASSES];
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t m = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    const InstDesc &d = insts[t.inst];
    const uint32_t *st = start + d.soff;
    for (int i = threadIdx.x; i < PAIR_CLASSES; i += 256) hist[i] = 0;
    const bool live = m < t.count && !d.smdeg;
    const uint32_t na = live ? st[m + 1] - st[m] : 0u;
    // the pieces' scratch runs exist only if all of them fit; else every pair
    // is one piece (decided alike for all pairs, so the result does not depend
    // on which fit)
    const bool split = int64_t(ctrl[CTRL_NXTRA]) <= xcap;
    if (live) {
        // this leaf's flags for the final pass
        const int nside = 1 << d.L;
        const int ix = int(compact_bits(uint32_t(m))), iy = int(compact_bits(uint32_t(m) >> 1));
        uint32_t fl = 0;
        if (na >= d.pair_min) {
            fl |= LF_SELF;
            for (int k = 0; k < 4; ++k) {
                if (pairwise(na, leaf_count(st, nside, ix + c_fwd[k][0], iy + c_fwd[k][1]),
                             d.pair_min))
                    fl |= LF_FWD << k;
                const uint32_t nbk = leaf_count(st, nside, ix - c_fwd[k][0], iy - c_fwd[k][1]);
                if (pairwise(nbk, na, d.pair_min)) {
                    fl |= LF_BWD << k;
                    uint32_t pc;
                    if (split && pair_pieces(nbk, na, &pc) > 1) fl |= LF_SPLIT << k;
                }
            }
        }
        lflags[d.loff + m] = fl;
    }
    if (!__syncthreads_or(na >= d.pair_min)) return;
    if (live)
        leaf_pair_items(d, st, uint32_t(m), uint32_t(t.inst), ordered,
                        [&](uint32_t cls, const uint4 &, uint32_t, unsigned long long) {
                            atomicAdd(&hist[cls], 1u);
                        });
    __syncthreads();
    // this block's run within each class
    if (threadIdx.x < PAIR_CLASSES) {
        uint32_t first = 0;
        for (int i = 0; i < int(threadIdx.x); ++i) first += ccount[i];
        const uint32_t n = hist[threadIdx.x];
        base[threadIdx.x] = first + (n ? atomicAdd(cplace + threadIdx.x, n) : 0u);
        hist[threadIdx.x] = 0;
    }
    __syncthreads();
    if (live)
        leaf_pair_items(
            d, st, uint32_t(m), uint32_t(t.inst), ordered,
            [&](uint32_t cls, uint4 item, uint32_t xtra, unsigned long long) {
                const uint32_t o = base[cls] + atomicAdd(&hist[cls], 1u);
                const int k = int(item.z & 7u);
                if (k < 4 && (item.z >> 4) == 0 && xtra)  // a pair in pieces: its scratch runs
                    xtab[(d.loff + m) * 4 + k] =
                        split ? atomicAdd(cplace + PAIR_CLASSES, xtra) : 0xffffffffu;
                // (the pieces of a pair follow one another in this thread)
                if (k < 4) {
                    uint32_t pc;
                    const uint32_t nb = leaf_count(st, 1 << d.L,
                                                   int(compact_bits(item.y)) + c_fwd[k][0],
                                                   int(compact_bits(item.y >> 1)) + c_fwd[k][1]);
                    item.w = pair_pieces(na, nb, &pc) > 1 ? xtab[(d.loff + m) * 4 + k]
                                                          : (split ? 0u : 0xffffffffu);
                }
                if (PF_IN(o, cap)) items[o] = item;
            });
}

// One target (in A's frame) against the travelling source (already in A's
// frame): the target gains gs K, the source -ga K.
template <int DEG, bool GENERAL>
__device__ __forceinline__ void pair_sym(float xa, float ya, float ga, float xs, float ys, float gs,
                                         const float (&a)[DEG + 1], float kappa, float split,
                                         float &ua, float &va, float &bu, float &bv) {
    const float dx = xa - xs, dy = ya - ys;
    const float r2 = fmaf(dx, dx, dy * dy);
    const float g = g_of<DEG, GENERAL>(a, r2, kappa, split);
    const float kx = -dy * g, ky = dx * g;
    ua = fmaf(gs, kx, ua);
    va = fmaf(gs, ky, va);
    bu = fmaf(-ga, kx, bu);
    bv = fmaf(-ga, ky, bv);
}

// placeholders of missing targets / sources: far apart (finite kernel
// values), zero strength (they add nothing and their sums are dropped)
constexpr float kPairFar = 64.f;

// p[0] = w, or p[0] += w
__device__ __forceinline__ void put2(float2 *p, float2 w, bool add) {
    if (add) {
        const float2 o = *p;
        w = make_float2(o.x + w.x, o.y + w.y);
    }
    *p = w;
}

// One pass of a source chunk around the warp: W = 32 sources, one per lane,
// or W = 16 (a tail of at most 16 sources held by both half-warps, each half
// rotating its own copy).  Each step every lane evaluates its TPL targets
// against the source it holds, the source's reaction sum travelling with it;
// after W steps every sum is back at its source's lane (for W = 16 the two
// halves' sums are then added).
template <int DEG, bool GENERAL, int TPL, int W>
__device__ __forceinline__ void source_pass(const float (&tx)[TPL], const float (&ty)[TPL],
                                            const float (&tg)[TPL], float (&u)[TPL],
                                            float (&v)[TPL], const float (&a)[DEG + 1],
                                            float kappa, float split, float xs, float ys,
                                            float gs, float &bu, float &bv, int lane) {
    const int next = (lane & ~(W - 1)) | ((lane + 1) & (W - 1));
    bu = 0.f;
    bv = 0.f;
#pragma unroll 2
    for (int k = 0; k < W; ++k) {
#pragma unroll
        for (int t = 0; t < TPL; ++t)
            pair_sym<DEG, GENERAL>(tx[t], ty[t], tg[t], xs, ys, gs, a, kappa, split, u[t], v[t], bu,
                                   bv);
        xs = __shfl_sync(0xffffffffu, xs, next);
        ys = __shfl_sync(0xffffffffu, ys, next);
        gs = __shfl_sync(0xffffffffu, gs, next);
        bu = __shfl_sync(0xffffffffu, bu, next);
        bv = __shfl_sync(0xffffffffu, bv, next);
    }
    if (W < 32) {
        bu += __shfl_xor_sync(0xffffffffu, bu, 16);
        bv += __shfl_xor_sync(0xffffffffu, bv, 16);
    }
}

// The same pass with 2 H targets per lane held as H pairs and evaluated with
// packed FP32x2 instructions (polynomial near-field factor only): the same
// products per pair as source_pass, each packed instruction doing two of
// them, so half the issue slots.  The reaction sums of a step run in the two
// halves of a pair and are added before the source moves on.  Signs are
// folded out of the loop: the source travels as (-x, -y), the targets keep
// U = -u and the reaction BV = -bv (round-to-nearest is symmetric in sign,
// so the sums are bit for bit the negated ones), which saves the negated
// copies of the strengths and one broadcast per step.
template <int DEG, int H, int W>
__device__ __forceinline__ void source_pass_x2(const float2 (&tx)[H], const float2 (&ty)[H],
                                               const float2 (&tg)[H], float2 (&U)[H],
                                               float2 (&v)[H], const float2 (&a2)[DEG + 1],
                                               float nxs, float nys, float gs, float &bu,
                                               float &BV, int lane) {
    const int next = (lane & ~(W - 1)) | ((lane + 1) & (W - 1));
    bu = 0.f;
    BV = 0.f;
#pragma unroll 2
    for (int k = 0; k < W; ++k) {
        // with K = (-dy, dx) g: u_a += g_s K, reaction u_b -= g_a K
        const float2 nx = make_float2(nxs, nxs), ny = make_float2(nys, nys);
        const float2 g2 = make_float2(gs, gs);
        float2 bu2 = make_float2(bu, 0.f), bv2 = make_float2(BV, 0.f);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const float2 dx = __fadd2_rn(tx[h], nx), dy = __fadd2_rn(ty[h], ny);
            const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
            float2 g = a2[DEG];
#pragma unroll
            for (int q = DEG - 1; q >= 0; --q) g = __ffma2_rn(g, r2, a2[q]);
            const float2 py = __fmul2_rn(dy, g), px = __fmul2_rn(dx, g);
            U[h] = __ffma2_rn(g2, py, U[h]);
            v[h] = __ffma2_rn(g2, px, v[h]);
            bu2 = __ffma2_rn(tg[h], py, bu2);
            bv2 = __ffma2_rn(tg[h], px, bv2);
        }
        bu = bu2.x + bu2.y;
        BV = bv2.x + bv2.y;
        nxs = __shfl_sync(0xffffffffu, nxs, next);
        nys = __shfl_sync(0xffffffffu, nys, next);
        gs = __shfl_sync(0xffffffffu, gs, next);
        bu = __shfl_sync(0xffffffffu, bu, next);
        BV = __shfl_sync(0xffffffffu, BV, next);
    }
    if (W < 32) {
        bu += __shfl_xor_sync(0xffffffffu, bu, 16);
        BV += __shfl_xor_sync(0xffffffffu, BV, 16);
    }
}

// Source chunk bc of B as seen by this lane: the source it starts with (in
// A's frame; placeholders past the end) and whether the chunk is a tail of
// at most 16 (half-warp pass).
struct SourceSlot {
    float xs, ys, gs;
    uint32_t sb;
    bool hs, half;
};
__device__ __forceinline__ SourceSlot source_slot(const float4 *__restrict__ rec, uint32_t b0,
                                                  uint32_t bc, uint32_t nb, int ox, int oy,
                                                  int lane) {
    // the next chunk's records into L1 while this one is evaluated
    if (bc + 32 + uint32_t(lane) < nb)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + b0 + bc + 32 + lane));
    SourceSlot o;
    o.half = nb - bc <= 16;
    o.sb = bc + uint32_t(o.half ? (lane & 15) : lane);
    o.hs = o.sb < nb;
    const float4 s = o.hs ? rec[b0 + o.sb] : make_float4(-kPairFar, -kPairFar, 0.f, 0.f);
    // B's centre is A's plus (ox, oy) leaves
    o.xs = s.x + float(ox);
    o.ys = s.y + float(oy);
    o.gs = s.z;
    return o;
}

// One chunk of a leaf pair: targets ac .. min(ac + 32 TPL, aend) - 1 of leaf A
// (TPL per lane: lane + 32 t) against all nb sources of leaf B, B in chunks
// of 32 sources travelling around the warp with their reaction sums (a last
// chunk of at most 16 in a half-warp pass).  fwd[i]: A's blob i from B;
// bwd[j]: B's blob j from A (bwd_add / fwd_add: the chunk adds to them, else
// writes).
template <int DEG, bool GENERAL, int TPL>
__device__ __noinline__ void pair_chunk(const float4 *__restrict__ rec, uint32_t a0,
                                        uint32_t ac, uint32_t aend, uint32_t b0, uint32_t nb,
                                        int ox, int oy, const float (&a)[DEG + 1], float kappa,
                                        float split, float cn, float2 *fwd, float2 *bwd,
                                        bool bwd_add, bool fwd_add, int lane) {
    float tx[TPL], ty[TPL], tg[TPL], u[TPL], v[TPL];
#pragma unroll
    for (int t = 0; t < TPL; ++t) {
        const bool h = ac + lane + 32 * t < aend;
        const float4 r =
            h ? rec[a0 + ac + lane + 32 * t] : make_float4(kPairFar, kPairFar, 0.f, 0.f);
        tx[t] = r.x;
        ty[t] = r.y;
        tg[t] = r.z;
        u[t] = v[t] = 0.f;
    }
    for (uint32_t bc = 0; bc < nb; bc += 32) {
        const SourceSlot ss = source_slot(rec, b0, bc, nb, ox, oy, lane);
        float bu, bv;
        if (ss.half)
            source_pass<DEG, GENERAL, TPL, 16>(tx, ty, tg, u, v, a, kappa, split, ss.xs, ss.ys,
                                               ss.gs, bu, bv, lane);
        else
            source_pass<DEG, GENERAL, TPL, 32>(tx, ty, tg, u, v, a, kappa, split, ss.xs, ss.ys,
                                               ss.gs, bu, bv, lane);
        if (ss.hs && (!ss.half || lane < 16))
            put2(bwd + ss.sb, make_float2(cn * bu, cn * bv), bwd_add);
    }
#pragma unroll
    for (int t = 0; t < TPL; ++t)
        if (ac + lane + 32 * t < aend)
            put2(fwd + ac + lane + 32 * t, make_float2(cn * u[t], cn * v[t]), fwd_add);
}

// The same chunk with 2 H targets per lane held as H pairs (targets lane +
// 64 h and lane + 64 h + 32), evaluated by source_pass_x2 (which keeps -u
// and the reaction's -v; the signs are restored on the way out).
template <int DEG, int H>
__device__ __noinline__ void pair_chunk_x2(const float4 *__restrict__ rec, uint32_t a0,
                                           uint32_t ac, uint32_t aend, uint32_t b0, uint32_t nb,
                                           int ox, int oy, const float (&a)[DEG + 1], float cn,
                                           float2 *fwd, float2 *bwd, bool bwd_add, bool fwd_add,
                                           int lane) {
    float2 tx[H], ty[H], tg[H], U[H], v[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const uint32_t i0 = ac + lane + 64 * h, i1 = i0 + 32;
        const float4 r0 = i0 < aend ? rec[a0 + i0] : make_float4(kPairFar, kPairFar, 0.f, 0.f);
        const float4 r1 = i1 < aend ? rec[a0 + i1] : make_float4(kPairFar, kPairFar, 0.f, 0.f);
        tx[h] = make_float2(r0.x, r1.x);
        ty[h] = make_float2(r0.y, r1.y);
        tg[h] = make_float2(r0.z, r1.z);
        U[h] = v[h] = make_float2(0.f, 0.f);
    }
    float2 a2[DEG + 1];
#pragma unroll
    for (int k = 0; k <= DEG; ++k) a2[k] = make_float2(a[k], a[k]);
    for (uint32_t bc = 0; bc < nb; bc += 32) {
        const SourceSlot ss = source_slot(rec, b0, bc, nb, ox, oy, lane);
        float bu, BV;
        if (ss.half)
            source_pass_x2<DEG, H, 16>(tx, ty, tg, U, v, a2, -ss.xs, -ss.ys, ss.gs, bu, BV, lane);
        else
            source_pass_x2<DEG, H, 32>(tx, ty, tg, U, v, a2, -ss.xs, -ss.ys, ss.gs, bu, BV, lane);
        if (ss.hs && (!ss.half || lane < 16))
            put2(bwd + ss.sb, make_float2(cn * bu, -(cn * BV)), bwd_add);
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const uint32_t i0 = ac + lane + 64 * h, i1 = i0 + 32;
        if (i0 < aend) put2(fwd + i0, make_float2(-(cn * U[h].x), cn * v[h].x), fwd_add);
        if (i1 < aend) put2(fwd + i1, make_float2(-(cn * U[h].y), cn * v[h].y), fwd_add);
    }
}

// The pairs of blobs abeg .. aend - 1 of leaf A (from a0) with the nb blobs
// of leaf B (from b0): A in chunks of 320, 256, 128, 64 or 32 targets.  Leaf
// pairs take the largest chunk that the remaining targets fill to at least
// three quarters (for 320: more than 256, where one 320-chunk is faster
// than 256 + a tail chunk); more targets per lane amortise the shuffles of
// a step over more pairs (measured in isolation on GB300: 10 targets per
// lane 0.776 of the FP32 peak, 8 per lane 0.727).  A range of whole 32-blob
// chunks (exact) is cut without padding.  The first chunk writes bwd (unless bwd_add), later ones
// add to it; fwd_add: the chunks add to fwd.
template <int DEG, bool GENERAL>
__device__ __forceinline__ void pair_leaves(const float4 *__restrict__ rec, uint32_t a0,
                                            uint32_t abeg, uint32_t aend, uint32_t b0, uint32_t nb,
                                            int ox, int oy, const float (&a)[DEG + 1],
                                            float kappa, float split, float cn, float2 *fwd,
                                            float2 *bwd, bool bwd_add, bool fwd_add, bool exact,
                                            int lane) {
    const uint32_t t10 = exact ? 320 : 257, t8 = exact ? 256 : 192, t4 = exact ? 128 : 96,
                   t2 = exact ? 64 : 33;
    for (uint32_t ac = abeg; ac < aend; bwd_add = true) {
        const uint32_t rem = aend - ac;
        if (!GENERAL && rem >= t10) {
            pair_chunk_x2<DEG, 5>(rec, a0, ac, aend, b0, nb, ox, oy, a, cn, fwd, bwd, bwd_add,
                                  fwd_add, lane);
            ac += 320;
        } else if (!GENERAL && rem >= t8) {
            pair_chunk_x2<DEG, 4>(rec, a0, ac, aend, b0, nb, ox, oy, a, cn, fwd, bwd, bwd_add,
                                  fwd_add, lane);
            ac += 256;
        } else if (rem >= t4) {
            if (GENERAL)
                pair_chunk<DEG, GENERAL, 4>(rec, a0, ac, aend, b0, nb, ox, oy, a, kappa, split, cn,
                                            fwd, bwd, bwd_add, fwd_add, lane);
            else
                pair_chunk_x2<DEG, 2>(rec, a0, ac, aend, b0, nb, ox, oy, a, cn, fwd, bwd, bwd_add,
                                      fwd_add, lane);
            ac += 128;
        } else if (rem >= t2) {
            pair_chunk<DEG, GENERAL, 2>(rec, a0, ac, aend, b0, nb, ox, oy, a, kappa, split, cn,
                                        fwd, bwd, bwd_add, fwd_add, lane);
            ac += 64;
        } else {
            pair_chunk<DEG, GENERAL, 1>(rec, a0, ac, aend, b0, nb, ox, oy, a, kappa, split, cn,
                                        fwd, bwd, bwd_add, fwd_add, lane);
            ac += 32;
        }
    }
}

// The pairs within one leaf (n >= 32 blobs from a0), each once, summed into
// slf[0 .. n) by one warp in a fixed order.  For each 32-blob sub-chunk j:
// the pairs inside it -- the blobs rotate around the warp for 16 steps, so
// that every lane meets every other lane's blob once (at step 16 the two
// halves of the warp meet each other, so only lanes 0..15 count it), and a
// final shuffle brings each travelling reaction back to its blob -- then its
// pairs with all blobs before it, as a pair range (targets 0 .. 32 j,
// sources the sub-chunk).
template <int DEG, bool GENERAL>
__device__ __forceinline__ void self_leaf(const float4 *__restrict__ rec, uint32_t a0,
                                          uint32_t n, const float (&a)[DEG + 1], float kappa,
                                          float split, float cn, float2 *slf, int lane) {
    const int next = (lane + 1) & 31;
    for (uint32_t s0 = 0; s0 < n; s0 += 32) {
        const uint32_t ns = min(32u, n - s0);
        const bool h = uint32_t(lane) < ns;
        const float4 r = h ? rec[a0 + s0 + lane] : make_float4(kPairFar, kPairFar, 0.f, 0.f);
        float xs = r.x, ys = r.y, gs = r.z, bu = 0.f, bv = 0.f, u = 0.f, v = 0.f;
        for (int k = 1; k <= 16; ++k) {
            xs = __shfl_sync(0xffffffffu, xs, next);
            ys = __shfl_sync(0xffffffffu, ys, next);
            gs = __shfl_sync(0xffffffffu, gs, next);
            bu = __shfl_sync(0xffffffffu, bu, next);
            bv = __shfl_sync(0xffffffffu, bv, next);
            const bool on = k < 16 || lane < 16;
            pair_sym<DEG, GENERAL>(r.x, r.y, on ? r.z : 0.f, xs, ys, on ? gs : 0.f, a, kappa,
                                   split, u, v, bu, bv);
        }
        // lane l holds the reaction of the blob of lane l + 16
        bu = __shfl_sync(0xffffffffu, bu, (lane + 16) & 31);
        bv = __shfl_sync(0xffffffffu, bv, (lane + 16) & 31);
        if (h) slf[s0 + lane] = make_float2(cn * (u + bu), cn * (v + bv));
        __syncwarp();
        if (s0)
            pair_leaves<DEG, GENERAL>(rec, a0, 0, s0, a0 + s0, ns, 0, 0, a, kappa, split, cn, slf,
                                      slf + s0, true, true, true, lane);
        __syncwarp();
    }
}

// One item of the pairwise near field: piece item.z >> 4 of leaf A (item.y)
// with its forward neighbour B, direction item.z & 7 (4: the leaf's own
// pairs, to slot 8); bit 3: B's blobs are the targets (a pair in one piece);
// item.w = the pair's scratch base (all ones: the pair is not split, piece 0
// takes all of it).
template <int DEG, bool GENERAL>
__device__ __forceinline__ void pair_item(const uint4 item, const InstDesc *__restrict__ insts,
                                          const uint32_t *__restrict__ start,
                                          const float4 *__restrict__ rec,
                                          float2 *__restrict__ part, int64_t nslot,
                                          float2 *__restrict__ xs, int64_t xcap, int lane) {
    const InstDesc &d = insts[item.x];
    float a[DEG + 1];
#pragma unroll
    for (int k = 0; k <= DEG; ++k) a[k] = d.poly[k];
    const float kappa = d.kappa, split = d.qsplit_rho2, cn = d.cnear;
    const uint32_t m = item.y;
    const int dir = int(item.z & 7u);
    const bool swap = (item.z >> 3) & 1u;
    const uint32_t piece = item.z >> 4;
    const uint32_t *st = start + d.soff;
    const uint32_t a0 = st[m], na = st[m + 1] - a0;
    // checked build: the leaf and its range lie inside the instance
    if (!(PF_IN(m, int64_t(1) << (2 * d.L)) && PF_IN(int64_t(a0) - d.poff, d.n + 1) &&
          PF_IN(int64_t(a0) + na - d.poff, d.n + 1) && PF_IN(int64_t(a0) + na, nslot + 1)))
        return;
    if (dir == 4) {
        self_leaf<DEG, GENERAL>(rec, a0, na, a, kappa, split, cn, part + 8 * nslot + a0, lane);
        return;
    }
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    const int ox = c_fwd[dir][0], oy = c_fwd[dir][1];
    const uint32_t mb = morton_key(uint32_t(ix + ox), uint32_t(iy + oy));
    const uint32_t b0 = st[mb], nb = st[mb + 1] - b0;
    if (!(PF_IN(mb, int64_t(1) << (2 * d.L)) && PF_IN(int64_t(b0) - d.poff, d.n + 1) &&
          PF_IN(int64_t(b0) + nb - d.poff, d.n + 1)))
        return;
    float2 *fwd = part + int64_t(dir) * nslot + a0;      // A's particles, from B
    float2 *bwd = part + int64_t(4 + dir) * nslot + b0;  // B's particles, from A
    if (swap) {
        pair_leaves<DEG, GENERAL>(rec, b0, 0, nb, a0, na, -ox, -oy, a, kappa, split, cn, bwd, fwd,
                                  false, false, false, lane);
        return;
    }
    uint32_t abeg = 0, aend = na;
    if (item.w != 0xffffffffu) {
        uint32_t pc;
        pair_pieces(na, nb, &pc);
        abeg = piece * pc;
        aend = min(na, abeg + pc);
        if (piece) {
            if (!PF_IN(int64_t(item.w) + int64_t(piece) * nb - 1, xcap)) return;
            bwd = xs + item.w + int64_t(piece - 1) * nb;
        }
    } else if (piece) {
        return;
    }
    pair_leaves<DEG, GENERAL>(rec, a0, abeg, aend, b0, nb, ox, oy, a, kappa, split, cn, fwd, bwd,
                              false, false, false, lane);
}

// The pair items of the pairwise mode, heaviest first, in one persistent
// launch (64 registers for the four targets per lane: 4 CTAs per SM); the
// leaves' not-pairwise neighbours follow in
// k_p2p_mixed<.., PAIRS = true> at its higher occupancy.  Measured on GB300,
// one queue over both kinds of item (the directed ones filling the pairs'
// tail) was slower: the directed items ran at this kernel's occupancy.
template <int DEG, bool GENERAL>
__global__ void __launch_bounds__(P2P_THREADS, 3) k_p2p_pairs(
    const uint4 *__restrict__ pitems, uint32_t *ctrl, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const float4 *__restrict__ rec, const PairBufs pb,
    unsigned long long *busy) {
    const int lane = threadIdx.x & 31;
    const uint32_t npairs = *reinterpret_cast<volatile uint32_t *>(ctrl + CTRL_NPAIRS);
    const uint64_t t_begin = busy ? global_ns() : 0;
    for (;;) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(ctrl + CTRL_QUEUE2, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= npairs) break;
        pair_item<DEG, GENERAL>(pitems[it], insts, start, rec, pb.part, pb.nslot, pb.xs, pb.xcap,
                                lane);
    }
    if (busy && lane == 0) {
        const size_t gw = size_t(blockIdx.x) * (P2P_THREADS / 32) + (threadIdx.x >> 5);
        busy[2 * gw] = t_begin;
        busy[2 * gw + 1] = global_ns();
    }
}

// The final pass of the mixed near field, one thread per blob: u, v = its
// leaf's far field (L2P of the local expansion, Sec. 2.2), plus its directly
// summed near part, plus (pairwise mode, pb.part != nullptr) the slots of its
// pairwise neighbours, a split pair's scratch runs after its slot in piece
// order; a fixed order throughout, written at the caller's index.
// blobs per occupied leaf from which the final pass requests every pair
// slot of a blob up front (see k_p2p_final)
constexpr int64_t kEagerBlobsPerLeaf = 48;

__global__ void __launch_bounds__(256, 4) k_p2p_final(
    const Task *__restrict__ tasks, int ntasks, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const uint32_t *__restrict__ skeys,
    const float4 *__restrict__ rec, const float2 *__restrict__ le, const PairBufs pb,
    int dtype_f32, float *__restrict__ stage, int64_t nstage, const uint32_t *__restrict__ ctrl,
    int64_t ntotal) {
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t j = (int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x;
    if (j >= t.count) return;
    const InstDesc &d = insts[t.inst];
    if (d.smdeg) return;  // k_sm_final's
    const int64_t r = d.poff + j;
    const uint32_t *st = start + d.soff;
    const int nside = 1 << d.L;
    // Where the occupied leaves hold many blobs on average (pair slots
    // nearly everywhere), this blob's near-field parts are requested at once,
    // with its key and record, instead of after its leaf's flags: one latency
    // instead of three on the way to the sum.  The flags still decide which
    // of them are added, in the same order.
    const bool eager = pb.part && int64_t(ntotal) >= kEagerBlobsPerLeaf * int64_t(ctrl[CTRL_NOCC]);
    float2 e_own = make_float2(0.f, 0.f), e_self = e_own, e_fwd[4], e_bwd[4];
    if (eager) {
        e_own = pb.own[r];
        e_self = pb.part[8 * pb.nslot + r];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            e_fwd[k] = pb.part[int64_t(k) * pb.nslot + r];
            e_bwd[k] = pb.part[int64_t(4 + k) * pb.nslot + r];
        }
    }
    const uint32_t m = skeys[r] & ((d.L >= 16) ? 0xffffffffu : ((1u << (2 * d.L)) - 1u));
    const int ix = int(compact_bits(m)), iy = int(compact_bits(m >> 1));
    const float4 rr = rec[r];
    float2 w = make_float2(0.f, 0.f);
    if (d.L >= 2) {
        // w = (1/r) sum c_m zeta^m, zeta the offset from the leaf centre
        const int p = d.p;
        const float2 *c =
            le + d.eoff + (lvl_off(d.L) + box_index(d.L, uint32_t(ix), uint32_t(iy))) * p;
        const float2 z = far_series(c, p, rr.x, rr.y);
        // vortex: u - i v = cfar w; Laplace: the potential is Re of the LE
        w = d.kernel == KERNEL_LAPLACE ? make_float2(z.x, 0.f)
                                       : make_float2(d.cfar * z.y, d.cfar * z.x);
    }
    // then the directly summed part and the slots this leaf has, in a fixed
    // order
    const uint32_t fl = pb.part ? pb.lflags[d.loff + m] : 0u;
    const float2 o = eager ? e_own : pb.own[r];
    w.x += o.x;
    w.y += o.y;
    if (fl & LF_SELF) {
        const float2 sp = eager ? e_self : pb.part[8 * pb.nslot + r];
        w.x += sp.x;
        w.y += sp.y;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (fl & (LF_FWD << k)) {
            const float2 p = eager ? e_fwd[k] : pb.part[int64_t(k) * pb.nslot + r];
            w.x += p.x;
            w.y += p.y;
        }
        if (!(fl & (LF_BWD << k))) continue;
        const float2 p = eager ? e_bwd[k] : pb.part[int64_t(4 + k) * pb.nslot + r];
        w.x += p.x;
        w.y += p.y;
        if (fl & (LF_SPLIT << k)) {
            // pieces 1 .. of the pair (A = the backward neighbour, B = this leaf)
            const int ax = ix - c_fwd[k][0], ay = iy - c_fwd[k][1];
            const uint32_t na = leaf_count(st, nside, ax, ay), nme = st[m + 1] - st[m];
            const uint32_t jme = uint32_t(r) - st[m];
            uint32_t pc;
            const uint32_t np = pair_pieces(na, nme, &pc);
            const uint32_t ma = morton_key(uint32_t(ax), uint32_t(ay));
            const uint32_t base = pb.xtab[(d.loff + int64_t(ma)) * 4 + k];
            for (uint32_t i = 1; i < np; ++i) {
                const float2 x = pb.xs[base + int64_t(i - 1) * nme + jme];
                w.x += x.x;
                w.y += x.y;
            }
        }
    }
    if (stage) {
        // sorted order; k_unsort writes the caller's arrays
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

cudaError_t launch_pair_worklist(const Task *tasks, int ntasks, int64_t nblocks,
                                 const InstDesc *insts, const uint32_t *start, int ordered,
                                 uint4 *items, int64_t cap, uint32_t *ctrl, const PairBufs &pb,
                                 cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    uint32_t *ccount = ctrl + CTRL_CLASSES, *cplace = ccount + PAIR_CLASSES;
    static_assert(CTRL_CLASSES + 2 * PAIR_CLASSES + 1 <= CTRL_WORDS, "class counters");
    k_pair_count<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, ordered, ctrl,
                                                    ccount);
    PF_LAUNCHED(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_pair_emit<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, ordered, ctrl,
                                                   ccount, cplace, pb.xcap, cap, pb.xtab,
                                                   pb.lflags, items);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// The near field outside the pair kernel, one thread per target blob: own[r]
// = its sum over the leaves of its neighbourhood that are not summed pairwise
// with its own (Laplace kernel, and vortex cores narrow against a leaf: all
// nine).  Bound by issue (74 % of the slots; 26 instructions a pair and lane with
// the idle lanes of uneven leaves, two of them special functions): every lane has
// a target of its own, so leaves of any count fill the warps, where a warp per
// leaf of 17 blobs kept 17 of 32 lanes busy; the lanes of a leaf read the
// same source (one request), and no work list is needed.
// Measured on one GB300 (this kernel alone, against work items and the pair
// kernel with their lists): 512 uneven trees, 3.9e9 pairs: 9.0 -> 3.6 ms;
// 1,048,576 blobs, 16 per leaf: 0.29 -> 0.13 ms; 349,185 clustered blobs, 530
// per leaf, kappa = 7.6: 3.3 -> 1.3 ms.
constexpr int NEAR_THREADS = 128;  // half a particle task block: more blocks, better balance

__global__ void __launch_bounds__(NEAR_THREADS, 8) k_near_direct(
    const Task *__restrict__ tasks, int ntasks, const InstDesc *__restrict__ insts,
    const uint32_t *__restrict__ start, const uint32_t *__restrict__ skeys,
    const float4 *__restrict__ rec, float2 *__restrict__ own, uint32_t *ctrl,
    unsigned long long *busy, uint32_t nbusy) {
    __shared__ unsigned long long spairs;
    // busy: first start and last end of this kernel's blocks on each SM, by
    // %smid; the identifiers need not be contiguous, and those from nbusy on
    // have no entry
    uint32_t sm = 0;
    if (threadIdx.x == 0) {
        spairs = 0;
        if (busy) {
            asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
            if (sm < nbusy) atomicMin(busy + 2 * sm, (unsigned long long)global_ns());
        }
    }
    __syncthreads();
    const int64_t blk = blockIdx.x / (256 / NEAR_THREADS);
    const int ti = find_task(tasks, ntasks, blk);
    const Task t = tasks[ti];
    const int64_t j = (blk - t.block0) * 256 + (blockIdx.x % (256 / NEAR_THREADS)) * NEAR_THREADS +
                      threadIdx.x;
    const InstDesc &d = insts[t.inst];
    unsigned long long pairs = 0;
    if (j < t.count && d.direct) {
        const int64_t r = d.poff + j;
        const uint32_t *st = start + d.soff;
        const uint32_t m = skeys[r] & ((1u << (2 * d.L)) - 1u);
        const NearLeaves q{&d, st, int(compact_bits(m)), int(compact_bits(m >> 1)), 0x1ffu,
                           st[m + 1] - st[m], d.pair_min};
        const float4 rr = rec[r];
        uint32_t total;
        float2 w;
        if (d.kernel == KERNEL_LAPLACE) {
            const float logw = float(d.logw0 - double(d.L) * 0.69314718055994530942);
            w = make_float2(near_laplace(q, rec, rr.x, rr.y, logw, total), 0.f);
        } else {
            w = near_vortex_of(q, rec, rr.x, rr.y, total);
            w.x *= d.cfar;  // cnear / kappa = cfar
            w.y *= d.cfar;
        }
        pairs = total - 1u;  // not with itself
        own[r] = w;
    }
    // ordered near pairs, for the statistics
#pragma unroll
    for (int o = 16; o; o >>= 1) pairs += __shfl_down_sync(0xffffffffu, pairs, o);
    if ((threadIdx.x & 31) == 0 && pairs) atomicAdd(&spairs, pairs);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (spairs)
            atomicAdd(reinterpret_cast<unsigned long long *>(ctrl + CTRL_PAIRS_LO), spairs);
        if (busy && sm < nbusy) atomicMax(busy + 2 * sm + 1, (unsigned long long)global_ns());
    }
}

cudaError_t launch_near_direct(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                               const uint32_t *start, const uint32_t *skeys, const float4 *rec,
                               float2 *own, uint32_t *ctrl, unsigned long long *busy, int nbusy,
                               cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_near_direct<<<unsigned(nblocks * (256 / NEAR_THREADS)), NEAR_THREADS, 0, st>>>(
        tasks, ntasks, insts, start, skeys, rec, own, ctrl, busy, uint32_t(nbusy));
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Launch helpers
// ----------------------------------------------------------------------------
typedef void (*MixedKernel)(const uint4 *, uint32_t *, const InstDesc *, const uint32_t *,
                            const float4 *, float2 *, unsigned long long *);
template <int D>
static MixedKernel pick2(int general) {
    return general ? k_p2p_mixed<D, true, false> : k_p2p_mixed<D, false, false>;
}

static MixedKernel pick_mixed(int deg, int general, bool lap = false) {
    if (lap) return k_p2p_mixed<4, false, true>;  // no polynomial
    switch (deg) {
        case 4: return pick2<4>(general);
        case 5: return pick2<5>(general);
        case 6: return pick2<6>(general);
        case 7: return pick2<7>(general);
        case 8: return pick2<8>(general);
        case 9: return pick2<9>(general);
        case 10: return pick2<10>(general);
        case 11: return pick2<11>(general);
        case 12: return pick2<12>(general);
        default: return nullptr;
    }
}

static int g_sms = 0;

int device_sm_count() {
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

int p2p_grid(int precision_mixed, int deg, int general, int laplace) {
    int per_sm = 1;
    if (precision_mixed) {
        MixedKernel k = pick_mixed(deg, general, laplace != 0);
        if (!k) return 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, P2P_THREADS, 0);
    } else {
        if (laplace)
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p_f64<true>, P2P_THREADS, 0);
        else
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p_f64<false>, P2P_THREADS, 0);
    }
    if (per_sm < 1) per_sm = 1;
    return per_sm * device_sm_count();
}

cudaError_t launch_p2p_mixed(int grid, int deg, int general, const uint4 *items, uint32_t *ctrl,
                             const InstDesc *insts, const uint32_t *start, const float4 *rec,
                             float2 *own, int laplace, unsigned long long *busy, cudaStream_t st,
                             uint64_t *launches) {
    MixedKernel k = pick_mixed(deg, general, laplace != 0);
    if (!k) return cudaErrorInvalidValue;
    k<<<grid, P2P_THREADS, 0, st>>>(items, ctrl, insts, start, rec, own, busy);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

typedef void (*PairsKernel)(const uint4 *, uint32_t *, const InstDesc *, const uint32_t *,
                            const float4 *, const PairBufs, unsigned long long *);

template <int D>
static PairsKernel pick_pairs2(int general) {
    return general ? k_p2p_pairs<D, true> : k_p2p_pairs<D, false>;
}

static PairsKernel pick_pairs(int deg, int general) {
    switch (deg) {
        case 4: return pick_pairs2<4>(general);
        case 5: return pick_pairs2<5>(general);
        case 6: return pick_pairs2<6>(general);
        case 7: return pick_pairs2<7>(general);
        case 8: return pick_pairs2<8>(general);
        case 9: return pick_pairs2<9>(general);
        case 10: return pick_pairs2<10>(general);
        case 11: return pick_pairs2<11>(general);
        case 12: return pick_pairs2<12>(general);
        default: return nullptr;
    }
}

int p2p_pairs_grid(int deg, int general) {
    PairsKernel k = pick_pairs(deg, general);
    if (!k) return 0;
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, P2P_THREADS, 0);
    if (per_sm < 1) per_sm = 1;
    return per_sm * device_sm_count();
}

cudaError_t launch_p2p_pairs(int grid, int deg, int general, const uint4 *pitems, uint32_t *ctrl,
                             const InstDesc *insts, const uint32_t *start, const float4 *rec,
                             const PairBufs &pb, unsigned long long *busy, cudaStream_t st,
                             uint64_t *launches) {
    PairsKernel k = pick_pairs(deg, general);
    if (!k) return cudaErrorInvalidValue;
    k<<<grid, P2P_THREADS, 0, st>>>(pitems, ctrl, insts, start, rec, pb, busy);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

// The caller's u (comp 0) or v (comp 1) from the sorted-order stage, FP32
// outputs.  One component per launch: its scattered 4-byte writes then fit in
// L2 and leave it as whole sectors, where writing u and v together from the
// final pass evicts partly written sectors (each one read back and written
// again).
__global__ void __launch_bounds__(256) k_unsort_f32(const Task *__restrict__ tasks, int ntasks,
                                                    const InstDesc *__restrict__ insts,
                                                    const uint32_t *__restrict__ perm,
                                                    const float *__restrict__ stage, int comp) {
    // four consecutive sorted ranks per thread (tasks of 1024 per block):
    // four independent scattered stores after two 16-byte loads
    const int ti = find_task(tasks, ntasks, blockIdx.x);
    const Task t = tasks[ti];
    const int64_t j0 = ((int64_t(blockIdx.x) - t.block0) * blockDim.x + threadIdx.x) * 4;
    if (j0 >= t.count) return;
    const InstDesc &d = insts[t.inst];
    const int64_t r0 = d.poff + j0;
    float *out = static_cast<float *>(comp ? d.v : d.u);
    if (j0 + 4 <= t.count && (r0 & 3) == 0) {
        const uint4 q = *reinterpret_cast<const uint4 *>(perm + r0);
        const float4 w = *reinterpret_cast<const float4 *>(stage + r0);
        if (PF_IN(int64_t(q.x) - d.poff, d.n)) out[int64_t(q.x) - d.poff] = w.x;
        if (PF_IN(int64_t(q.y) - d.poff, d.n)) out[int64_t(q.y) - d.poff] = w.y;
        if (PF_IN(int64_t(q.z) - d.poff, d.n)) out[int64_t(q.z) - d.poff] = w.z;
        if (PF_IN(int64_t(q.w) - d.poff, d.n)) out[int64_t(q.w) - d.poff] = w.w;
    } else {
        for (int e = 0; e < 4; ++e)
            if (j0 + e < t.count && PF_IN(int64_t(perm[r0 + e]) - d.poff, d.n))
                out[int64_t(perm[r0 + e]) - d.poff] = stage[r0 + e];
    }
}

cudaError_t launch_p2p_final(const Task *tasks, int ntasks, int64_t nblocks,
                             const InstDesc *insts, const uint32_t *start, const uint32_t *skeys,
                             const float4 *rec, const float2 *le, const PairBufs &pb,
                             int dtype_f32, float *stage, int64_t nstage, const uint32_t *ctrl,
                             int64_t ntotal, cudaStream_t st, uint64_t *launches) {
    if (nblocks <= 0) return cudaSuccess;
    k_p2p_final<<<unsigned(nblocks), 256, 0, st>>>(tasks, ntasks, insts, start, skeys, rec, le, pb,
                                                   dtype_f32, stage, nstage, ctrl, ntotal);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

cudaError_t launch_unsort(const InstDesc *insts, const uint32_t *perm, const float *stage,
                          int64_t nstage, const Task *utasks, int nutasks, int64_t unblocks,
                          cudaStream_t st, uint64_t *launches) {
    if (unblocks <= 0) return cudaSuccess;
    for (int comp = 0; comp < 2; ++comp) {
        k_unsort_f32<<<unsigned(unblocks), 256, 0, st>>>(utasks, nutasks, insts, perm,
                                                         stage + comp * nstage, comp);
        PF_LAUNCHED(1);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_p2p_f64(int grid, const uint4 *items, uint32_t *ctrl, const InstDesc *insts,
                           const uint32_t *start, const double *xs, const double *ys,
                           const double *gs, const uint32_t *perm, const double2 *le,
                           const double *gtab, int laplace, int dtype_f32,
                           unsigned long long *busy, cudaStream_t st, uint64_t *launches) {
    auto *k = laplace ? k_p2p_f64<true> : k_p2p_f64<false>;
    k<<<grid, P2P_THREADS, 0, st>>>(items, ctrl, insts, start, xs, ys, gs, perm, le, gtab,
                                    dtype_f32, busy);
    PF_LAUNCHED(1);
    return cudaGetLastError();
}

PF_DEFINE_CHECK_READER(p2p)

}  // namespace petfmm
