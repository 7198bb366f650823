// kernels.cuh -- host-side launchers of the FMM kernels (internal).
#pragma once
#include <vector>

#include "common.cuh"

namespace petfmm {

// Every launcher returns cudaGetLastError() after the launch and adds the
// number of kernels it launched to *launches.

// Bounds-checked build: the first failing PF_IN check's source line in each
// file (0: none), read and cleared (always 0 in the regular build).
unsigned pf_checks_tree();
unsigned pf_checks_expansions();
unsigned pf_checks_p2p();
unsigned pf_checks_smooth();
unsigned pf_checks_shifts();
unsigned pf_checks_orbits();
unsigned pf_checks_fmm3d();

// ---- tree.cu ---------------------------------------------------------------
// Sec. 2.1 binning + z-order key of every particle (composite key for batches);
// if recu != nullptr also its mixed-path record (see launch_gather_mixed) in
// input order.
cudaError_t launch_morton(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                          int dtype_f32, uint32_t *keys, float4 *recu, int *status,
                          cudaStream_t st, uint64_t *launches);

// Scratch (uint32 words) needed by exclusive_scan for n elements.
int64_t scan_scratch_words(int64_t n);
// out[i] = sum_{j < i} in[j]; in may equal out.  If total != nullptr the sum
// of all elements is written there (device).
cudaError_t exclusive_scan(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *scratch,
                           uint32_t *total, cudaStream_t st, uint64_t *launches);

// Stable LSD radix sort of (key, value) over the low nbits bits (8-bit
// digits, at most 4 passes, n < 2^32); the initial values are the element
// indices.  Result ends up in (k0, v0) or (k1, v1): *result_in_first tells
// which.  scratch: radix_scratch_words(n) words (per-tile digit counts and
// their scan).
int64_t radix_blocks(int64_t n);
int64_t radix_scratch_words(int64_t n);
cudaError_t radix_sort(uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1, int64_t n,
                       int nbits, uint32_t *scratch, bool *result_in_first, cudaStream_t st,
                       uint64_t *launches);

// start[soff + b] = first sorted rank of leaf b (b = 0..4^L).
cudaError_t launch_leaf_start(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                              const uint32_t *skeys, uint32_t *start, cudaStream_t st,
                              uint64_t *launches);

// Sorted particle arrays.
cudaError_t launch_gather_f64(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                              int dtype_f32, const uint32_t *perm, double *xs, double *ys,
                              double *gs, cudaStream_t st, uint64_t *launches);
// rec[r] = recu[perm[r]]: (xi, eta, gamma, batch index) in sorted order, with
// (xi, eta) the offset from the leaf centre in leaf widths.
cudaError_t launch_gather_mixed(const float4 *recu, const uint32_t *perm, float4 *rec, int64_t n,
                                cudaStream_t st, uint64_t *launches);

// ---- expansions.cu ---------------------------------------------------------
// Operator tables for p (FP64 build; the mixed path's rounded to FP32),
// device-resident.
struct OpTables {
    int p = 0;
    void *blob = nullptr;       // the allocation behind the tables
    double *shift64 = nullptr;  // M2M and L2L (shifts.cu)
    float *shift32 = nullptr;
    float2 *m2l32 = nullptr;    // per-box M2L of the tensor cores' sparse units
    double *orbit64 = nullptr;  // M2L by orbits (m2l_orbits.cu)
    float *orbit32 = nullptr;
    float *m2l_tc = nullptr;  // hi/lo B images for the tensor-core M2L (p <= 24)
    float *m2l_tcb = nullptr; // ... the four target classes side by side (block units)
};
// Those of one precision, copied on st: the launches that follow there find them
// complete.  build_tc_image: one of the tensor cores' images (mixed path, p <=
// 24), if it is not there yet; 0.35 ms of host time at p = 17, so only where a
// plan has such units.
cudaError_t build_op_tables(int p, int kernel, bool fp64, OpTables *out, cudaStream_t st);
cudaError_t build_tc_image(int kernel, bool blocks, OpTables *t, cudaStream_t st);
cudaError_t copy_table(void *dst, const void *src, size_t bytes, cudaStream_t st);
// The FP64 table behind them: which = 0 M2M [c][l][k], 1 L2L [c][n][m],
// 2 M2L [op][k][m], complex as (re, im) pairs.
void host_op_table(int p, int kernel, int which, std::vector<double> &out);
void free_op_tables(OpTables *t);
void host_m2l_table(int p, double *out_re_im /* 40 * p * p * 2, [op][k][m] */);
// Interaction list exactly as the kernels enumerate it; returns the count.
int host_interaction_list(int level, int ix, int iy, int32_t *out);
// Number of (target, source) M2L translations of levels 2..L.
int64_t m2l_pair_count(int L);

// occ[0 .. ctrl[CTRL_NOCC]) = (instance, leaf) of every occupied leaf, in no
// particular order (one thread per leaf of the tasks).
cudaError_t launch_occ_list(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, uint2 *occ, uint32_t *ctrl, cudaStream_t st,
                            uint64_t *launches);
// P2M of the listed leaves by a persistent grid (max_occ bounds the list).
template <typename R>
cudaError_t launch_p2m(const uint2 *occ, const uint32_t *ctrl, int64_t max_occ,
                       const InstDesc *insts, int pmax, const uint32_t *start, const double *xs,
                       const double *ys, const double *gs, const float4 *rec,
                       typename Cplx<R>::T *me, cudaStream_t st, uint64_t *launches);
// M2M, M2L and L2L skip boxes with no particles in their subtree (and M2L
// skips empty sources): their coefficients would be exactly zero and are
// never read.  start = the batch's leaf-start array.
//
// Per-box M2L (mixed path) of the boxes that the tensor-core units of the
// tasks' levels leave: those of sparse units (ucount, dense_pct).
cudaError_t launch_m2l(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                       const uint32_t *start, const float2 *me, float2 *le, const uint32_t *ucount,
                       int dense_pct, cudaStream_t st, uint64_t *launches);

// ---- shifts.cu -------------------------------------------------------------
// M2M (into the tasks' parents) and L2L (from them) of one level per instance;
// ex: ME or LE.  A task: instance, the parents' level; units: shift_units
// blocks.  smem: the largest shift_smem of the orders in the plan.
// InstDesc::t_shift = host_shift_table of its order and kernel.
void host_shift_table(int p, int kernel, std::vector<double> &out);
int64_t shift_units(int p, int level);
size_t shift_smem(int p, bool fp64, bool top);
template <typename R>
cudaError_t launch_shift(bool l2l, const Task *tasks, int ntasks, int64_t nblocks, size_t smem,
                         const InstDesc *insts, const uint32_t *start, typename Cplx<R>::T *ex,
                         cudaStream_t st, uint64_t *launches);
// Mixed path: the parents' levels 2 .. kShiftTop of every instance in one
// launch, a block each.  (64 + 16 parents take 11 to 12 us there, one way, p = 17;
// the FP64 path spreads them over the SMs.)
constexpr int kShiftTop = 3;
cudaError_t launch_shift_top(bool l2l, int ninst, size_t smem, const InstDesc *insts,
                             const uint32_t *start, float2 *ex, cudaStream_t st,
                             uint64_t *launches);

// ---- m2l_tc.cu -------------------------------------------------------------
// Tensor-core M2L (mixed path) for levels with at least 128 parent cells per
// row and p <= 24: one CTA per (target class, parent row, segment) unit.
bool m2l_tc_supported(int p, int level, int segmax);
// block units (8 x 16 parent cells, all four target classes), levels >= 5
bool m2l_tcb_supported(int p, int level);
int64_t m2l_tcb_units(int level);
size_t m2l_tcb_smem_bytes(int p);
void host_m2l_tcb_images(int p, int kernel, std::vector<float> &out);
// pmax: the largest order among the launch's units (sizes shared memory)
cudaError_t launch_m2l_tcb(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                           const uint32_t *start, const float2 *me, float2 *le,
                           const uint32_t *ucount, int dense_pct, int pmax, long long spin_limit,
                           int pipe, int *status, cudaStream_t st, uint64_t *launches);
int64_t m2l_tc_units(int level, int segmax);
size_t m2l_tc_smem_bytes(int p, int seg);
int m2l_tc_seg(int level, int segmax);
void host_m2l_tc_images(int p, int kernel, std::vector<float> &out);
void host_lap_m2l_table(int p, double *out_re_im /* 40 * p * p * 2, [op][k][m] */);
// Laplace kernel: the level-dependent constant of M2L, added after every M2L
// kernel (tasks: instance, level; units: 4^l target boxes).
template <typename R>
cudaError_t launch_m2l_logterm(const Task *tasks, int ntasks, int64_t nblocks,
                               const InstDesc *insts, const uint32_t *start,
                               const typename Cplx<R>::T *me, typename Cplx<R>::T *le,
                               cudaStream_t st, uint64_t *launches);
// ucount[u] = targets holding particles in unit u of the launch.
cudaError_t launch_tc_unit_count(const Task *tasks, int ntasks, int64_t nunits,
                                 const InstDesc *insts, const uint32_t *start, uint32_t *ucount,
                                 cudaStream_t st, uint64_t *launches);
// Dense units (tc_unit_dense) on the tensor cores; the SIMT launch covers the
// boxes of the other units of the same levels.
cudaError_t launch_m2l_tc(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                          const uint32_t *start, const float2 *me, float2 *le,
                          const uint32_t *ucount, int dense_pct, size_t smem_bytes,
                          long long spin_limit, int *status, cudaStream_t st, uint64_t *launches);

// ---- m2l_orbits.cu ---------------------------------------------------------
// M2L by orbits of quarter turns: the FP64 path, and the mixed path's levels
// that the tensor cores do not take (InstDesc::t_m2l = the
// host_m2l_orbit_table of its order and kernel).  A unit (one block) is a run
// of target boxes of one class holding about ni 128 (box, coefficient) pairs;
// ni is 1 or M2L_ORBIT_NI_MAX, the same results either way.
constexpr int M2L_ORBIT_NI_MAX = 2;  // (FP64 path only)
void host_m2l_orbit_table(int p, int kernel, std::vector<double> &out);
int64_t m2l_orbit_units(int p, int level, int ni);
size_t m2l_orbit_smem(int p, int ni, bool fp64);
template <typename R>
cudaError_t launch_m2l_orbits(const Task *tasks, int ntasks, int64_t nblocks, int ni, size_t smem,
                              const InstDesc *insts, const uint32_t *start,
                              const typename Cplx<R>::T *me, typename Cplx<R>::T *le,
                              cudaStream_t st, uint64_t *launches);

// units of work per block of each expansion kernel (the host plans with them)
constexpr int P2M_WARPS = 4;      // warps per block
constexpr int M2L_WARPS = 4;      // warps per block
// Each warp of the SIMT M2L owns a run of consecutive boxes and skips the
// empty ones after one ballot: at the clustered workload 87% of the leaves
// are empty, and a block per few boxes made the kernel bound by block
// scheduling.
constexpr int BOX_RUN = 8;
constexpr int M2L_BOXES = M2L_WARPS * BOX_RUN;   // target boxes per block
constexpr int EXP_THREADS = 256;  // (box, coefficient) pairs per block of petfmm_debug_plan's M2M / L2L

// ---- p2p.cu ----------------------------------------------------------------
// Work list: items (inst, leaf, first target rank, target count) for every
// occupied leaf, tpi targets per item.  ctrl[CTRL_NITEMS] receives the count.
enum { CTRL_STATUS = 0, CTRL_NITEMS = 1, CTRL_QUEUE = 2, CTRL_PAIRS_LO = 4, CTRL_NOCC = 6,
       CTRL_NPAIRS = 7, CTRL_QUEUE2 = 8, CTRL_NXTRA = 9, CTRL_SYM_LO = 10, CTRL_NSMOOTH = 12,
       CTRL_CLASSES = 16, CTRL_WORDS = 288 };  // from CTRL_CLASSES: the items' work classes
cudaError_t launch_p2p_worklist(const Task *tasks, int ntasks, int64_t nblocks,
                                const InstDesc *insts, const uint32_t *start, int tpi, int ordered,
                                uint4 *items, int64_t cap, uint32_t *ctrl, cudaStream_t st,
                                uint64_t *launches);
cudaError_t launch_p2p_f64(int grid, const uint4 *items, uint32_t *ctrl, const InstDesc *insts,
                           const uint32_t *start, const double *xs, const double *ys,
                           const double *gs, const uint32_t *perm, const double2 *le,
                           const double *gtab, int laplace, int dtype_f32,
                           unsigned long long *busy, cudaStream_t st, uint64_t *launches);
// The table behind its kernel factor (vortex), G64_WORDS doubles.
constexpr int G64_CELLS = 640, G64_TERMS = 7, G64_WORDS = G64_CELLS * (G64_TERMS + 1);
const double *host_g64_table();
// g(q) by it, on the device.
cudaError_t launch_g64(const double *q, double *g, int64_t n, const double *gtab, cudaStream_t st);
// Mixed near field from work items, every leaf against all 9 leaves: own[r] =
// the near sum of sorted blob r (launch_p2p_final then adds the far field).
cudaError_t launch_p2p_mixed(int grid, int deg, int general, const uint4 *items, uint32_t *ctrl,
                             const InstDesc *insts, const uint32_t *start, const float4 *rec,
                             float2 *own, int laplace, unsigned long long *busy, cudaStream_t st,
                             uint64_t *launches);
// Mixed near field, one thread per target: own[r] = blob r's sum over the
// leaves not summed pairwise with its own (tasks over blobs).
cudaError_t launch_near_direct(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                               const uint32_t *start, const uint32_t *skeys, const float4 *rec,
                               float2 *own, uint32_t *ctrl, unsigned long long *busy, int nbusy,
                               cudaStream_t st, uint64_t *launches);
// (busy: of the SMs with identifiers below nbusy the first start, preset to
// all ones, and the last end.)
// Fewest blobs in both leaves of a pair for the pair kernel.
constexpr uint32_t P2P_PAIR_MIN = 32;
// Pairwise near field between neighbouring leaves (mixed path).  Buffers:
// own[N]: each blob's directly summed part (sorted order; the only one used
// by the modes without pairs, part == nullptr there); part: 9 slots of
// nslot float2 (slot d: A's blobs from forward neighbour d, slot 4 + d: B's
// blobs from A, slot 8: each blob from the other blobs of its leaf); xtab[4 nleaves]: per (leaf, direction) of a split
// pair its scratch base (all ones: not split); lflags[nleaves]: per leaf,
// which of these hold its blobs' sums; xs[xcap]: the scratch runs of pieces
// 1 .. of split pairs.
struct PairBufs {
    float2 *own, *part;
    int64_t nslot;
    uint32_t *xtab, *lflags;
    float2 *xs;
    int64_t xcap;
};
// ... the item list (inst, leaf A, direction | swap << 3 | piece << 4,
// scratch base; direction 4: the leaf's own pairs), at most cap of them,
// heaviest first (ordered),
// ctrl[CTRL_NPAIRS] its count, ctrl[CTRL_NXTRA] the scratch entries wanted ...
cudaError_t launch_pair_worklist(const Task *tasks, int ntasks, int64_t nblocks,
                                 const InstDesc *insts, const uint32_t *start, int ordered,
                                 uint4 *items, int64_t cap, uint32_t *ctrl, const PairBufs &pb,
                                 cudaStream_t st, uint64_t *launches);
// ... the pair items, one persistent launch ...
int p2p_pairs_grid(int deg, int general);
cudaError_t launch_p2p_pairs(int grid, int deg, int general, const uint4 *pitems, uint32_t *ctrl,
                             const InstDesc *insts, const uint32_t *start, const float4 *rec,
                             const PairBufs &pb, unsigned long long *busy, cudaStream_t st,
                             uint64_t *launches);
// Either mode's final pass: far field (L2P) + own + pair slots per blob,
// written at the caller's index (tasks over blobs).
cudaError_t launch_p2p_final(const Task *tasks, int ntasks, int64_t nblocks,
                             const InstDesc *insts, const uint32_t *start, const uint32_t *skeys,
                             const float4 *rec, const float2 *le, const PairBufs &pb,
                             int dtype_f32, float *stage, int64_t nstage, const uint32_t *ctrl, int64_t ntotal, cudaStream_t st, uint64_t *launches);
// (stage != nullptr, FP32 outputs: the pass writes u, v in sorted order to
// stage[0 .. nstage) and stage[nstage ..), and launch_unsort scatters them
// to the caller's arrays through perm, one launch per component; utasks: the
// blobs of every instance, 1024 per block.)
cudaError_t launch_unsort(const InstDesc *insts, const uint32_t *perm, const float *stage,
                          int64_t nstage, const Task *utasks, int nutasks, int64_t unblocks,
                          cudaStream_t st, uint64_t *launches);
// ---- smooth.cu -------------------------------------------------------------
// Near field by expansions where the blob core is wide against a leaf
// (instances with InstDesc::smdeg > 0).  sm_degree: the degree for
// kappa = w^2 / 2 sigma^2 and the context's near-field tolerance, 0 where
// the pairs are summed.
// (kNearTolDefault: that of a new context, PETFMM_OPT_NEAR_TOL.)
constexpr double kNearTolDefault = 2.5e-6;
int sm_degree(double kappa, double near_tol);
size_t sm_row_floats(int n);
int64_t sm_max_rows(int n, int64_t blobs, int64_t leaves);
void host_sm_operators(double kappa, int n, std::vector<float> &out);
// The operators of one (degree, kappa) on the device: sm_operator_floats(n)
// floats at out, from the degree's host_sm_fixed table (a device copy), launched
// on st; work: sm_work_bytes of the largest degree and the number of operators.
const std::vector<double> &host_sm_fixed(int n);
size_t sm_operator_floats(int n);
size_t sm_work_bytes(int n, size_t ops);
struct SmOperator {
    int n;
    double kappa;
    const double *fixed;
    float *out;
};
cudaError_t launch_sm_operators(const std::vector<SmOperator> &ops, int nmax, double *work,
                                cudaStream_t st, uint64_t *launches);
// lmask, lrank: per leaf, its neighbours summed directly / by expansion, and
// its row of mom (moments) and loc (local expansions); list: (instance, leaf)
// of each row; rows of `row` floats.
struct SmBufs {
    uint32_t *lmask, *lrank;
    uint2 *list;
    float *mom, *loc;
    int64_t rows;
    int row;
};
// The occupied list (in place of launch_occ_list) and the lists of sb.
cudaError_t launch_sm_lists(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, uint2 *occ, uint32_t *ctrl, const SmBufs &sb,
                            cudaStream_t st, uint64_t *launches);
// Moments and local expansions of the degrees in the bit set; needs the
// lists and the gathered records.
cudaError_t launch_sm_near(uint32_t degrees, const uint32_t *ctrl, const InstDesc *insts,
                           const uint32_t *start, const float4 *rec, const SmBufs &sb,
                           cudaStream_t st, uint64_t *launches);
// These instances' blobs: far field, near field, output (or stage, sorted).
cudaError_t launch_sm_final(const Task *tasks, int ntasks, int64_t nblocks, const InstDesc *insts,
                            const uint32_t *start, const uint32_t *skeys, const float4 *rec,
                            const float2 *le, const SmBufs &sb, int dtype_f32, float *stage,
                            int64_t nstage, cudaStream_t st, uint64_t *launches);

int p2p_grid(int precision_mixed, int deg, int general, int laplace);
int device_sm_count();
constexpr int P2P_TPI_F64 = 16;
constexpr int P2P_TPI_MIXED = 64;

}  // namespace petfmm
