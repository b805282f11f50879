// nb_internal.cuh - internal types shared by the translation units of the
// GB300 non-bonded library (never installed; the public ABI is acenb.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>
#include <vector>

#include "acenb.h"

namespace acenb {

constexpr int kCluster = 8;          // atoms per cluster (column chunk)
constexpr int kMaxTypes = 64;        // type-pair table lives in shared memory
constexpr int kMaxPartners = 16;     // exclusion + 1-4 partners per atom
constexpr int kErfcDeg = 8;          // degree of the erfcx polynomial in t
constexpr int kExp2Deg = 6;          // degree of the 2^f polynomial on [-1/2, 1/2]
constexpr int kDefaultListSplit = 1; // tile kernels: work units per segment of a group list
constexpr int kMaxGroup = 8;         // clusters per i-group, largest (the masks hold 8 bits)
constexpr int kDefaultGroup = 1;     // clusters per i-group, default (the autotuner may choose 4 or 8)
constexpr int kMaskRecsPerCluster = 6; // exclusion-mask records allocated per cluster
constexpr int kListSegs = 4;         // segments of a group's list (one per list-kernel warp)
constexpr double kFixScale = 4294967296.0;   // 2^32: fixed-point scale
constexpr int kTaskVals = 8;         // per system: E_lj, E_c (scale 2^32), W[6] (scale 2^20)
constexpr double kVirScale = 1048576.0;      // 2^20: fixed-point scale of the virial sums
constexpr int kPmeAcc = 9;           // PME sums: E_recip, E_self, E_excl (2^32), W[6] (2^20)
constexpr int kPmeMaxGrid = 1024;    // largest PME grid edge
struct PmeState;                     // smooth PME state of a single-system context (nb_pme.cu)
struct MdState;                      // molecular-dynamics state of a single-system context (nb_md.cu)
// Padding slots of the sorted arrays sit at this finite, far-away coordinate:
// their squared distance to any atom (about 3e36) stays finite and is never
// inside a cutoff, so masked pair arithmetic needs no further guards.
constexpr float kPadCoord = -1.0e18f;
__host__ __device__ inline bool is_real_coord(float x) { return x > -1.0e17f; }

// Group list entry (uint2).  x: J (bits 0..24) | shift codes x,y,z (2 bits
// each, bits 25..30: 0 none, 1 = j-side shift x_j - L, 2 = i-side shift
// x_i - L) | mask flag (bit 31: the entry's tiles have exclusion masks).
// y: the group's clusters in reach of J (low bits, one per cluster of the
// group) | mask record (the bits above, when flagged; see mask_field).
constexpr uint32_t kJMask = 0x01FFFFFFu;
constexpr int kShiftBit = 25;
constexpr uint32_t kExclFlag = 0x80000000u;
// Clusters of a context, capacity: at most kJMask, so that every index fits
// an entry and the list kernel's packed partners (index << 7, all ones: none).
constexpr int64_t kMaxClusterCap = kJMask;

// Device status bits (first error wins when reported).
enum : int {
    ST_NONFINITE = 1 << 0,
    ST_CAPACITY = 1 << 1,
    ST_STALE = 1 << 2,
    ST_OVERFLOW = 1 << 3,
    ST_BADTYPE = 1 << 4,
    ST_TIMEOUT = 1 << 5,
};

// Per-system descriptor (device resident).
struct SysDesc {
    float L[3];          // box edges
    float half[3];       // 0.5 * L (FP32, exact)
    float inv_w[2];      // nx / Lx, ny / Ly rounded to FP32 (column scale)
    float w[2];          // Lx / nx, Ly / ny (FP32, for list bounds)
    int nx, ny;          // columns per axis
    int atom_begin;      // first atom in the concatenated input arrays
    int n_atoms;
    int col_begin;       // first global column
    // z-bin index of every column: bins of height dz = Lz / nzb; per column
    // nzb + 1 pairs (first cluster with z_hi >= b dz, first cluster with
    // z_lo > (b + 1) dz), at zb_begin + local column * (nzb + 1)
    int nzb;
    int zb_begin;
    float inv_dz;        // nzb / Lz (FP32)
    float dz;            // Lz / nzb (FP32)
};

// Pair-model constants passed by value to kernels.
struct PairParams {
    float rc2;           // rc * rc (FP32, the membership threshold)
    float rc, rs2;       // FP32 cutoff and switch distance squared
    float sw_c0;         // rc2 - 3 rs2
    float sw_inv;        // 1 / (rc2 - rs2)^3
    float sw_a, sw_b, sw_c;  // 1 / (rc2 - rs2)^2, -2 sw_inv, 12 sw_inv (forward kernel's form of the switch)
    float ke;            // Coulomb constant
    float alpha_half;    // alpha / 2: t = 1 / (1 + (alpha/2) r)
    float alpha;         // Ewald alpha
    float neg_a2_log2e;  // -alpha^2 log2(e): exp(-alpha^2 r^2) = 2^(r2 * this)
    float neg_a2_log2e_lo; // the FP32 remainder: -alpha^2 log2(e) = neg_a2_log2e + this (to ~2^-48)
    float two_a_sqpi;    // 2 alpha / sqrt(pi)
    float s14_lj, s14_c;
    float list_margin;   // additive margin on bounding-box distances (A)
    float rcm2;          // (rc + list_margin)^2, bounding-box pruning threshold
    int n_types;
    int switched;        // rs < rc
    int ewald;           // alpha > 0
    float erfc_c[kErfcDeg + 1]; // erfcx(x) ~ sum c_k t^k on [0, alpha rc]
    float exp2_c[kExp2Deg + 1]; // 2^f ~ sum c_k f^k on [-1/2, 1/2]
    float rs;            // FP32 switch distance
    float tab_inv_h;     // n / rc (FP32) of the radial-function tables
    int tab_n;           // intervals of the tables (0: direct evaluation)
};

// The constants of the packed pair arithmetic (pair_radial2), each twice in
// one 64-bit word: an operand of fma.rn.f32x2 and the like.  Signs are chosen
// so that no operand has to be negated.
using f32x2 = unsigned long long;
struct PairConst2 {
    f32x2 rc2, rs2;
    f32x2 sw_a, sw_b, neg_sw_c;
    f32x2 neg_alpha_half;
    f32x2 a2_hi, neg_a2_hi, neg_a2_lo;  // c = -alpha^2 log2(e) as hi + lo: hi, -hi, -lo
    f32x2 two_a_sqpi;
    f32x2 magic;                        // 1.5 2^23
    f32x2 one, neg_one, neg_half, neg_zero;
    f32x2 erfc_c[kErfcDeg + 1];
    f32x2 exp2_c[kExp2Deg + 1];
};

// Where the binning of an atom goes (bin_atom).
struct BinArgs {
    const SysDesc *sys;
    float4 *wpos;
    int *atom_col;
    int *col_count;
    int *stage_fix;
    int col_cap;
    int *status;
};

struct DevBuffers {
    SysDesc *sys = nullptr;          // [n_sys]
    int *atom_sys = nullptr;         // [N]
    int *atom_col = nullptr;         // [N] global column of each atom
    float4 *wpos = nullptr;          // [N] wrapped coordinates (w: the charge when the step packs them)
    int *atom_t = nullptr;           // [N] range-checked types in caller order (nb_step and MD steps)
    int *part_orig = nullptr;        // [N*K] partner (orig << 1) | is14, -1 pad (static)
    int *col_sys = nullptr;          // [C] system of each column (static)
    int *col_count = nullptr;        // [2C+1] column histogram (zero between builds); with a scan (many columns)
                                     // [C] = completion ticket of the binning kernel, [C+1+c] = column c's count
                                     // for the column sort
    int *col_slot = nullptr;         // [C+1] padded slot offsets
    int *stage = nullptr;            // [S] unsorted atoms of a column whose staging row overflowed
    int *stage_fix = nullptr;        // [C * col_cap] unsorted atoms per column, fixed capacity
    float4 *xyzq = nullptr;          // [S] sorted x, y, z, q (kPadCoord for padding)
    int *tslot = nullptr;            // [S] sorted types
    int *perm = nullptr;             // [S] slot -> atom (-1 padding)
    int *inv = nullptr;              // [N] atom -> slot
    float4 *bb = nullptr;            // [NC*2] cluster bounding boxes (lo, hi interleaved)
    int *clus_sys = nullptr;         // [NC] system of each cluster
    long long *sys_acc = nullptr;    // [n_sys*kTaskVals] per-system fixed-point energies (2^32) and virial (2^20)
    long long *facc = nullptr;       // [S*3] fixed-point forces in sorted order (both atoms of each pair)
    long long *gacc = nullptr;       // [S*4] adjoint: fixed-point dL/dx, dL/dq in sorted order
    int *col_grp = nullptr;          // [C+1] first i-group of each column
    int2 *grp = nullptr;             // [GC] i-group: (first cluster, clusters)
    int *clus_grp = nullptr;         // [NC] i-group of each cluster
    uint2 *glist = nullptr;          // [GC*list_cap] per i-group: its list (Newton's third law at group level)
    int *glist_n = nullptr;          // [GC*kListSegs] lengths of the segments (list_cap / kListSegs entries each)
    ulonglong2 *gmask = nullptr;     // [MC*kMaxGroup] per flagged entry and group cluster: (excluded, 1-4) bits
    int2 *zbin = nullptr;            // [zb_total] z-bin index of the columns (see SysDesc)
    long long *tab_grad = nullptr;   // [T*T*2] adjoint dL/dsig_ab, dL/deps_ab (fixed point, one ordered half)
    int *counts = nullptr;           // [8]: n_slots, n_clusters, unpack ticket, work-unit counter,
                                     //      n_groups, mask records used, -, -
    int *status = nullptr;           // [1]
    float4 *lj_tab = nullptr;        // [T*T] (A, B, A - fl(A), B - fl(B)): FP32 and the FP32 remainders
    float4 *lj_d = nullptr;          // [T*T] 48 eps sig^11, 24 eps sig^5, 4 sig^12, 4 sig^6
    float4 *rtab = nullptr;          // [tab_n*3] tabulated radial functions (nb_set_tables)
    float4 *gslot = nullptr;         // [S] adjoint input dL/dF in sorted order
    float *eps_type = nullptr;       // [T] per-type epsilon (Lorentz-Berthelot chain)
    long long *dbg_n = nullptr;      // [4] debug counters: pair evaluations, pairs, tile halves with a pair, tiles
    int *dbg_ij = nullptr;           // [cap*2]
    int64_t dbg_cap = 0;
    float *scratch_f = nullptr;      // [N*3] debug force sink
    double *scratch_g = nullptr;     // [T*T*2] adjoint scratch
};

}  // namespace acenb

struct nb_ctx {
    int n_sys = 0;
    int64_t n_atoms = 0;
    int n_cols = 0;
    int64_t slot_cap = 0;
    int64_t clus_cap = 0;
    int K = 1;                     // partners per atom (>= 1)
    int comb_rule = 0;
    int stage_cap = 96;            // nb_tuning.stage_capacity (no effect on the kernels)
    int list_cap = 512;            // entries per group list
    int group = acenb::kDefaultGroup;  // clusters per i-group of the last/next build (4 or 8)
    int built_group = 0;           // the group size the current lists were built with
    int64_t grp_cap = 0;           // i-group slots (enough for groups of 4)
    int64_t mask_cap = 0;          // exclusion-mask records
    int col_cap = 0;               // atoms per column staging row (about twice the mean column)
    int tab_n = 0;                 // radial-function table intervals (0: direct evaluation)
    int64_t zb_total = 0;          // entries of the z-bin index
    int smem_optin = 0;            // device opt-in shared memory per block
    cudaStream_t stream = nullptr;
    int device = 0;
    int num_sms = 0;
    // resident blocks per SM of the single-cluster force kernel's instances
    // (block shape, radial functions, virial / debug), -1: not asked yet
    int force1_res[3][3][4] = {{{-1, -1, -1, -1}, {-1, -1, -1, -1}, {-1, -1, -1, -1}},
                               {{-1, -1, -1, -1}, {-1, -1, -1, -1}, {-1, -1, -1, -1}},
                               {{-1, -1, -1, -1}, {-1, -1, -1, -1}, {-1, -1, -1, -1}}};
    bool built = false;
    bool host_inputs = false;      // the step's charges and types were in host memory at the last query
    bool hist_dirty = false;       // an abandoned build's column counts could not be cleared yet
    acenb::PairParams pp{};
    nb_tuning tune{};
    std::vector<acenb::SysDesc> sys_h;
    std::vector<double> sig_tab, eps_tab;  // FP64 type-pair parameters
    acenb::DevBuffers d;
    acenb::PmeState *pme = nullptr;  // smooth PME, when enabled by nb_set_pme
    acenb::MdState *md = nullptr;    // molecular dynamics, after nb_md_init
    // profiling: event pairs around force-kernel launches
    bool profiling = false;
    std::vector<cudaEvent_t> prof_ev;
    int prof_n = 0;
};

namespace acenb {

// Wrap one FP32 coordinate into [0, L) with IEEE round-to-nearest operations
// in a fixed order: k = floor(x / L); x = fma(-k, L, x); then one conditional
// +L and one conditional -L.
__device__ __forceinline__ float wrap_coord(float x, float L)
{
    if (x >= 0.0f && x < L) return x;
    float k = floorf(__fdiv_rn(x, L));
    x = __fmaf_rn(-k, L, x);
    if (x < 0.0f) x = __fadd_rn(x, L);
    if (x >= L) x = __fsub_rn(x, L);
    return x;
}

// A fixed-point value (2^32) as the nearest FP32, the bits of
// __ll2float_rn(v) * 2^-32.  The 64-bit conversions run on the FP64 unit
// here, one warp in 64 cycles per SM sub-partition (measured: 0.015 warp
// instructions per cycle, 0.12 for the 32-bit ones); this takes about 14
// integer instructions and one 32-bit conversion: the leading 32 bits, the
// others ORed into the lowest one so that the rounding sees them.
__device__ __forceinline__ float fixed_to_float(long long v)
{
    const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = min(__clzll((long long)u), 63);
    const unsigned long long n = u << lz;
    const unsigned hi = (unsigned)(n >> 32) | ((unsigned)n != 0u ? 1u : 0u);
    const float f = __uint2float_rn(hi) * __int_as_float((127 - lz) << 23);  // 2^-lz: exact
    return v < 0 ? -f : f;
}

// The nearest fixed-point value (2^32) of an FP32, the bits of
// __float2ll_rn(f * 2^32), without the 64-bit conversion: the multiple of 1/2
// next to f by adding 1.5 2^22 (exact remainder, at most 1/4), the remainder
// by a 32-bit conversion.  |f| < 2^20 here; anything else takes the conversion.
__device__ __noinline__ inline long long float_to_fixed_wide(float f) { return __float2ll_rn(f * 4294967296.0f); }

__device__ __forceinline__ long long float_to_fixed(float f)
{
    if (!(fabsf(f) < 1048576.0f)) return float_to_fixed_wide(f);
    const float t = __fadd_rn(f, 6291456.0f);
    const float r = __fsub_rn(f, __fsub_rn(t, 6291456.0f));
    const int lo = __float2int_rn(__fmul_rn(r, 4294967296.0f));
    return (long long)(__float_as_int(t) - 0x4AC00000) * 2147483648ll + lo;
}

// Programmatic dependent launch.  Every kernel of the library calls
// pdl_entry() before it reads or writes anything that another kernel writes
// (at its start, or after a prologue that only fills shared memory from
// tables set at creation): griddepcontrol.wait blocks until the preceding
// kernel in the stream has completed and its memory is visible (a no-op for
// a plain launch), then launch_dependents lets the next kernel's blocks be
// scheduled while this one runs, so consecutive launches do not leave the
// GPU idle.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_entry()
{
    pdl_wait();
    pdl_trigger();
}

// Launch with programmatic stream serialization (see pdl_entry).  shared:
// with the largest shared-memory carve-out.  An SM changes its split between
// L1 and shared memory only when it is empty, so kernels that are to share
// SMs with the force kernel, which needs most of it, have to run with the same
// split (the steps with PME whose two chains run side by side: pme_beside).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_split(bool shared, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                             Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    cfg.attrs = attr;
    cfg.numAttrs = shared ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args)
{
    return launch_pdl_split(false, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

// Work units of the one-cluster force kernel per warp of a grid that fills the
// SMs with 32 warps.
inline int64_t force_rounds(const nb_ctx *ctx) { return kListSegs * ctx->clus_cap / (32 * ctx->num_sms); }

// Whether the PME chain is to share the SMs with the list and force kernels: then
// all kernels of a step ask for the same shared-memory split, the force kernel's
// blocks are not let in before the lists are done, and its grid leaves room.  Not
// for large systems, where each kernel fills the SMs by itself: the room left
// makes the force kernel, which is most of the step, longer, and the split takes
// the L1 that tables are read through.  Shared and not, us a step: 311 and 324 at
// 90,000 atoms, 408 and 407 at 120,000, 540 and 537 at 165,000, 641 and 630 at
// 200,001, 2,826 and 2,553 at 999,999; with tables 184 and 195 at 39,999, 264 and
// 264 at 60,000, 386 and 374 at 90,000, 610 and 560 at 150,000, 3,609 and 3,095 at
// 999,999.
constexpr int kShareRounds = 16, kShareRoundsTab = 7;
inline bool pme_beside(const nb_ctx *ctx)
{
    return ctx->pme && force_rounds(ctx) < (ctx->tab_n > 0 ? kShareRoundsTab : kShareRounds);
}

// i-group slots for a context: every column's clusters form groups of
// `group` clusters, the last one partial, so at most NC / group + C; the
// capacity covers every supported group size (groups of one cluster: NC).
inline int64_t group_capacity(int64_t clus_cap) { return clus_cap + 1; }
// exclusion-mask records (one 16-byte mask pair per cluster of the group, so
// `group` of them per record): the self tiles (one per cluster) and the
// entries whose cluster holds a topology partner of a group atom (a few per
// cluster).  Group (c0, n) fills records c0 kMaskRecsPerCluster ..
// (c0 + n) kMaskRecsPerCluster - 1, the rest come from a shared pool behind
// them.
inline int64_t mask_pool_base(int64_t clus_cap) { return clus_cap * kMaskRecsPerCluster; }
inline int64_t mask_capacity(int64_t clus_cap) { return mask_pool_base(clus_cap) + clus_cap / 2 + 64; }
// The mask record in an entry's y, above the group's cluster bits (1, 4 or 8).
// The 31 or 28 bits of the smaller groups hold the record's index.  The 24 bits
// of groups of 8 would name the records of 2.8 million clusters only: they
// count the group's own records (own >= 0: the record's place among them) from
// the group's first, then those of the pool.  (The same form for groups of 4
// cost 0.5 % of a step.)
constexpr int kOwnRecs8 = 8 * kMaskRecsPerCluster;
__host__ __device__ constexpr int mask_bit(int group) { return group; }
__host__ __device__ inline uint32_t mask_field(int group, long long slot, int own, long long pool_base)
{
    const long long k = group != 8 ? slot : (own >= 0 ? own : kOwnRecs8 + (slot - pool_base));
    return (uint32_t)k << mask_bit(group);
}
// atoms per column staging row for a mean column population: twice the mean
// and 32 more, in whole warps (rows that overflow are gathered by the column
// sort's slow fallback)
inline int column_capacity(double mean_atoms) { return ((int)(2.0 * mean_atoms) + 32 + 31) / 32 * 32; }

// Launchers implemented in the .cu files (all asynchronous on ctx->stream).
cudaError_t launch_build(nb_ctx *ctx, const float *d_pos);
// the two halves of launch_build: binning, column sort and cluster boxes;
// then the cluster-pair lists
// binned: the atoms were binned by the kernel before (the MD half-steps, when
// bins_elsewhere: one system, no scan, charges in device memory)
cudaError_t launch_build_cells(nb_ctx *ctx, const float *d_pos, const float *d_q = nullptr,
                               const int32_t *d_type = nullptr, bool binned = false);
// a build that failed on the host behind its binning: clears the counts that its
// list kernel would have cleared; returns e
cudaError_t abandon_build(nb_ctx *ctx, cudaError_t e);
// before anything bins: the column counts are zero
cudaError_t ready_histogram(nb_ctx *ctx);
BinArgs bin_args(const nb_ctx *ctx);
bool bins_elsewhere(nb_ctx *ctx, const float *d_q);
// beside_pme: the PME chain was forked before and is to run beside the lists
cudaError_t launch_build_lists(nb_ctx *ctx, bool beside_pme = false);
cudaError_t launch_forces(nb_ctx *ctx, const float *d_pos, const float *d_q, const int32_t *d_type,
                          float *d_F, double *d_energy, double *d_virial, bool debug_pairs);
// launch_forces after its pack (and, when pme_forked, the PME fork): the
// short-range kernel, the PME join and the unpack; beside_pme: the PME chain
// was forked early enough to share the SMs with the short-range kernel
cudaError_t launch_forces_packed(nb_ctx *ctx, float *d_F, double *d_energy, double *d_virial, bool debug_pairs,
                                 bool pme_forked, bool beside_pme);
size_t force_smem_for(int T, int scap, int K);
cudaError_t launch_pack(nb_ctx *ctx, const float *d_pos, const float *d_q, const int32_t *d_type, bool zero_sums);
cudaError_t launch_type_grad(nb_ctx *ctx, const double *gsig_tab, const double *geps_tab, double *gsig, double *geps);
cudaError_t launch_adjoint_tile(nb_ctx *ctx, const double *d_dLdE, float *d_dpos, float *d_dq);
// Smooth PME (nb_pme.cu): the reciprocal-space chain into the context's PME
// force and energy sums; the sums' device arrays (NULL when PME is off).
cudaError_t launch_pme(nb_ctx *ctx, const float *d_pos, const float *d_q);
// the same chain forked onto the PME side stream, and the join back.
// sums: also the pair-correction energy and virial (the forces always);
// zeroed: the PME sums were zeroed by the column sort
cudaError_t launch_pme_fork(nb_ctx *ctx, const float *d_pos, const float *d_q, bool sums = true, bool zeroed = false);
long long *pme_sums(const nb_ctx *ctx);
cudaError_t launch_pme_join(nb_ctx *ctx);
// the context's stream waits for whatever was launched on the PME streams (after an error)
void pme_rejoin(nb_ctx *ctx);
void pme_free(nb_ctx *ctx);
const long long *pme_forces_acc(const nb_ctx *ctx);
const long long *pme_sums_acc(const nb_ctx *ctx);
double pme_self_coef(const nb_ctx *ctx);  // -ke alpha / sqrt(pi), multiplies sum q^2
void md_free(nb_ctx *ctx);
// nb_debug_pair_terms: the forward kernel's pair arithmetic for given pairs
cudaError_t launch_debug_pair_terms(nb_ctx *ctx, long long n, const float4 *xi, const float4 *xj, const int *ti,
                                    const int *tj, float4 *out);
cudaError_t launch_backward(nb_ctx *ctx, const float *d_pos, const float *d_q, const int32_t *d_type,
                            const float *d_dLdF, const double *d_dLdE, float *d_dLdpos, float *d_dLdq,
                            double *d_dsig, double *d_deps);

}  // namespace acenb
