// nb_force.cu - the non-bonded force kernels (section "Molecular dynamics on
// the GPU": the non-bonded kernel computes the full Lennard-Jones and
// electrostatic force on each particle).  The paper's kernel does not reuse
// the reciprocal force F_ji; here both kernels do (Newton's third law): every
// unique pair is evaluated once, from the i-group whose list holds it, and
// its contribution goes to both atoms as 64-bit fixed point (2^32), so the
// sums stay exact and order independent.
//
// Forward: k_force1 for i-groups of one cluster (one warp per listed
// cluster pair as an 8 x 8 tile, the i cluster and its forces in registers,
// forces on j summed over lanes; see the comment above k_force1), k_force<G>
// for groups of 4 or 8 clusters (the group's atoms and i-force partials in
// shared memory; see the comment above k_force).
//
// Adjoint: k_adjoint1 and k_adjoint<G>, the same tiles, work units and
// staging with the pair adjoint; the type-pair gradients go to a block table
// in shared memory.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <atomic>

#include "nb_pair.cuh"

namespace acenb {

constexpr unsigned kFull = 0xffffffffu;

struct ForceArgs {
    const SysDesc *sys;
    const int *counts;
    int *work;                // work-unit counter of the tile kernels (zeroed by k_pack or the column sort)
    const float4 *xyzq;
    const int *tslot;
    const int *perm;
    const int *clus_sys;
    const int2 *grp;          // [GC] i-groups: (first cluster, clusters)
    const uint2 *glist;       // [GC*cap] per group: its list, kListSegs segments of cap / kListSegs
    const int *glist_n;       // [GC*kListSegs] segment lengths
    const ulonglong2 *gmask;  // exclusion bitmask records of the flagged entries
    int cap;                  // entries per group list
    int K;
    const float4 *lj_tab;     // [T*T] (A, B, A - fl(A), B - fl(B))
    const float4 *rtab;       // [n*3] tabulated radial functions, or null
    long long *facc;          // [S*3] fixed-point forces in sorted order (forward)
    long long *sys_acc;
    int *status;
    long long *dbg_n;
    int *dbg_ij;
    long long dbg_cap;
    PairParams P;
    PairConst2 C;             // packed constants of P
    // adjoint only
    const float4 *gslot;     // [S] dL/dF in sorted order (x, y, z, 0)
    const double *dLdE;      // [n_sys*2] dL/dE_LJ, dL/dE_C, or null
    const float4 *lj_d;      // [T*T] 48 eps sig^11, 24 eps sig^5, 4 sig^12, 4 sig^6
    long long *tab_acc;      // [T*T*2] fixed-point dL/dsig_ab, dL/deps_ab (each unique pair in one order)
    long long *gacc;         // [S*4] fixed-point dL/dx, dL/dq in sorted order (both atoms of each pair)
    const ulonglong2 *pool8;  // groups of 8: where record number 0 of the pool's count would be
};

// The masks of a flagged entry of a group of G clusters, one pair per cluster
// (own8: groups of 8, the group's first own record).
template <int G>
__device__ __forceinline__ const ulonglong2 *entry_record(const ForceArgs &A, uint32_t y, const ulonglong2 *own8)
{
    const uint32_t k = y >> mask_bit(G);
    if constexpr (G == 8) return (k < kOwnRecs8 ? own8 : A.pool8) + k * 8ull;
    return A.gmask + (unsigned long long)k * G;
}

__device__ __forceinline__ long long to_fixed(float v, int *status)
{
    // |v| < 2^26 keeps a sum of 32 lanes inside int64 at scale 2^32
    if (!(fabsf(v) < 67108864.0f)) {
        atomicOr(status, ST_OVERFLOW);
        return 0;
    }
    return __float2ll_rn(v * 4294967296.0f);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Slot of atom k of staged entry e (swizzle by e, conflict-free lane access).
__device__ __forceinline__ int swz(int e, int k) { return e * kCluster + (k ^ (e & (kCluster - 1))); }

struct Acc {
    float fx, fy, fz, elj, ec;
};

struct AccAdj {
    float dx, dy, dz, dq;
};

constexpr double kTabScale = 4294967296.0;  // fixed-point scale of the parameter gradients (2^32)

__device__ __forceinline__ long long to_fixed_tab(float v, int *status)
{
    if (!(fabsf(v) < 1073741824.0f)) {  // 2^30 per contribution
        atomicOr(status, ST_OVERFLOW);
        return 0;
    }
    return __float2ll_rn(v * (float)kTabScale);
}

// Adjoint of one ordered pair (i, j) for L = sum G.F + gE_lj E_lj + gE_c E_C.
// With d = x_j - x_i, F_i = h d where h = U'(r)/r, and g = G_i - G_j:
//   dL/dx_i -= h g + (h'/r)(g.d) d + (gE-weighted h) d     (h' = dh/dr)
//   dL/dq_i += w_c ke q_j (phi'(r)/r (g.d) + gE_c phi(r))
//   dL/dsig_ab, dL/deps_ab (each unique pair is visited once)
// through dU/dA = w S r^-12, dU/dB = -w S r^-6 and the chain factors
// dA/dsig = 48 eps sig^11, dB/dsig = 24 eps sig^5, dA/deps = 4 sig^12,
// dB/deps = 4 sig^6 of the type pair.
struct AdjTables {
    const float2 *lj;           // (A, B) per type pair
    const float4 *ljd;          // derivative factors per type pair
    unsigned long long *tacc;   // block table of fixed-point parameter gradients
};

template <bool EWALD>
__device__ __forceinline__ void eval_pair_adj(const PairParams &P, const AdjTables &S, int ti_row, float qi_ke, float gix,
                                              float giy, float giz, float gE_lj, float gE_c, bool in, float dx,
                                              float dy, float dz, float r2, float qj, int tj, float4 gj, bool is14,
                                              int *status, AccAdj &acc, float &jx, float &jy, float &jz, float &jq,
                                              float &dsig, float &deps)
{
    if (!in) {  // masked lanes: keep every product finite (padding sits far away)
        dx = 0.0f;
        dy = 0.0f;
        dz = 0.0f;
    }
    const float rinv = fast_rsqrt(r2);
    const float r = r2 * rinv, ir2 = rinv * rinv;
    const float2 ab = S.lj[ti_row + tj];
    const float ir6 = ir2 * ir2 * ir2, ir12 = ir6 * ir6;
    // LJ V = A r^-12 - B r^-6 and its r-derivatives
    const float t12 = ab.x * ir12, t6 = ab.y * ir6;
    const float V = t12 - t6;
    const float V1 = (6.0f * t6 - 12.0f * t12) * rinv;
    const float V2 = (156.0f * t12 - 42.0f * t6) * ir2;
    // switch S(r), S', S'' (r > rs)
    float Sw = 1.0f, S1 = 0.0f, S2 = 0.0f;
    if (r2 > P.rs2) {
        const float t = P.rc2 - r2, u = P.rs2 - r2;
        Sw = t * t * fmaf(2.0f, r2, P.sw_c0) * P.sw_inv;
        S1 = 12.0f * r * t * u * P.sw_inv;
        S2 = 12.0f * (t * u - 2.0f * r2 * u - 2.0f * r2 * t) * P.sw_inv;
    }
    const float wlj = is14 ? P.s14_lj : 1.0f;
    const float wc = is14 ? P.s14_c : 1.0f;
    const float Ulj1 = wlj * fmaf(S1, V, Sw * V1);
    const float Ulj2 = wlj * (S2 * V + 2.0f * S1 * V1 + Sw * V2);
    // Coulomb phi = erfc(a r)/r and its r-derivatives (without q_i q_j)
    float phi, phi1, phi2;
    if (EWALD) {
        const float tt = fast_rcp(fmaf(P.alpha_half, r, 1.0f));
        const float ex = fast_exp2(r2 * P.neg_a2_log2e);
        const float erfcv = ex * erfcx_poly(P, tt);
        const float cg = P.two_a_sqpi * ex;
        phi = erfcv * rinv;
        phi1 = -(cg + phi) * rinv;
        phi2 = 2.0f * P.alpha * P.alpha * cg + 2.0f * (cg + phi) * ir2;
    } else {
        phi = rinv;
        phi1 = -ir2;
        phi2 = 2.0f * ir2 * rinv;
    }
    const float qq = qi_ke * qj;
    const float U1 = fmaf(wc * qq, phi1, Ulj1);
    const float U2 = fmaf(wc * qq, phi2, Ulj2);
    const float h = U1 * rinv;
    const float h1r = (U2 - U1 * rinv) * ir2;  // (dh/dr) / r
    const float gx = gix - gj.x, gy = giy - gj.y, gz = giz - gj.z;
    const float gd = fmaf(gx, dx, fmaf(gy, dy, gz * dz));
    const float hE = (gE_lj * Ulj1 + gE_c * wc * qq * phi1) * rinv;
    const float cd = fmaf(h1r, gd, hE);
    const float m = in ? 1.0f : 0.0f;
    // the pair seen from j: d -> -d and g -> -g, so dL/dx_j gets the opposite
    // of dL/dx_i's term and dL/dq_j the same bracket times q_j's partner q_i
    jx = m * fmaf(h, gx, cd * dx);
    jy = m * fmaf(h, gy, cd * dy);
    jz = m * fmaf(h, gz, cd * dz);
    acc.dx -= jx;
    acc.dy -= jy;
    acc.dz -= jz;
    const float xq = m * wc * fmaf(phi1 * rinv, gd, gE_c * phi);
    acc.dq += xq * P.ke * qj;
    jq = xq * qi_ke;
    // type-pair parameters
    const float uA = wlj * Sw * ir12, uB = -wlj * Sw * ir6;
    const float uA1 = wlj * fmaf(S1, ir12, -12.0f * Sw * ir12 * rinv);
    const float uB1 = -wlj * fmaf(S1, ir6, -6.0f * Sw * ir6 * rinv);
    const float gA = fmaf(uA1 * rinv, gd, gE_lj * uA), gB = fmaf(uB1 * rinv, gd, gE_lj * uB);
    const float4 c = S.ljd[ti_row + tj];
    dsig = in ? fmaf(gA, c.x, gB * c.y) : 0.0f;
    deps = in ? fmaf(gA, c.z, gB * c.w) : 0.0f;
}

// 64-bit integer add to shared memory by two native 32-bit atomics: the low
// word's carry (seen from the value the first atomic returns) goes into the
// high word, so the 64-bit sum is exact and order independent.  (A 64-bit
// shared-memory atomic add is a compare-and-swap loop here, and many lanes
// of a warp hit the same few type-pair slots: the loop's retries cost more
// than the whole pair adjoint.)
__device__ __forceinline__ void shared_add64(unsigned long long *p, unsigned long long v)
{
    unsigned int *w = reinterpret_cast<unsigned int *>(p);  // little endian: low word first
    const unsigned int lo = (unsigned int)v, hi = (unsigned int)(v >> 32);
    const unsigned int old = atomicAdd(w, lo);
    const unsigned int h = hi + ((unsigned int)(old + lo) < old ? 1u : 0u);
    if (h) atomicAdd(w + 1, h);
}

// Add a lane's type-pair derivatives (key = t_i T + t_j, -1 for a masked
// lane) to the block table.  (Summing equal keys over the warp first, by
// match/ballot rounds or by the warp's integer reduction on 21-bit parts, was
// slower than the atomics: 0.37 and 0.50 ms against 0.19 ms per adjoint
// step.)
__device__ __forceinline__ void add_type_grads(const AdjTables &S, int key, float dsig, float deps, int *status)
{
    if (key >= 0) {
        shared_add64(&S.tacc[2 * key], (unsigned long long)to_fixed_tab(dsig, status));
        shared_add64(&S.tacc[2 * key + 1], (unsigned long long)to_fixed_tab(deps, status));
    }
}

// One candidate pair of the forward kernel: d = x_j - x_i (exact-shift
// image), r2 its FP32 squared length; the arithmetic is done for every
// candidate and masked by `in`.  RAD: radial functions evaluated directly
// with plain Coulomb (0) or Ewald (1), or interpolated from the tables (2).
// W14: the pair may be a scaled 1-4 pair (is14), else both weights are 1
// (the same bits either way for an unscaled pair).  lj holds (A, B, 12 A,
// 6 B) per type pair.  The force on i is subtracted from acc and the force
// on j added to fj with explicit FMA, so that the bits do not depend on how
// the caller was inlined.
// The LJ coefficients of the forward kernels in shared memory: lj (A, B,
// 12 A, 6 B) per type pair, followed by lo (the FP32 remainders of A, B).
template <int RAD, bool W14>
__device__ __forceinline__ float pair_fs(const PairParams &P, const float4 *__restrict__ lj,
                                         const float4 *__restrict__ rtab, int ti_row, float qi, bool in, float r2,
                                         float qj, int tj, bool is14, float &elj_acc, float &ec_acc)
{
    float rinv, r;
    pair_rinv(r2, rinv, r);
    const float r2inv = __fmul_rn(rinv, rinv);
    const float4 ab = lj[ti_row + tj];
    const float2 lo = reinterpret_cast<const float2 *>(lj + P.n_types * P.n_types)[ti_row + tj];
    float elj, frlj, ec, frc;
    if constexpr (RAD == 2)
        pair_radial_tab(P, rtab, r, ab.x, ab.y, lo, qi * qj, elj, frlj, ec, frc);
    else
        pair_radial<RAD == 1, true>(P, r2, r, rinv, r2inv, ab, lo, qi * qj, elj, frlj, ec, frc);
    // F_i = U'(r) d / r = -fs d with fs = -U'(r) / r
    float fs, wel, wec;
    if (W14) {
        const float wlj = is14 ? P.s14_lj : 1.0f;
        const float wc = is14 ? P.s14_c : 1.0f;
        fs = __fmul_rn(__fmaf_rn(wlj, frlj, __fmul_rn(wc, frc)), r2inv);
        wel = __fmul_rn(wlj, elj);
        wec = __fmul_rn(wc, ec);
    } else {
        fs = __fmul_rn(__fadd_rn(frlj, frc), r2inv);
        wel = elj;
        wec = ec;
    }
    elj_acc = __fadd_rn(elj_acc, in ? wel : 0.0f);
    ec_acc = __fadd_rn(ec_acc, in ? wec : 0.0f);
    return in ? fs : 0.0f;
}

// One pair: fs as above, the force on i subtracted from acc and the force on
// j added to fj with explicit FMA (bits independent of inlining).
template <int RAD, bool W14>
__device__ __forceinline__ void eval_pair(const PairParams &P, const float4 *__restrict__ lj,
                                          const float4 *__restrict__ rtab, int ti_row, float qi, bool in, float dx,
                                          float dy, float dz, float r2, float qj, int tj, bool is14, Acc &acc,
                                          float &fjx, float &fjy, float &fjz)
{
    const float fs = pair_fs<RAD, W14>(P, lj, rtab, ti_row, qi, in, r2, qj, tj, is14, acc.elj, acc.ec);
    acc.fx = __fmaf_rn(-fs, dx, acc.fx);
    acc.fy = __fmaf_rn(-fs, dy, acc.fy);
    acc.fz = __fmaf_rn(-fs, dz, acc.fz);
    fjx = __fmaf_rn(fs, dx, fjx);  // F_j = -F_i
    fjy = __fmaf_rn(fs, dy, fjy);
    fjz = __fmaf_rn(fs, dz, fjz);
}

// ---------------------------------------------------------------------------
// Pair export of the debug instantiation: every evaluated pair inside the
// cutoff and not excluded, as caller indices (i < j).
__device__ __forceinline__ void record_pair(const ForceArgs &A, int io, int jo)
{
    atomicAdd((unsigned long long *)&A.dbg_n[0], 1ull);
    const long long q = (long long)atomicAdd((unsigned long long *)&A.dbg_n[1], 1ull);
    if (q < A.dbg_cap) {
        A.dbg_ij[2 * q] = min(io, jo);
        A.dbg_ij[2 * q + 1] = max(io, jo);
    }
}

// Tile fill counters of the debug instantiation: tiles visited (dbg_n[3])
// and tile halves with a pair in range (dbg_n[2]), the halves whose arithmetic
// runs in k_force<G> (k_force1 evaluates both halves of a tile with a pair);
// with the pair count they give the fill of the tiles and of those halves.
__device__ __forceinline__ void count_tile(const ForceArgs &A, bool anyA, bool anyB)
{
    if ((threadIdx.x & 31) == 0) {
        atomicAdd((unsigned long long *)&A.dbg_n[3], 1ull);
        const unsigned long long h = (anyA ? 1ull : 0ull) + (anyB ? 1ull : 0ull);
        if (h) atomicAdd((unsigned long long *)&A.dbg_n[2], h);
    }
}

// Forward kernel (k_force) on i-group tiles.
//
// A work unit is one part of one segment of an i-group's list (the group:
// G consecutive clusters of a column, 8 G atoms).  A warp holds the group's
// atoms in its shared memory and walks the entries; an entry (J, image,
// cluster mask) stands for the tiles (group cluster c, J) of the clusters c
// in its mask.  Lane = ia + 8 jb computes, for every tile, the pairs of i
// atom ia of cluster c with j atoms jb and jb + 4 of J (an 8 x 8 tile, two
// pairs per lane, nothing compacted: pairs beyond the cutoff, excluded pairs
// and padding are evaluated and masked).  J's atoms are read once per entry
// and the force on them is summed over all tiles of the entry in registers,
// then over the 8 lanes of each j atom and added to the global 64-bit
// fixed-point sums (one atomic per atom and component), so the per-entry
// cost (staging, decode, j-force reduction and atomics) is shared by the
// entry's tiles.  The force on i accumulates per lane and cluster in shared
// memory and is summed and added when the unit is done.  J's z-sorted atoms
// form a lower half (jb) and an upper half (jb + 4), which are often not
// both within reach of cluster c: the membership of both pairs comes first
// and the radial arithmetic of a half runs only when one of its 32 pairs is
// in range (warp vote).  Flagged entries carry exclusion bitmasks per tile
// (excluded pairs dropped, 1-4 pairs scaled; the direct self tile's pairs
// j <= i excluded).  The FP32 sums run in a fixed order and meet only in
// integer sums, so results are run-to-run bit-identical.
constexpr int kTileWarps = 8;            // warps per block of the tile kernel
constexpr int kBatch = 16;               // entries staged per batch
#ifndef ACENB_TILE_MIN_BLOCKS
#define ACENB_TILE_MIN_BLOCKS 3          // resident blocks per SM the register budget is cut for
#endif
constexpr float kFarCoord = 3.0e18f;     // i-side padding: far from every atom and from the j-side padding

// Fixed-point value (2^32) of an FP32 sum; a value too large for the sums
// (or not finite) adds zero and sets ovf.
__device__ __forceinline__ long long tile_fixed(float f, bool &ovf)
{
    const bool ok = fabsf(f) < 67108864.0f;
    ovf = ovf || !ok;
    return __float2ll_rn((ok ? f : 0.0f) * 4294967296.0f);
}

// Work units are taken without a claim first: warp w of block b starts with
// unit b + w gridDim (so that few units spread over all SMs), and every further
// unit is claimed from the counter, which counts from the n_first units of the
// first round.  A warp claims its next unit when the current one's entries
// are done, so that the counter's latency hides behind the unit's sums: a
// claim made before the unit ran kept a unit from the idle warps for a whole
// unit's time (13 us at 23,500 atoms), and with fewer units than warps some
// warps ran two units and others none.
__device__ __forceinline__ int claim_unit(const ForceArgs &A, int n_first) { return n_first + atomicAdd(A.work, 1); }

// (Taken on lane 0 and broadcast like a claim: with the index computed on every
// lane the compiler treats it as uniform and the entry loop comes out 12 %
// slower.)
__device__ __forceinline__ int first_unit(int w)
{
    int u = 0;
    if ((threadIdx.x & 31) == 0) u = (int)blockIdx.x + w * (int)gridDim.x;
    return __shfl_sync(kFull, u, 0);
}

// Work unit u of the tile kernels: group, segment of its list, part of the
// segment, and the entry range [e_begin, e_end) of that part.
struct Unit {
    int g, e_begin, e_end;
    long long base;  // first entry of the segment in the group lists
};

__device__ __forceinline__ Unit unit_of(const ForceArgs &A, int u, int parts)
{
    Unit U;
    const int per_g = kListSegs * parts;
    U.g = u / per_g;
    const int r = u - U.g * per_g;
    const int seg = r / parts, part = r - seg * parts;
    const int n = __ldg(A.glist_n + (long long)U.g * kListSegs + seg);
    const int per = (n + parts - 1) / parts;
    U.e_begin = min(n, part * per);
    U.e_end = min(n, U.e_begin + per);
    U.base = (long long)U.g * A.cap + (long long)seg * (A.cap / kListSegs);
    return U;
}

// The exclusion and 1-4 bits of a lane's two pairs (i atom ia, j atoms jb
// and jb + 4) in a flagged tile.
__device__ __forceinline__ void tile_mask_bits(ulonglong2 m, int ia, int jb, bool &inA, bool &inB, bool &s14A,
                                               bool &s14B)
{
    const int bA = ia * kCluster + jb, bB = bA + 4;
    inA = inA && !((m.x >> bA) & 1ull);
    inB = inB && !((m.x >> bB) & 1ull);
    s14A = (m.y >> bA) & 1ull;
    s14B = (m.y >> bB) & 1ull;
}

// One tile (group cluster c, entry J) of a lane: i atom ia of cluster c at
// its image (IMG: x_i - L on axes with code 2), the pairs with the lane's
// j atoms pjA (jb) and pjB (jb + 4), already at their image (code 1 axes).
// SPECIAL: the entry carries exclusion bitmasks (gm).
template <int RAD, bool DEBUG, bool SPECIAL, bool IMG>
__device__ __forceinline__ void tile_pair2(const ForceArgs &A, const float4 *__restrict__ lj, float4 pi, int trow,
                                           int iorig, float4 pjA, float4 pjB, int tjA, int tjB, int jorigA,
                                           int jorigB, uint32_t code, float Lx, float Ly, float Lz, ulonglong2 gm,
                                           int ia, int jb, float4 &fi, float &elj, float &ec, float &fjAx,
                                           float &fjAy, float &fjAz, float &fjBx, float &fjBy, float &fjBz)
{
    if (IMG) {
        if ((code & 3u) == 2u) pi.x = __fsub_rn(pi.x, Lx);
        if (((code >> 2) & 3u) == 2u) pi.y = __fsub_rn(pi.y, Ly);
        if ((code >> 4) == 2u) pi.z = __fsub_rn(pi.z, Lz);
    }
    float dxA, dyA, dzA, dxB, dyB, dzB;
    const float r2A = disp_r2(pjA.x, pjA.y, pjA.z, pi.x, pi.y, pi.z, dxA, dyA, dzA);
    const float r2B = disp_r2(pjB.x, pjB.y, pjB.z, pi.x, pi.y, pi.z, dxB, dyB, dzB);
    bool inA = r2A < A.P.rc2, inB = r2B < A.P.rc2;
    bool s14A = false, s14B = false;
    if (SPECIAL) tile_mask_bits(gm, ia, jb, inA, inB, s14A, s14B);
    const bool anyA = __any_sync(kFull, inA), anyB = __any_sync(kFull, inB);
    if (DEBUG) count_tile(A, anyA, anyB);
    if (!anyA && !anyB) return;
    Acc acc = {fi.x, fi.y, fi.z, elj, ec};
    if (anyA) {
        if (DEBUG && inA) record_pair(A, iorig, jorigA);
        // only a special (flagged) tile can hold r2 = 0 (the self tile's diagonal, masked)
        eval_pair<RAD, SPECIAL>(A.P, lj, A.rtab, trow, pi.w, inA, dxA, dyA, dzA, SPECIAL ? (inA ? r2A : 1.0f) : r2A,
                                pjA.w, tjA, s14A, acc, fjAx, fjAy, fjAz);
    }
    if (anyB) {
        if (DEBUG && inB) record_pair(A, iorig, jorigB);
        eval_pair<RAD, SPECIAL>(A.P, lj, A.rtab, trow, pi.w, inB, dxB, dyB, dzB, SPECIAL ? (inB ? r2B : 1.0f) : r2B,
                                pjB.w, tjB, s14B, acc, fjBx, fjBy, fjBz);
    }
    fi = make_float4(acc.fx, acc.fy, acc.fz, 0.0f);
    elj = acc.elj;
    ec = acc.ec;
}

// One entry: J's atoms for the lane (jb, jb + 4) from the staged batch, the
// tiles of every group cluster in its mask, then the force on J's atoms.
template <int G, int RAD, bool VIRIAL, bool DEBUG, bool SPECIAL, bool IMG>
__device__ __forceinline__ void tile_entry(const ForceArgs &A, const float4 *__restrict__ lj,
                                           const float4 *__restrict__ s_ix, const int *__restrict__ s_it,
                                           const int *__restrict__ s_io, float4 *__restrict__ s_fi,
                                           const ulonglong2 *own8, uint2 ent, float4 pjA, float4 pjB, int tjA, int tjB, int ia, int jb, int lane, float Lx,
                                           float Ly, float Lz, float &elj, float &ec, float (&wimg)[6], bool &ovf)
{
    const int J = (int)(ent.x & kJMask);
    const uint32_t code = IMG ? (ent.x >> kShiftBit) & 0x3Fu : 0u;
    if (IMG) {  // j-side images (code 1): fl(x_j - L), as the other kernels stage them
        if ((code & 3u) == 1u) { pjA.x = __fsub_rn(pjA.x, Lx); pjB.x = __fsub_rn(pjB.x, Lx); }
        if (((code >> 2) & 3u) == 1u) { pjA.y = __fsub_rn(pjA.y, Ly); pjB.y = __fsub_rn(pjB.y, Ly); }
        if ((code >> 4) == 1u) { pjA.z = __fsub_rn(pjA.z, Lz); pjB.z = __fsub_rn(pjB.z, Lz); }
    }
    const int jorigA = DEBUG ? __ldg(A.perm + (long long)J * kCluster + jb) : -1;
    const int jorigB = DEBUG ? __ldg(A.perm + (long long)J * kCluster + jb + 4) : -1;
    const ulonglong2 *rec = SPECIAL ? entry_record<G>(A, ent.y, own8) : nullptr;
    float fjAx = 0.0f, fjAy = 0.0f, fjAz = 0.0f, fjBx = 0.0f, fjBy = 0.0f, fjBz = 0.0f;
    for (unsigned cm = ent.y & ((1u << mask_bit(G)) - 1u); cm; cm &= cm - 1u) {
        const int c = __ffs(cm) - 1;
        const int ii = c * kCluster + ia;
        const ulonglong2 gm = SPECIAL ? rec[c] : make_ulonglong2(0ull, 0ull);
        float4 fi = s_fi[c * 32 + lane];
        tile_pair2<RAD, DEBUG, SPECIAL, IMG>(A, lj, s_ix[ii], s_it[ii], DEBUG ? s_io[ii] : -1, pjA, pjB, tjA, tjB,
                                             jorigA, jorigB, code, Lx, Ly, Lz, gm, ia, jb, fi, elj, ec, fjAx, fjAy,
                                             fjAz, fjBx, fjBy, fjBz);
        s_fi[c * 32 + lane] = fi;
    }
    // the force on J's atoms: sum over the 8 lanes of each (lanes ia), then
    // lanes ia = 0, 1, 2 add atom jb's x, y, z and ia = 3, 4, 5 atom jb + 4's
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        fjAx = __fadd_rn(fjAx, __shfl_xor_sync(kFull, fjAx, o));
        fjAy = __fadd_rn(fjAy, __shfl_xor_sync(kFull, fjAy, o));
        fjAz = __fadd_rn(fjAz, __shfl_xor_sync(kFull, fjAz, o));
        fjBx = __fadd_rn(fjBx, __shfl_xor_sync(kFull, fjBx, o));
        fjBy = __fadd_rn(fjBy, __shfl_xor_sync(kFull, fjBy, o));
        fjBz = __fadd_rn(fjBz, __shfl_xor_sync(kFull, fjBz, o));
    }
    const float fv = ia == 0 ? fjAx : ia == 1 ? fjAy : ia == 2 ? fjAz : ia == 3 ? fjBx : ia == 4 ? fjBy : fjBz;
    const long long fx = tile_fixed(fv, ovf);  // every lane (ia = 6, 7 hold z of B again): no branch
    if (ia < 6 && fx != 0) {
        const int j = ia < 3 ? jb : jb + 4;
        atomicAdd((unsigned long long *)&A.facc[24ll * J + 3 * j + (ia < 3 ? ia : ia - 3)], (unsigned long long)fx);
    }
    if (VIRIAL && IMG && ia == 0) {
        // periodic-image part of the virial: s (x) f_j with the entry's
        // shift s of j (code 1: -L, code 2: +L per axis)
        const uint32_t cx = code & 3u, cy = (code >> 2) & 3u, cz = code >> 4;
        const float sx = cx == 1u ? -Lx : (cx == 2u ? Lx : 0.0f);
        const float sy = cy == 1u ? -Ly : (cy == 2u ? Ly : 0.0f);
        const float sz = cz == 1u ? -Lz : (cz == 2u ? Lz : 0.0f);
        const float gx = __fadd_rn(fjAx, fjBx), gy = __fadd_rn(fjAy, fjBy), gz = __fadd_rn(fjAz, fjBz);
        wimg[0] = __fmaf_rn(sx, gx, wimg[0]);
        wimg[1] = __fmaf_rn(sy, gy, wimg[1]);
        wimg[2] = __fmaf_rn(sz, gz, wimg[2]);
        wimg[3] = __fmaf_rn(sx, gy, wimg[3]);
        wimg[4] = __fmaf_rn(sx, gz, wimg[4]);
        wimg[5] = __fmaf_rn(sy, gz, wimg[5]);
    }
}

// The image virial of a work unit (FP32 per lane) to the warp's fixed-point
// sums (2^20): lane k < 6 holds component k in wv.  Rounded per unit, so the
// sums do not depend on which warp took which unit.
__device__ __forceinline__ void tile_virial_unit(float (&wimg)[6], long long &wv, int lane)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        long long x = __float2ll_rn(wimg[k] * (float)kVirScale);
        wimg[k] = 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == k) wv += x;
    }
}

// Warp sums of a system's energies (2^32) and image virial (2^20); clears
// the per-lane sums.
template <bool VIRIAL>
__device__ __forceinline__ void tile_warp_sums(long long (&e)[2], long long &wv, long long (&out)[kTaskVals])
{
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        long long x = e[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        out[k] = x;
    }
    if (VIRIAL)
#pragma unroll
        for (int k = 0; k < 6; ++k) out[2 + k] = __shfl_sync(kFull, wv, k);
    e[0] = e[1] = 0;
    wv = 0;
}

// Bytes of the forward kernels' LJ table: (A, B, 12 A, 6 B) and (A, B)
// remainders per type pair, rounded up to 16.
__host__ __device__ inline size_t lj_table_bytes(int T) { return align16((size_t)T * T * 24); }

// Shared memory of the forward kernel: the type-pair table (A, B, 12 A, 6 B)
// and per warp the unit's i atoms (coordinates + ke q, type row, caller
// index), the lanes' i-force partials per cluster, and one staged batch of
// entries' j atoms (coordinates + charge, type).
__host__ __device__ inline size_t tile_warp_bytes(int G)
{
    return (size_t)kCluster * G * (16 + 4 + 4) + (size_t)G * 32 * 16 + (size_t)kBatch * kCluster * (16 + 4);
}

template <int G, int RAD, bool VIRIAL, bool DEBUG>
__global__ void __launch_bounds__(kTileWarps * 32, ACENB_TILE_MIN_BLOCKS) k_force(ForceArgs A, int parts, int n_first)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_val[kTileWarps][kTaskVals];
    __shared__ int s_sys[kTileWarps];
    const int T = A.P.n_types;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, ia = lane & 7, jb = lane >> 3;
    float4 *lj = reinterpret_cast<float4 *>(smem);  // (A, B, 12 A, 6 B) per type pair
    unsigned char *wbase = smem + lj_table_bytes(T) + (size_t)w * tile_warp_bytes(G);
    float4 *s_ix = reinterpret_cast<float4 *>(wbase);                          // [8 G]
    float4 *s_fi = s_ix + kCluster * G;                                          // [G * 32]
    float4 *sjp = s_fi + G * 32;                                                 // [kBatch * 8]
    int *s_it = reinterpret_cast<int *>(sjp + kBatch * kCluster);                // [8 G]
    int *s_io = s_it + kCluster * G;                                             // [8 G]
    int *sjt = s_io + kCluster * G;                                              // [kBatch * 8]
    for (int k = threadIdx.x; k < T * T; k += blockDim.x) {
        const float4 ab = A.lj_tab[k];
        lj[k] = make_float4(ab.x, ab.y, 12.0f * ab.x, 6.0f * ab.y);
        reinterpret_cast<float2 *>(lj + T * T)[k] = make_float2(ab.z, ab.w);
    }
    pdl_entry();  // the type-pair tables do not depend on the preceding kernels
    __syncthreads();
    const int n_units = A.counts[4] * kListSegs * parts;
    int cur_sys = -1;
    float Lx = 0.0f, Ly = 0.0f, Lz = 0.0f;
    long long esum[2] = {0, 0};  // per lane: fixed-point energies of the current system
    float wimg[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};  // image virial of the current unit
    long long wv = 0;  // lane k < 6: fixed-point image virial component k of the current system
    bool ovf = false;  // a force sum out of the fixed-point range
    int u = first_unit(w);
    while (u < n_units) {
        const Unit U = unit_of(A, u, parts);
        int u_next = 0;
        if (U.e_begin < U.e_end) {
            const int2 gr = __ldg(A.grp + U.g);
            const int c0 = gr.x, ncl = gr.y;
            const ulonglong2 *own8 = G == 8 ? A.gmask + (long long)c0 * kMaskRecsPerCluster * 8 : nullptr;
            const int sys_id = __ldg(A.clus_sys + c0);
            if (sys_id != cur_sys) {
                if (!DEBUG && cur_sys >= 0) {
                    long long v[kTaskVals];
                    tile_warp_sums<VIRIAL>(esum, wv, v);
                    if (lane == 0)
                        for (int k = 0; k < (VIRIAL ? kTaskVals : 2); ++k)
                            if (v[k]) atomicAdd((unsigned long long *)&A.sys_acc[cur_sys * kTaskVals + k], (unsigned long long)v[k]);
                }
                cur_sys = sys_id;
                Lx = A.sys[sys_id].L[0];
                Ly = A.sys[sys_id].L[1];
                Lz = A.sys[sys_id].L[2];
            }
            // the group's atoms (padding slots and absent clusters far away)
            for (int t = lane; t < kCluster * G; t += 32) {
                const long long slot = (long long)c0 * kCluster + t;
                float4 p = make_float4(kFarCoord, kFarCoord, kFarCoord, 0.0f);
                int tr = 0, orig = -1;
                if (t < kCluster * ncl) {
                    p = __ldg(A.xyzq + slot);
                    if (!is_real_coord(p.x)) p.x = p.y = p.z = kFarCoord;
                    p.w *= A.P.ke;
                    tr = __ldg(A.tslot + slot) * T;
                    orig = DEBUG ? __ldg(A.perm + slot) : -1;
                }
                s_ix[t] = p;
                s_it[t] = tr;
                s_io[t] = orig;
            }
#pragma unroll
            for (int c = 0; c < G; ++c) s_fi[c * 32 + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            __syncwarp();
            float elj = 0.0f, ec = 0.0f;
            const uint2 *row = A.glist + U.base;
            bool unit_img = false;  // the unit holds an image entry (warp uniform)
            for (int e0 = U.e_begin; e0 < U.e_end; e0 += kBatch) {
                const int ne = min(kBatch, U.e_end - e0);
                const uint2 my = lane < ne ? __ldg(row + e0 + lane) : make_uint2(0u, 0u);
                // stage the batch's j atoms: lane k copies the 8 coordinates
                // and types of entry k (atom a at swz(k, a))
                if (lane < ne) {
                    const long long jbase = (long long)(my.x & kJMask) * kCluster;
#pragma unroll
                    for (int a = 0; a < kCluster; ++a) {
                        cp_async16(sjp + swz(lane, a), A.xyzq + jbase + a);
                        cp_async4(sjt + swz(lane, a), A.tslot + jbase + a);
                    }
                }
                cp_async_wait_all();
                __syncwarp();
                // the batch's plain entries first (no image code, no masks:
                // one code path without a dispatch), then the others
                const bool my_img = ((my.x >> kShiftBit) & 0x3Fu) != 0u;
                const bool my_spc = (my.x & kExclFlag) != 0u;
                const bool in_batch = lane < ne;
                unsigned plain = __ballot_sync(kFull, in_batch && !my_img && !my_spc);
                unsigned other = __ballot_sync(kFull, in_batch) & ~plain;
                unit_img = unit_img || __ballot_sync(kFull, in_batch && my_img) != 0u;
                while (plain) {
                    const int k = __ffs(plain) - 1;
                    plain &= plain - 1u;
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    tile_entry<G, RAD, VIRIAL, DEBUG, false, false>(
                        A, lj, s_ix, s_it, s_io, s_fi, own8, ent, sjp[swz(k, jb)], sjp[swz(k, jb + 4)], sjt[swz(k, jb)],
                        sjt[swz(k, jb + 4)], ia, jb, lane, Lx, Ly, Lz, elj, ec, wimg, ovf);
                }
                while (other) {
                    const int k = __ffs(other) - 1;
                    other &= other - 1u;
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    const float4 pjA = sjp[swz(k, jb)], pjB = sjp[swz(k, jb + 4)];
                    const int tjA = sjt[swz(k, jb)], tjB = sjt[swz(k, jb + 4)];
                    const bool img = ((ent.x >> kShiftBit) & 0x3Fu) != 0u;
                    const bool special = (ent.x & kExclFlag) != 0u;
                    if (img) {
                        if (special)
                            tile_entry<G, RAD, VIRIAL, DEBUG, true, true>(A, lj, s_ix, s_it, s_io, s_fi, own8, ent, pjA,
                                                                         pjB, tjA, tjB, ia, jb, lane, Lx, Ly, Lz, elj, ec,
                                                                         wimg, ovf);
                        else
                            tile_entry<G, RAD, VIRIAL, DEBUG, false, true>(A, lj, s_ix, s_it, s_io, s_fi, own8, ent,
                                                                          pjA, pjB, tjA, tjB, ia, jb, lane, Lx, Ly, Lz, elj,
                                                                          ec, wimg, ovf);
                    } else {
                        tile_entry<G, RAD, VIRIAL, DEBUG, true, false>(A, lj, s_ix, s_it, s_io, s_fi, own8, ent, pjA,
                                                                      pjB, tjA, tjB, ia, jb, lane, Lx, Ly, Lz, elj, ec, wimg,
                                                                      ovf);
                    }
                }
                __syncwarp();  // the staging buffer is rewritten by the next batch
            }
            if (lane == 0) u_next = claim_unit(A, n_first);
            // force on the group's atoms: each lane's partials summed over the
            // 4 lanes of the same atom (jb) in FP32 (a fixed butterfly: every
            // lane ends with the same bits), then lane jb adds clusters c with
            // c % 4 == jb in fixed point
#pragma unroll
            for (int c = 0; c < G; ++c) {
                float4 f = s_fi[c * 32 + lane];
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    f.x = __fadd_rn(f.x, __shfl_xor_sync(kFull, f.x, o));
                    f.y = __fadd_rn(f.y, __shfl_xor_sync(kFull, f.y, o));
                    f.z = __fadd_rn(f.z, __shfl_xor_sync(kFull, f.z, o));
                }
                if ((c & 3) == jb && c < ncl) {
                    const long long slot = (long long)c0 * kCluster + c * kCluster + ia;
                    const long long fx = tile_fixed(f.x, ovf), fy = tile_fixed(f.y, ovf), fz = tile_fixed(f.z, ovf);
                    if (fx) atomicAdd((unsigned long long *)&A.facc[3 * slot], (unsigned long long)fx);
                    if (fy) atomicAdd((unsigned long long *)&A.facc[3 * slot + 1], (unsigned long long)fy);
                    if (fz) atomicAdd((unsigned long long *)&A.facc[3 * slot + 2], (unsigned long long)fz);
                }
            }
            esum[0] += tile_fixed(elj, ovf);
            esum[1] += tile_fixed(ec, ovf);
            if (VIRIAL && unit_img) tile_virial_unit(wimg, wv, lane);  // image entries only add to wimg
            if (__any_sync(kFull, ovf)) {
                if (lane == 0) atomicOr(A.status, ST_OVERFLOW);
                ovf = false;
            }
            __syncwarp();  // the i atoms and partials are rewritten by the next unit
        } else if (lane == 0) {
            u_next = claim_unit(A, n_first);
        }
        u = __shfl_sync(kFull, u_next, 0);
    }
    if (DEBUG) return;
    // the block's sums: one atomic per value for the system most warps
    // ended in, direct atomics for any other
    long long v[kTaskVals];
    tile_warp_sums<VIRIAL>(esum, wv, v);
    if (lane == 0) {
        s_sys[w] = cur_sys;
        for (int k = 0; k < kTaskVals; ++k) s_val[w][k] = k < (VIRIAL ? kTaskVals : 2) ? v[k] : 0;
    }
    __syncthreads();
    if (threadIdx.x < (VIRIAL ? kTaskVals : 2)) {
        const int k = threadIdx.x;
        const int nw = blockDim.x >> 5;
        int base = -1;
        long long sum = 0;
        for (int q = 0; q < nw; ++q) {
            const int sq = s_sys[q];
            if (sq < 0) continue;
            if (base < 0) base = sq;
            if (sq == base) sum += s_val[q][k];
            else if (s_val[q][k]) atomicAdd((unsigned long long *)&A.sys_acc[sq * kTaskVals + k], (unsigned long long)s_val[q][k]);
        }
        if (base >= 0 && sum) atomicAdd((unsigned long long *)&A.sys_acc[base * kTaskVals + k], (unsigned long long)sum);
    }
}

// ---------------------------------------------------------------------------
// Forward kernel for i-groups of one cluster (k_force1): the lists are the
// same, each entry holds one tile (I, J).  Lane = jj + 8 ih holds j atom jj
// of J and the i atoms ih and ih + 4 of I in registers, so every lane
// computes two pairs of the 8 x 8 tile and the force on j is summed over only
// 4 lanes.  With one cluster per group the per-entry work is per tile, but
// the i side needs no shared memory and the j-force sum is short; which of
// this and the group kernel is faster depends on the system (the autotuner
// measures it).
//
// The kernel is bound by instruction issue and register reads, not by the
// FMA pipe (about half busy), so the two pairs of a lane share one
// instruction: i atom ih in the low word and ih + 4 in the high word of
// packed FP32 operations (pair_radial2), which round like the scalar ones.
// A tile with a pair in range is evaluated whole; voting on its two halves
// and skipping one (scalar code, 1.35 halves per tile) took 47.9 M warp
// instructions and 63.4 us per launch at 23,500 atoms and 1,661 us at
// 999,999; packed it was 40.3 M, 60.8 us and 1,621 us, and with the unit claims
// and block shapes below it is 39.7 M, 57.0 us and 1,569 us.  (An FMA with three
// register operands, packed or not, issues at about 0.6 of its rate for the
// register reads: the constants of the polynomials come from the parameter
// bank and run at the full rate.)
constexpr int kBatch1 = 32;  // entries staged per batch (one per lane)

// The i cluster of a work unit for one lane: its atoms ih (low words) and
// ih + 4 (high words).
struct TileI2 {
    f32x2 x, y, z, q;  // q: ke q
    int trowA, trowB;  // type rows
    int origA, origB;  // caller indices (pair export)
};

__device__ __forceinline__ TileI2 load_tile_i2(const ForceArgs &A, long long slot, int T, bool debug)
{
    float4 p[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        p[k] = __ldg(A.xyzq + slot + 4 * k);
        if (!is_real_coord(p[k].x)) p[k].x = p[k].y = p[k].z = kFarCoord;
    }
    TileI2 t;
    t.x = pack2(p[0].x, p[1].x);
    t.y = pack2(p[0].y, p[1].y);
    t.z = pack2(p[0].z, p[1].z);
    t.q = pack2(p[0].w * A.P.ke, p[1].w * A.P.ke);
    t.trowA = __ldg(A.tslot + slot) * T;
    t.trowB = __ldg(A.tslot + slot + 4) * T;
    t.origA = debug ? __ldg(A.perm + slot) : -1;
    t.origB = debug ? __ldg(A.perm + slot + 4) : -1;
    return t;
}

// Sums of a lane's two pairs over a work unit: the force on the i atoms and
// the energies.
struct Acc2 {
    f32x2 fx, fy, fz, elj, ec;
};

// v where the lane's pair is inside the cutoff, else 0.
__device__ __forceinline__ f32x2 masked2(f32x2 v, bool inA, bool inB)
{
    float a, b;
    unpack2(v, a, b);
    return pack2(inA ? a : 0.0f, inB ? b : 0.0f);
}

// Both pairs of a lane: -U'(r)/r of each (0 where masked), the energies added
// to acc (the packed pair_fs).
template <int RAD, bool W14>
__device__ __forceinline__ f32x2 pair_fs2(const ForceArgs &A, const float4 *__restrict__ lj, const TileI2 &ti, bool inA,
                                          bool inB, f32x2 r2, f32x2 qj, int tj, bool s14A, bool s14B, Acc2 &acc)
{
    if constexpr (RAD == 2) {
        // the tables' loads, not arithmetic, bound this: scalar, and a half
        // without a pair in range is skipped
        float ra, rb, qa, qb, qjv, el[2], ec[2], fs[2] = {0.0f, 0.0f};
        unpack2(r2, ra, rb);
        unpack2(ti.q, qa, qb);
        unpack2(qj, qjv, qjv);
        unpack2(acc.elj, el[0], el[1]);
        unpack2(acc.ec, ec[0], ec[1]);
        if (__any_sync(kFull, inA))
            fs[0] = pair_fs<2, W14>(A.P, lj, A.rtab, ti.trowA, qa, inA, ra, qjv, tj, s14A, el[0], ec[0]);
        if (__any_sync(kFull, inB))
            fs[1] = pair_fs<2, W14>(A.P, lj, A.rtab, ti.trowB, qb, inB, rb, qjv, tj, s14B, el[1], ec[1]);
        acc.elj = pack2(el[0], el[1]);
        acc.ec = pack2(ec[0], ec[1]);
        return pack2(fs[0], fs[1]);
    } else {
        const float2 *lj_lo = reinterpret_cast<const float2 *>(lj + A.P.n_types * A.P.n_types);
        const int kA = ti.trowA + tj, kB = ti.trowB + tj;
        f32x2 elj, frlj, ec, frc, r2inv;
        pair_radial2<RAD == 1>(A.C, A.P, r2, lj[kA], lj_lo[kA], lj[kB], lj_lo[kB], mul2(ti.q, qj), elj, frlj, ec, frc,
                               r2inv);
        f32x2 fs;
        if (W14) {
            const f32x2 wlj = pack2(s14A ? A.P.s14_lj : 1.0f, s14B ? A.P.s14_lj : 1.0f);
            const f32x2 wc = pack2(s14A ? A.P.s14_c : 1.0f, s14B ? A.P.s14_c : 1.0f);
            fs = mul2(fma2(wlj, frlj, mul2(wc, frc)), r2inv);
            elj = mul2(wlj, elj);
            ec = mul2(wc, ec);
        } else {
            fs = mul2(add2(frlj, frc), r2inv);
        }
        acc.elj = add2(acc.elj, masked2(elj, inA, inB));
        acc.ec = add2(acc.ec, masked2(ec, inA, inB));
        return masked2(fs, inA, inB);
    }
}

// One entry (tile (I, J)) of a warp: the membership of the lane's two pairs,
// their arithmetic packed (when any pair of the tile is in range), the force
// on i added to acc, and the force on j summed over its 4 lanes.
template <int RAD, bool VIRIAL, bool DEBUG, bool SPECIAL, bool IMG>
__device__ __forceinline__ void tile1_entry(const ForceArgs &A, const float4 *__restrict__ lj, uint2 ent, float4 pj,
                                            int tj, const TileI2 &ti, int jj, int ih, float Lx, float Ly, float Lz,
                                            Acc2 &acc, float (&wimg)[3], bool &ovf)
{
    const int J = (int)(ent.x & kJMask);
    const uint32_t code = IMG ? (ent.x >> kShiftBit) & 0x3Fu : 0u;
    f32x2 ix = ti.x, iy = ti.y, iz = ti.z;
    if (IMG) {  // code 1: fl(x_j - L) on the j side, code 2: fl(x_i - L) on the i side
        if ((code & 3u) == 1u) pj.x = __fsub_rn(pj.x, Lx);
        if (((code >> 2) & 3u) == 1u) pj.y = __fsub_rn(pj.y, Ly);
        if ((code >> 4) == 1u) pj.z = __fsub_rn(pj.z, Lz);
        if ((code & 3u) == 2u) ix = sub2(ix, pack2(Lx, Lx));
        if (((code >> 2) & 3u) == 2u) iy = sub2(iy, pack2(Ly, Ly));
        if ((code >> 4) == 2u) iz = sub2(iz, pack2(Lz, Lz));
    }
    // e = x_i - x_j = -d; r2 as disp_r2
    const f32x2 ex = sub2(ix, pack2(pj.x, pj.x)), ey = sub2(iy, pack2(pj.y, pj.y)), ez = sub2(iz, pack2(pj.z, pj.z));
    f32x2 r2 = fma2(ez, ez, fma2(ey, ey, mul2(ex, ex)));
    float r2A, r2B;
    unpack2(r2, r2A, r2B);
    bool inA = r2A < A.P.rc2, inB = r2B < A.P.rc2;
    bool s14A = false, s14B = false;
    if (SPECIAL) {  // exclusion bitmask of the tile: bit 8 i + j
        const ulonglong2 m = A.gmask[ent.y >> mask_bit(1)];  // records of one cluster
        const int bA = ih * kCluster + jj, bB = bA + 4 * kCluster;
        inA = inA && !((m.x >> bA) & 1ull);
        inB = inB && !((m.x >> bB) & 1ull);
        s14A = (m.y >> bA) & 1ull;
        s14B = (m.y >> bB) & 1ull;
        // only a flagged tile can hold r2 = 0 (the self tile's diagonal, masked)
        r2 = pack2(inA ? r2A : 1.0f, inB ? r2B : 1.0f);
    }
    if (DEBUG) count_tile(A, __any_sync(kFull, inA), __any_sync(kFull, inB));
    if (!__any_sync(kFull, inA || inB)) return;
    if (DEBUG) {
        const int jorig = __ldg(A.perm + (long long)J * kCluster + jj);
        if (inA) record_pair(A, ti.origA, jorig);
        if (inB) record_pair(A, ti.origB, jorig);
    }
    const f32x2 fs = pair_fs2<RAD, SPECIAL>(A, lj, ti, inA, inB, r2, pack2(pj.w, pj.w), tj, s14A, s14B, acc);
    acc.fx = fma2(fs, ex, acc.fx);  // F_i = fs e
    acc.fy = fma2(fs, ey, acc.fy);
    acc.fz = fma2(fs, ez, acc.fz);
    // F_j = -fs e: both pairs, then the 4 lanes of j atom jj (ih = 0..3) as
    // (0 + 1) + (2 + 3).  The lanes trade components instead of all summing
    // all three: lanes ih = 0, 1, 2 end with x, y, z (ih = 3 with y again).
    float fA, fB, e0, e1, fj[3];
    unpack2(fs, fA, fB);
    unpack2(ex, e0, e1);
    fj[0] = __fmaf_rn(fB, -e1, __fmul_rn(fA, -e0));
    unpack2(ey, e0, e1);
    fj[1] = __fmaf_rn(fB, -e1, __fmul_rn(fA, -e0));
    unpack2(ez, e0, e1);
    fj[2] = __fmaf_rn(fB, -e1, __fmul_rn(fA, -e0));
    const bool odd = ih & 1, upper = ih & 2;
    const float xy = __fadd_rn(odd ? fj[1] : fj[0], __shfl_xor_sync(kFull, odd ? fj[0] : fj[1], 8));
    const float zz = __fadd_rn(fj[2], __shfl_xor_sync(kFull, fj[2], 8));
    const bool take_z = upper && !odd;
    const float fc = __fadd_rn(take_z ? zz : xy, __shfl_xor_sync(kFull, odd || upper ? xy : zz, 16));
    const long long fv = tile_fixed(fc, ovf);  // every lane: no branch
    if (ih < 3) atomicAdd((unsigned long long *)&A.facc[24ll * J + 3 * jj + ih], (unsigned long long)fv);
    if (VIRIAL && IMG) {
        // periodic-image part of the virial, s (x) f_j with the entry's shift
        // s of j: lane ih < 3 holds s_x, s_y, s_z times component ih
        const uint32_t cx = code & 3u, cy = (code >> 2) & 3u, cz = code >> 4;
        const float sx = cx == 1u ? -Lx : (cx == 2u ? Lx : 0.0f);
        const float sy = cy == 1u ? -Ly : (cy == 2u ? Ly : 0.0f);
        const float sz = cz == 1u ? -Lz : (cz == 2u ? Lz : 0.0f);
        wimg[0] = __fmaf_rn(sx, fc, wimg[0]);
        wimg[1] = __fmaf_rn(sy, fc, wimg[1]);
        wimg[2] = __fmaf_rn(sz, fc, wimg[2]);
    }
}

// The image virial of a work unit (FP32 per lane, see tile1_entry) to the
// warp's fixed-point sums (2^20): lane k < 6 holds component k (xx, yy, zz,
// xy, xz, yz) in wv.  Rounded per lane and unit, so the sums do not depend on
// which warp took which unit.
__device__ __forceinline__ void tile1_virial_unit(float (&wimg)[3], long long &wv, int lane)
{
    const int ih = lane >> 3;
    // the component of s and of f (its lane ih) of each virial component
    constexpr int ks[6] = {0, 1, 2, 0, 0, 1}, kf[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        long long x = ih == kf[k] ? __float2ll_rn(wimg[ks[k]] * (float)kVirScale) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == k) wv += x;
    }
    wimg[0] = wimg[1] = wimg[2] = 0.0f;
}

__host__ __device__ inline size_t tile1_warp_bytes() { return (size_t)kBatch1 * kCluster * (16 + 4); }

template <int W, int MB, int RAD, bool VIRIAL, bool DEBUG>
__global__ void __launch_bounds__(W * 32, MB) k_force1(ForceArgs A, int parts,
                                                                                        int n_first)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_val[W][kTaskVals];
    __shared__ int s_sys[W];
    const int T = A.P.n_types;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, jj = lane & 7, ih = lane >> 3;
    float4 *lj = reinterpret_cast<float4 *>(smem);  // (A, B, 12 A, 6 B) per type pair
    float4 *sjp = reinterpret_cast<float4 *>(smem + lj_table_bytes(T) + (size_t)w * tile1_warp_bytes());
    int *sjt = reinterpret_cast<int *>(sjp + kBatch1 * kCluster);
    for (int k = threadIdx.x; k < T * T; k += blockDim.x) {
        const float4 ab = A.lj_tab[k];
        lj[k] = make_float4(ab.x, ab.y, 12.0f * ab.x, 6.0f * ab.y);
        reinterpret_cast<float2 *>(lj + T * T)[k] = make_float2(ab.z, ab.w);
    }
    pdl_entry();  // the type-pair tables do not depend on the preceding kernels
    __syncthreads();
    const int n_units = A.counts[4] * kListSegs * parts;
    int cur_sys = -1;
    float Lx = 0.0f, Ly = 0.0f, Lz = 0.0f;
    long long esum[2] = {0, 0};
    float wimg[3] = {0.0f, 0.0f, 0.0f};
    long long wv = 0;
    bool ovf = false;
    int u = first_unit(w);
    while (u < n_units) {
        const Unit U = unit_of(A, u, parts);
        // what needs only the unit's group and segment is loaded before the
        // segment's length is known: one-cluster groups are numbered like
        // their clusters, and a segment holds at least its first batch
        const int I = U.g;
        const int sys_id = __ldg(A.clus_sys + I);
        const long long s0 = (long long)I * kCluster;
        const TileI2 ti = load_tile_i2(A, s0 + ih, T, DEBUG);
        const uint2 *row = A.glist + U.base;
        const uint2 first = lane < A.cap / kListSegs ? __ldg(row + lane) : make_uint2(0u, 0u);
        int u_next = 0;
        if (U.e_begin < U.e_end) {
            if (sys_id != cur_sys) {
                if (!DEBUG && cur_sys >= 0) {
                    long long v[kTaskVals];
                    tile_warp_sums<VIRIAL>(esum, wv, v);
                    if (lane == 0)
                        for (int k = 0; k < (VIRIAL ? kTaskVals : 2); ++k)
                            if (v[k]) atomicAdd((unsigned long long *)&A.sys_acc[cur_sys * kTaskVals + k], (unsigned long long)v[k]);
                }
                cur_sys = sys_id;
                Lx = A.sys[sys_id].L[0];
                Ly = A.sys[sys_id].L[1];
                Lz = A.sys[sys_id].L[2];
            }
            Acc2 acc = {0ull, 0ull, 0ull, 0ull, 0ull};
            bool unit_img = false;
            for (int e0 = U.e_begin; e0 < U.e_end; e0 += kBatch1) {
                const int ne = min(kBatch1, U.e_end - e0);
                const uint2 my = lane < ne ? (e0 == 0 ? first : __ldg(row + e0 + lane)) : make_uint2(0u, 0u);
                if (lane < ne) {
                    const long long jbase = (long long)(my.x & kJMask) * kCluster;
#pragma unroll
                    for (int a = 0; a < kCluster; ++a) {
                        cp_async16(sjp + swz(lane, a), A.xyzq + jbase + a);
                        cp_async4(sjt + swz(lane, a), A.tslot + jbase + a);
                    }
                }
                cp_async_wait_all();
                __syncwarp();
                const bool my_img = ((my.x >> kShiftBit) & 0x3Fu) != 0u;
                const bool my_spc = (my.x & kExclFlag) != 0u;
                const bool in_batch = lane < ne;
                unsigned plain = __ballot_sync(kFull, in_batch && !my_img && !my_spc);
                unsigned other = __ballot_sync(kFull, in_batch) & ~plain;
                unit_img = unit_img || __ballot_sync(kFull, in_batch && my_img) != 0u;
                while (plain) {
                    const int k = __ffs(plain) - 1;
                    plain &= plain - 1u;
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    tile1_entry<RAD, VIRIAL, DEBUG, false, false>(A, lj, ent, sjp[swz(k, jj)], sjt[swz(k, jj)], ti, jj, ih, Lx, Ly, Lz, acc, wimg, ovf);
                }
                while (other) {
                    const int k = __ffs(other) - 1;
                    other &= other - 1u;
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    const float4 pj = sjp[swz(k, jj)];
                    const int tj = sjt[swz(k, jj)];
                    const bool img = ((ent.x >> kShiftBit) & 0x3Fu) != 0u;
                    const bool special = (ent.x & kExclFlag) != 0u;
                    if (img) {
                        if (special)
                            tile1_entry<RAD, VIRIAL, DEBUG, true, true>(A, lj, ent, pj, tj, ti, jj, ih, Lx, Ly, Lz, acc, wimg, ovf);
                        else
                            tile1_entry<RAD, VIRIAL, DEBUG, false, true>(A, lj, ent, pj, tj, ti, jj, ih, Lx, Ly, Lz, acc, wimg, ovf);
                    } else {
                        tile1_entry<RAD, VIRIAL, DEBUG, true, false>(A, lj, ent, pj, tj, ti, jj, ih, Lx, Ly, Lz, acc, wimg, ovf);
                    }
                }
                __syncwarp();  // the staging buffer is rewritten by the next batch
            }
            if (lane == 0) u_next = claim_unit(A, n_first);
            // force on the i atoms: the 8 lanes of each atom summed in FP32
            // (a fixed butterfly), then lanes jj < 3 add atom ih, jj = 3..5
            // atom ih + 4 in fixed point
            float v[6];
            unpack2(acc.fx, v[0], v[3]);
            unpack2(acc.fy, v[1], v[4]);
            unpack2(acc.fz, v[2], v[5]);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int c = 0; c < 6; ++c) v[c] = __fadd_rn(v[c], __shfl_xor_sync(kFull, v[c], o));
            float mine = v[0];
#pragma unroll
            for (int c = 1; c < 6; ++c) mine = jj == c ? v[c] : mine;
            const long long fi = tile_fixed(mine, ovf);
            if (jj < 6 && fi != 0) {
                const long long slot = s0 + ih + (jj < 3 ? 0 : 4);
                atomicAdd((unsigned long long *)&A.facc[3 * slot + (jj < 3 ? jj : jj - 3)], (unsigned long long)fi);
            }
            float eA, eB;
            unpack2(acc.elj, eA, eB);
            esum[0] += tile_fixed(eA, ovf) + tile_fixed(eB, ovf);
            unpack2(acc.ec, eA, eB);
            esum[1] += tile_fixed(eA, ovf) + tile_fixed(eB, ovf);
            if (VIRIAL && unit_img) tile1_virial_unit(wimg, wv, lane);
            if (__any_sync(kFull, ovf)) {
                if (lane == 0) atomicOr(A.status, ST_OVERFLOW);
                ovf = false;
            }
        } else if (lane == 0) {
            u_next = claim_unit(A, n_first);
        }
        u = __shfl_sync(kFull, u_next, 0);
    }
    if (DEBUG) return;
    long long v[kTaskVals];
    tile_warp_sums<VIRIAL>(esum, wv, v);
    if (lane == 0) {
        s_sys[w] = cur_sys;
        for (int k = 0; k < kTaskVals; ++k) s_val[w][k] = k < (VIRIAL ? kTaskVals : 2) ? v[k] : 0;
    }
    __syncthreads();
    if (threadIdx.x < (VIRIAL ? kTaskVals : 2)) {
        const int k = threadIdx.x;
        const int nw = blockDim.x >> 5;
        int base = -1;
        long long sum = 0;
        for (int q = 0; q < nw; ++q) {
            const int sq = s_sys[q];
            if (sq < 0) continue;
            if (base < 0) base = sq;
            if (sq == base) sum += s_val[q][k];
            else if (s_val[q][k]) atomicAdd((unsigned long long *)&A.sys_acc[sq * kTaskVals + k], (unsigned long long)s_val[q][k]);
        }
        if (base >= 0 && sum) atomicAdd((unsigned long long *)&A.sys_acc[base * kTaskVals + k], (unsigned long long)sum);
    }
}

// ---------------------------------------------------------------------------
// Adjoint kernel on i-group tiles (k_adjoint): the forward kernel's units,
// entries, tiles, half-tile votes and staging, with the pair adjoint of
// eval_pair_adj.  Per entry the j-side terms (dL/dx_j, dL/dq_j) of all its
// tiles are summed in registers, then over the 8 lanes of each j atom, and
// lane ia adds component ia % 4 of atom jb (ia < 4) or jb + 4 to the
// fixed-point sums; the i-side terms accumulate per lane and cluster in
// shared memory until the unit is done; the type-pair gradients go to a
// block table in shared memory (integer atomics) flushed at the end.  One
// inlined instance of the entry code serves every entry kind (the pair
// adjoint is long; an instance per kind overflowed the instruction cache).
constexpr int kAdjWarps = 4;             // warps per block of the adjoint tile kernel

__host__ __device__ inline size_t adj_warp_bytes(int G)
{
    return (size_t)kCluster * G * (16 + 16 + 4) + (size_t)G * 32 * 16 + (size_t)kBatch * kCluster * (16 + 16 + 4);
}

template <int G, int RAD>
__device__ __forceinline__ void adj_entry(const ForceArgs &A, const AdjTables &tab, const float4 *__restrict__ s_ix,
                                          const int *__restrict__ s_it, const float4 *__restrict__ s_ig,
                                          float4 *__restrict__ s_ai, const ulonglong2 *own8, uint2 ent, float4 pjA,
                                          float4 pjB, float4 gjA, float4 gjB, int tjA, int tjB, float gE_lj, float gE_c, int ia, int jb,
                                          int lane, float Lx, float Ly, float Lz, bool &ovf)
{
    const int J = (int)(ent.x & kJMask);
    const uint32_t code = (ent.x >> kShiftBit) & 0x3Fu;
    const bool img = code != 0u, special = (ent.x & kExclFlag) != 0u;
    if (img) {
        if ((code & 3u) == 1u) { pjA.x = __fsub_rn(pjA.x, Lx); pjB.x = __fsub_rn(pjB.x, Lx); }
        if (((code >> 2) & 3u) == 1u) { pjA.y = __fsub_rn(pjA.y, Ly); pjB.y = __fsub_rn(pjB.y, Ly); }
        if ((code >> 4) == 1u) { pjA.z = __fsub_rn(pjA.z, Lz); pjB.z = __fsub_rn(pjB.z, Lz); }
    }
    const ulonglong2 *rec = special ? entry_record<G>(A, ent.y, own8) : nullptr;
    float jA[4] = {0.0f, 0.0f, 0.0f, 0.0f}, jB[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (unsigned cm = ent.y & ((1u << mask_bit(G)) - 1u); cm; cm &= cm - 1u) {
        const int c = __ffs(cm) - 1;
        const int ii = c * kCluster + ia;
        float4 pi = s_ix[ii];
        if (img) {
            if ((code & 3u) == 2u) pi.x = __fsub_rn(pi.x, Lx);
            if (((code >> 2) & 3u) == 2u) pi.y = __fsub_rn(pi.y, Ly);
            if ((code >> 4) == 2u) pi.z = __fsub_rn(pi.z, Lz);
        }
        float dxA, dyA, dzA, dxB, dyB, dzB;
        const float r2A = disp_r2(pjA.x, pjA.y, pjA.z, pi.x, pi.y, pi.z, dxA, dyA, dzA);
        const float r2B = disp_r2(pjB.x, pjB.y, pjB.z, pi.x, pi.y, pi.z, dxB, dyB, dzB);
        bool inA = r2A < A.P.rc2, inB = r2B < A.P.rc2;
        bool s14A = false, s14B = false;
        if (special) tile_mask_bits(rec[c], ia, jb, inA, inB, s14A, s14B);
        const bool anyA = __any_sync(kFull, inA), anyB = __any_sync(kFull, inB);
        if (!anyA && !anyB) continue;
        const int trow = s_it[ii];
        const float4 gi = s_ig[ii];
        float4 ai = s_ai[c * 32 + lane];
        AccAdj acc = {ai.x, ai.y, ai.z, ai.w};
        if (anyA) {
            float a, b, cc, d, ds, de;
            eval_pair_adj<RAD == 1>(A.P, tab, trow, pi.w, gi.x, gi.y, gi.z, gE_lj, gE_c, inA, dxA, dyA, dzA,
                                    inA ? r2A : 1.0f, pjA.w, tjA, gjA, s14A, A.status, acc, a, b, cc, d, ds, de);
            add_type_grads(tab, inA ? trow + tjA : -1, ds, de, A.status);
            jA[0] = __fadd_rn(jA[0], a);
            jA[1] = __fadd_rn(jA[1], b);
            jA[2] = __fadd_rn(jA[2], cc);
            jA[3] = __fadd_rn(jA[3], d);
        }
        if (anyB) {
            float a, b, cc, d, ds, de;
            eval_pair_adj<RAD == 1>(A.P, tab, trow, pi.w, gi.x, gi.y, gi.z, gE_lj, gE_c, inB, dxB, dyB, dzB,
                                    inB ? r2B : 1.0f, pjB.w, tjB, gjB, s14B, A.status, acc, a, b, cc, d, ds, de);
            add_type_grads(tab, inB ? trow + tjB : -1, ds, de, A.status);
            jB[0] = __fadd_rn(jB[0], a);
            jB[1] = __fadd_rn(jB[1], b);
            jB[2] = __fadd_rn(jB[2], cc);
            jB[3] = __fadd_rn(jB[3], d);
        }
        s_ai[c * 32 + lane] = make_float4(acc.dx, acc.dy, acc.dz, acc.dq);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            jA[k] = __fadd_rn(jA[k], __shfl_xor_sync(kFull, jA[k], o));
            jB[k] = __fadd_rn(jB[k], __shfl_xor_sync(kFull, jB[k], o));
        }
    float gv = jA[0];
#pragma unroll
    for (int k = 1; k < 4; ++k) gv = ia == k ? jA[k] : gv;
#pragma unroll
    for (int k = 0; k < 4; ++k) gv = ia == 4 + k ? jB[k] : gv;
    const long long gx = tile_fixed(gv, ovf);
    if (gx != 0) {
        const int j = ia < 4 ? jb : jb + 4;
        atomicAdd((unsigned long long *)&A.gacc[32ll * J + 4 * j + (ia & 3)], (unsigned long long)gx);
    }
}

template <int G, int RAD>
__global__ void __launch_bounds__(kAdjWarps * 32) k_adjoint(ForceArgs A, int parts, int n_first)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int T = A.P.n_types;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, ia = lane & 7, jb = lane >> 3;
    size_t off = 0;
    unsigned long long *tacc = reinterpret_cast<unsigned long long *>(smem + off);
    off += (size_t)T * T * 16;
    float4 *ljd = reinterpret_cast<float4 *>(smem + off);
    off += (size_t)T * T * 16;
    float2 *lj = reinterpret_cast<float2 *>(smem + off);
    off += align16((size_t)T * T * 8);
    unsigned char *wbase = smem + off + (size_t)w * adj_warp_bytes(G);
    float4 *s_ix = reinterpret_cast<float4 *>(wbase);    // [8 G] x, y, z, ke q
    float4 *s_ig = s_ix + kCluster * G;                    // [8 G] dL/dF of the i atoms
    float4 *s_ai = s_ig + kCluster * G;                    // [G * 32] i-side partials
    float4 *sjp = s_ai + G * 32;                           // [kBatch * 8]
    float4 *sjg = sjp + kBatch * kCluster;                 // [kBatch * 8]
    int *s_it = reinterpret_cast<int *>(sjg + kBatch * kCluster);  // [8 G]
    int *sjt = s_it + kCluster * G;                        // [kBatch * 8]
    for (int k = threadIdx.x; k < T * T; k += blockDim.x) {
        lj[k] = make_float2(A.lj_tab[k].x, A.lj_tab[k].y);
        ljd[k] = A.lj_d[k];
        tacc[2 * k] = 0ull;
        tacc[2 * k + 1] = 0ull;
    }
    pdl_entry();  // the type-pair tables do not depend on the preceding kernels
    __syncthreads();
    const AdjTables tab{lj, ljd, tacc};
    const int n_units = A.counts[4] * kListSegs * parts;
    int cur_sys = -1;
    float Lx = 0.0f, Ly = 0.0f, Lz = 0.0f, gE_lj = 0.0f, gE_c = 0.0f;
    bool ovf = false;
    int u = first_unit(w);
    while (u < n_units) {
        int u_next = 0;
        const Unit U = unit_of(A, u, parts);
        if (U.e_begin < U.e_end) {
            const int2 gr = __ldg(A.grp + U.g);
            const int c0 = gr.x, ncl = gr.y;
            const ulonglong2 *own8 = G == 8 ? A.gmask + (long long)c0 * kMaskRecsPerCluster * 8 : nullptr;
            const int sys_id = __ldg(A.clus_sys + c0);
            if (sys_id != cur_sys) {
                cur_sys = sys_id;
                Lx = A.sys[sys_id].L[0];
                Ly = A.sys[sys_id].L[1];
                Lz = A.sys[sys_id].L[2];
                gE_lj = A.dLdE ? (float)A.dLdE[2 * sys_id] : 0.0f;
                gE_c = A.dLdE ? (float)A.dLdE[2 * sys_id + 1] : 0.0f;
            }
            for (int t = lane; t < kCluster * G; t += 32) {
                const long long slot = (long long)c0 * kCluster + t;
                float4 p = make_float4(kFarCoord, kFarCoord, kFarCoord, 0.0f);
                float4 gi = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                int tr = 0;
                if (t < kCluster * ncl) {
                    p = __ldg(A.xyzq + slot);
                    if (!is_real_coord(p.x)) p.x = p.y = p.z = kFarCoord;
                    p.w *= A.P.ke;
                    gi = __ldg(A.gslot + slot);
                    tr = __ldg(A.tslot + slot) * T;
                }
                s_ix[t] = p;
                s_ig[t] = gi;
                s_it[t] = tr;
            }
#pragma unroll
            for (int c = 0; c < G; ++c) s_ai[c * 32 + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            __syncwarp();
            const uint2 *row = A.glist + U.base;
            for (int e0 = U.e_begin; e0 < U.e_end; e0 += kBatch) {
                const int ne = min(kBatch, U.e_end - e0);
                const uint2 my = lane < ne ? __ldg(row + e0 + lane) : make_uint2(0u, 0u);
                if (lane < ne) {
                    const long long jbase = (long long)(my.x & kJMask) * kCluster;
#pragma unroll
                    for (int a = 0; a < kCluster; ++a) {
                        cp_async16(sjp + swz(lane, a), A.xyzq + jbase + a);
                        cp_async16(sjg + swz(lane, a), A.gslot + jbase + a);
                        cp_async4(sjt + swz(lane, a), A.tslot + jbase + a);
                    }
                }
                cp_async_wait_all();
                __syncwarp();
                for (int k = 0; k < ne; ++k) {
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    adj_entry<G, RAD>(A, tab, s_ix, s_it, s_ig, s_ai, own8, ent, sjp[swz(k, jb)], sjp[swz(k, jb + 4)],
                                      sjg[swz(k, jb)], sjg[swz(k, jb + 4)], sjt[swz(k, jb)], sjt[swz(k, jb + 4)],
                                      gE_lj, gE_c, ia, jb, lane, Lx, Ly, Lz, ovf);
                }
                __syncwarp();  // the staging buffers are rewritten by the next batch
            }
            if (lane == 0) u_next = claim_unit(A, n_first);
            // i-side terms: the 4 lanes of each atom summed in FP32 (fixed
            // butterfly), then lane jb adds clusters c with c % 4 == jb
#pragma unroll
            for (int c = 0; c < G; ++c) {
                float4 a = s_ai[c * 32 + lane];
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    a.x = __fadd_rn(a.x, __shfl_xor_sync(kFull, a.x, o));
                    a.y = __fadd_rn(a.y, __shfl_xor_sync(kFull, a.y, o));
                    a.z = __fadd_rn(a.z, __shfl_xor_sync(kFull, a.z, o));
                    a.w = __fadd_rn(a.w, __shfl_xor_sync(kFull, a.w, o));
                }
                if ((c & 3) == jb && c < ncl) {
                    const long long slot = (long long)c0 * kCluster + c * kCluster + ia;
                    const long long v0 = tile_fixed(a.x, ovf), v1 = tile_fixed(a.y, ovf), v2 = tile_fixed(a.z, ovf),
                                    v3 = tile_fixed(a.w, ovf);
                    if (v0) atomicAdd((unsigned long long *)&A.gacc[4 * slot], (unsigned long long)v0);
                    if (v1) atomicAdd((unsigned long long *)&A.gacc[4 * slot + 1], (unsigned long long)v1);
                    if (v2) atomicAdd((unsigned long long *)&A.gacc[4 * slot + 2], (unsigned long long)v2);
                    if (v3) atomicAdd((unsigned long long *)&A.gacc[4 * slot + 3], (unsigned long long)v3);
                }
            }
            if (__any_sync(kFull, ovf)) {
                if (lane == 0) atomicOr(A.status, ST_OVERFLOW);
                ovf = false;
            }
            __syncwarp();
        } else if (lane == 0) {
            u_next = claim_unit(A, n_first);
        }
        u = __shfl_sync(kFull, u_next, 0);
    }
    // block table of parameter gradients -> global (integer sums)
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * T * T; k += blockDim.x)
        if (tacc[k]) atomicAdd((unsigned long long *)&A.tab_acc[k], tacc[k]);
}

// Adjoint kernel for i-groups of one cluster (k_adjoint1): the structure of
// k_force1.  Lane = jj + 8 ih holds j atom jj of the entry's cluster J and i
// atoms ih and ih + 4 of the unit's cluster, whose positions, dL/dF and
// type rows stay in registers for the whole unit; the i-side terms (dL/dx_i,
// dL/dq_i) accumulate per lane in registers.  Per entry the j-side terms of
// the lane's two pairs share its j atom: they are summed over the 4 lanes of
// that atom (two shuffle levels) and lane ih adds component ih (x, y, z, q)
// to the fixed-point sums.  The type-pair gradients go to the block table
// as in k_adjoint.
struct TileIA {
    float x, y, z, qk;  // position, ke q
    float4 g;           // dL/dF of the atom
    int trow;           // type row (t T)
};

__device__ __forceinline__ TileIA load_tile_ia(const ForceArgs &A, long long slot, int T)
{
    TileIA t;
    const float4 p = __ldg(A.xyzq + slot);
    const bool real = is_real_coord(p.x);
    t.x = real ? p.x : kFarCoord;
    t.y = real ? p.y : kFarCoord;
    t.z = real ? p.z : kFarCoord;
    t.qk = p.w * A.P.ke;
    t.g = __ldg(A.gslot + slot);
    t.trow = __ldg(A.tslot + slot) * T;
    return t;
}

template <int RAD>
__device__ __forceinline__ void adj1_entry(const ForceArgs &A, const AdjTables &tab, uint2 ent, float4 pj, float4 gj,
                                           int tj, const TileIA &ia, const TileIA &ib, int jj, int ih, float Lx,
                                           float Ly, float Lz, float gE_lj, float gE_c, AccAdj &acA, AccAdj &acB,
                                           bool &ovf)
{
    const int J = (int)(ent.x & kJMask);
    const uint32_t code = (ent.x >> kShiftBit) & 0x3Fu;
    const bool img = code != 0u, special = (ent.x & kExclFlag) != 0u;
    float ax = ia.x, ay = ia.y, az = ia.z, bx = ib.x, by = ib.y, bz = ib.z;
    if (img) {  // j side: x_j - L on code-1 axes; i side: x_i - L on code-2 axes
        if ((code & 3u) == 1u) pj.x = __fsub_rn(pj.x, Lx);
        if (((code >> 2) & 3u) == 1u) pj.y = __fsub_rn(pj.y, Ly);
        if ((code >> 4) == 1u) pj.z = __fsub_rn(pj.z, Lz);
        if ((code & 3u) == 2u) { ax = __fsub_rn(ax, Lx); bx = __fsub_rn(bx, Lx); }
        if (((code >> 2) & 3u) == 2u) { ay = __fsub_rn(ay, Ly); by = __fsub_rn(by, Ly); }
        if ((code >> 4) == 2u) { az = __fsub_rn(az, Lz); bz = __fsub_rn(bz, Lz); }
    }
    float dxA, dyA, dzA, dxB, dyB, dzB;
    const float r2A = disp_r2(pj.x, pj.y, pj.z, ax, ay, az, dxA, dyA, dzA);
    const float r2B = disp_r2(pj.x, pj.y, pj.z, bx, by, bz, dxB, dyB, dzB);
    bool inA = r2A < A.P.rc2, inB = r2B < A.P.rc2;
    bool s14A = false, s14B = false;
    if (special) {  // exclusion bitmask of the tile: bit 8 i + j
        const ulonglong2 m = A.gmask[ent.y >> mask_bit(1)];
        const int bA = ih * kCluster + jj, bB = bA + 4 * kCluster;
        inA = inA && !((m.x >> bA) & 1ull);
        inB = inB && !((m.x >> bB) & 1ull);
        s14A = (m.y >> bA) & 1ull;
        s14B = (m.y >> bB) & 1ull;
    }
    const bool anyA = __any_sync(kFull, inA), anyB = __any_sync(kFull, inB);
    if (!anyA && !anyB) return;
    float jt[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // the j atom's terms (x, y, z, q)
    if (anyA) {
        float a, b, c, d, ds, de;
        eval_pair_adj<RAD == 1>(A.P, tab, ia.trow, ia.qk, ia.g.x, ia.g.y, ia.g.z, gE_lj, gE_c, inA, dxA, dyA, dzA,
                                inA ? r2A : 1.0f, pj.w, tj, gj, s14A, A.status, acA, a, b, c, d, ds, de);
        add_type_grads(tab, inA ? ia.trow + tj : -1, ds, de, A.status);
        jt[0] = a;
        jt[1] = b;
        jt[2] = c;
        jt[3] = d;
    }
    if (anyB) {
        float a, b, c, d, ds, de;
        eval_pair_adj<RAD == 1>(A.P, tab, ib.trow, ib.qk, ib.g.x, ib.g.y, ib.g.z, gE_lj, gE_c, inB, dxB, dyB, dzB,
                                inB ? r2B : 1.0f, pj.w, tj, gj, s14B, A.status, acB, a, b, c, d, ds, de);
        add_type_grads(tab, inB ? ib.trow + tj : -1, ds, de, A.status);
        jt[0] = __fadd_rn(jt[0], a);
        jt[1] = __fadd_rn(jt[1], b);
        jt[2] = __fadd_rn(jt[2], c);
        jt[3] = __fadd_rn(jt[3], d);
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) jt[k] = __fadd_rn(jt[k], __shfl_xor_sync(kFull, jt[k], o));
    const float gv = ih == 0 ? jt[0] : (ih == 1 ? jt[1] : (ih == 2 ? jt[2] : jt[3]));
    const long long gx = tile_fixed(gv, ovf);
    if (gx != 0) atomicAdd((unsigned long long *)&A.gacc[32ll * J + 4 * jj + ih], (unsigned long long)gx);
}

constexpr int kBatchA = 16;  // entries staged per batch of the single-cluster adjoint (shared memory per block)

__host__ __device__ inline size_t adj1_warp_bytes() { return (size_t)kBatchA * kCluster * (16 + 16 + 4); }

size_t adjoint1_smem_bytes(int T)
{
    return (size_t)T * T * 32 + align16((size_t)T * T * 8) + (size_t)kAdjWarps * adj1_warp_bytes();
}

template <int RAD>
__global__ void __launch_bounds__(kAdjWarps * 32) k_adjoint1(ForceArgs A, int parts, int n_first)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int T = A.P.n_types;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, jj = lane & 7, ih = lane >> 3;
    size_t off = 0;
    unsigned long long *tacc = reinterpret_cast<unsigned long long *>(smem + off);
    off += (size_t)T * T * 16;
    float4 *ljd = reinterpret_cast<float4 *>(smem + off);
    off += (size_t)T * T * 16;
    float2 *lj = reinterpret_cast<float2 *>(smem + off);
    off += align16((size_t)T * T * 8);
    float4 *sjp = reinterpret_cast<float4 *>(smem + off + (size_t)w * adj1_warp_bytes());  // [kBatchA * 8]
    float4 *sjg = sjp + kBatchA * kCluster;                                                // [kBatchA * 8]
    int *sjt = reinterpret_cast<int *>(sjg + kBatchA * kCluster);                          // [kBatchA * 8]
    for (int k = threadIdx.x; k < T * T; k += blockDim.x) {
        lj[k] = make_float2(A.lj_tab[k].x, A.lj_tab[k].y);
        ljd[k] = A.lj_d[k];
        tacc[2 * k] = 0ull;
        tacc[2 * k + 1] = 0ull;
    }
    pdl_entry();  // the type-pair tables do not depend on the preceding kernels
    __syncthreads();
    const AdjTables tab{lj, ljd, tacc};
    const int n_units = A.counts[4] * kListSegs * parts;
    int cur_sys = -1;
    float Lx = 0.0f, Ly = 0.0f, Lz = 0.0f, gE_lj = 0.0f, gE_c = 0.0f;
    bool ovf = false;
    int u = first_unit(w);
    while (u < n_units) {
        int u_next = 0;
        const Unit U = unit_of(A, u, parts);
        // as in k_force1: what needs only the unit's group and segment is
        // loaded before the segment's length is known
        const int I = U.g;  // one-cluster groups are numbered like their clusters
        const int sys_id = __ldg(A.clus_sys + I);
        const long long s0 = (long long)I * kCluster;
        const TileIA ia = load_tile_ia(A, s0 + ih, T);
        const TileIA ib = load_tile_ia(A, s0 + ih + 4, T);
        const uint2 *row = A.glist + U.base;
        const uint2 first = lane < A.cap / kListSegs ? __ldg(row + lane) : make_uint2(0u, 0u);
        if (U.e_begin < U.e_end) {
            if (sys_id != cur_sys) {
                cur_sys = sys_id;
                Lx = A.sys[sys_id].L[0];
                Ly = A.sys[sys_id].L[1];
                Lz = A.sys[sys_id].L[2];
                gE_lj = A.dLdE ? (float)A.dLdE[2 * sys_id] : 0.0f;
                gE_c = A.dLdE ? (float)A.dLdE[2 * sys_id + 1] : 0.0f;
            }
            AccAdj acA = {0.0f, 0.0f, 0.0f, 0.0f}, acB = {0.0f, 0.0f, 0.0f, 0.0f};
            for (int e0 = U.e_begin; e0 < U.e_end; e0 += kBatchA) {
                const int ne = min(kBatchA, U.e_end - e0);
                const uint2 my = lane < ne ? (e0 == 0 ? first : __ldg(row + e0 + lane)) : make_uint2(0u, 0u);
                if (lane < ne) {
                    const long long jbase = (long long)(my.x & kJMask) * kCluster;
#pragma unroll
                    for (int a = 0; a < kCluster; ++a) {
                        cp_async16(sjp + swz(lane, a), A.xyzq + jbase + a);
                        cp_async16(sjg + swz(lane, a), A.gslot + jbase + a);
                        cp_async4(sjt + swz(lane, a), A.tslot + jbase + a);
                    }
                }
                cp_async_wait_all();
                __syncwarp();
                for (int k = 0; k < ne; ++k) {
                    const uint2 ent = make_uint2(__shfl_sync(kFull, my.x, k), __shfl_sync(kFull, my.y, k));
                    adj1_entry<RAD>(A, tab, ent, sjp[swz(k, jj)], sjg[swz(k, jj)], sjt[swz(k, jj)], ia, ib, jj, ih,
                                    Lx, Ly, Lz, gE_lj, gE_c, acA, acB, ovf);
                }
                __syncwarp();  // the staging buffers are rewritten by the next batch
            }
            if (lane == 0) u_next = claim_unit(A, n_first);
            // i-side terms: the 8 lanes of each atom summed in FP32 (a fixed
            // butterfly), then lanes jj < 4 add component jj of atom ih and
            // lanes jj >= 4 component jj - 4 of atom ih + 4
            float v[8] = {acA.dx, acA.dy, acA.dz, acA.dq, acB.dx, acB.dy, acB.dz, acB.dq};
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = __fadd_rn(v[c], __shfl_xor_sync(kFull, v[c], o));
            float mine = v[0];
#pragma unroll
            for (int c = 1; c < 8; ++c) mine = jj == c ? v[c] : mine;
            const long long gi = tile_fixed(mine, ovf);
            if (gi != 0) {
                const long long slot = s0 + ih + (jj < 4 ? 0 : 4);
                atomicAdd((unsigned long long *)&A.gacc[4 * slot + (jj & 3)], (unsigned long long)gi);
            }
            if (__any_sync(kFull, ovf)) {
                if (lane == 0) atomicOr(A.status, ST_OVERFLOW);
                ovf = false;
            }
        } else if (lane == 0) {
            u_next = claim_unit(A, n_first);
        }
        u = __shfl_sync(kFull, u_next, 0);
    }
    // block table of parameter gradients -> global (integer sums)
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * T * T; k += blockDim.x)
        if (tacc[k]) atomicAdd((unsigned long long *)&A.tab_acc[k], tacc[k]);
}

// Gather charges and types into sorted order and check that the positions
// are those of the last build.
__global__ void k_pack(int slot_cap, const int *__restrict__ counts, const int *__restrict__ perm,
                       float4 *__restrict__ xyzq, int *__restrict__ tslot, const float *__restrict__ pos,
                       const float *__restrict__ q, const int *__restrict__ type, const SysDesc *__restrict__ sys,
                       const int *__restrict__ atom_sys, int T, int *__restrict__ status,
                       long long *__restrict__ facc, long long *__restrict__ sys_acc, int n_acc,
                       int *__restrict__ work)
{
    pdl_entry();
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (work && s == 0) *work = 0;  // the force kernel's work-unit counter
    // zero the force kernel's fixed-point sums (forward calls pass them)
    if (facc && s < slot_cap) {
        facc[3ll * s] = 0;
        facc[3ll * s + 1] = 0;
        facc[3ll * s + 2] = 0;
    }
    if (sys_acc && s < n_acc) sys_acc[s] = 0;
    if (s >= slot_cap || s >= counts[0]) return;
    int a = perm[s];
    if (a < 0) return;
    const SysDesc &S = sys[atom_sys[a]];
    float4 p = xyzq[s];
    float x = wrap_coord(pos[3 * (long long)a], S.L[0]);
    float y = wrap_coord(pos[3 * (long long)a + 1], S.L[1]);
    float z = wrap_coord(pos[3 * (long long)a + 2], S.L[2]);
    if (x != p.x || y != p.y || z != p.z) atomicOr(status, ST_STALE);
    int t = type[a];
    if (t < 0 || t >= T) {
        atomicOr(status, ST_BADTYPE);
        t = 0;
    }
    xyzq[s] = make_float4(p.x, p.y, p.z, q[a]);
    tslot[s] = t;
}

// x v 2^-12 rounded to the nearest integer (half up), for a wrapped
// coordinate x >= 0 and a fixed-point force v (2^32): a virial term on the
// 2^20 grid.  Exact in integers, mantissa times v with one rounding: the
// FP64 unit would take 64 cycles per warp for each of the products and
// conversions (15 per atom).
// (beyond 2,048 A the product does not fit and FP64 takes over, in a function
// of its own: inlined, the compiler ran both sides for every atom)
__device__ __noinline__ long long virial_term_fp64(float x, long long v)
{
    return __double2ll_rn((double)x * ((double)v * (kVirScale / kFixScale)));
}

__device__ __forceinline__ long long virial_term(float x, long long v)
{
    const unsigned b = __float_as_uint(x);
    const int e = (int)(b >> 23);
    if (e > 137) return virial_term_fp64(x, v);  // x >= 2048
    const unsigned m = e > 0 ? (b & 0x7FFFFFu) | 0x800000u : 0u;  // x = m 2^(e - 150); subnormal: no term
    const long long hi = v >> 24;
    const unsigned lo = (unsigned)v & 0xFFFFFFu;
    // m v = q 2^24 + (a remainder that floor and half up never see)
    const long long q = (long long)m * hi + (long long)(((unsigned long long)m * lo) >> 24);
    const int sh = min(138 - e, 62);  // 24 + sh = 150 - e + 12
    return (q + (1ll << (sh - 1))) >> sh;
}

constexpr int kUnpackThreads = 64;  // 64 threads of at most 64 registers: what the force kernel's 24 warps of 80 leave

// Add a warp's per-lane virial terms (lanes with sys < 0 hold none) to the
// per-system sums: for each distinct system among the lanes one reduction in
// which the lanes trade components (8 to 4 to 2 to 1 per lane, then two more
// levels), and one atomic per component.
__device__ __forceinline__ void flush_virial_warp(long long (&w)[6], int sys, long long *sys_acc)
{
    const int lane = threadIdx.x & 31;
    unsigned rem = __ballot_sync(kFull, sys >= 0);
    while (rem) {
        const int cs = __shfl_sync(kFull, sys, __ffs(rem) - 1);
        const bool mine = sys == cs;
        long long v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = k < 6 && mine ? w[k] : 0;
#pragma unroll
        for (int n = 4; n >= 1; n >>= 1) {  // lane bit n set: keep the upper n components
#pragma unroll
            for (int k = 0; k < n; ++k) {
                const long long keep = lane & n ? v[k + n] : v[k], give = lane & n ? v[k] : v[k + n];
                v[k] = keep + __shfl_xor_sync(kFull, give, n);
            }
        }
        v[0] += __shfl_xor_sync(kFull, v[0], 8);
        v[0] += __shfl_xor_sync(kFull, v[0], 16);
        // lane k < 8 holds component k
        if (lane < 6 && v[0]) atomicAdd((unsigned long long *)&sys_acc[cs * kTaskVals + 2 + lane], (unsigned long long)v[0]);
        rem &= ~__ballot_sync(kFull, mine);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = 0;
}

// Fixed-point forces (sorted order) to FP32 in the caller's order, one
// thread per atom in caller order (gathers from the sorted sums, and
// coalesced writes of F, which may be page-locked host memory).  With
// VIRIAL, also the atom part of the virial: for central pair forces
// W_ab = sum_pairs d_a f_b (d = x_j' - x_i, f the force on j) equals
// sum_atoms x_a F_b over the wrapped coordinates x and total forces F, plus
// the periodic-image terms added by the force kernel.  Each atom's terms are
// rounded to the 2^20 fixed-point grid and summed as integers per thread
// (grid-stride loop, atoms in system order) and per warp.
//
// Latency bound at 23,500 atoms, memory bound at 1 M (about 100 bytes an
// atom in scattered 32-byte sectors).  Blocks of 64 threads fit beside the
// force kernel's warps, so most are resident when it ends; a thread's slot
// and position (complete before the force kernel began) are loaded before
// the wait; the arithmetic is integer.  With blocks of 256 threads and FP64
// products the kernel took 53 us at 999,999 atoms, now 25 us (ncu, cold);
// rebuild + forces 89.5 -> 85.6 us at 23,500 atoms, 52.2 -> 48.6 us at 6,144,
// 2173 -> 2129 us at 999,999.
template <bool VIRIAL>
__global__ void __launch_bounds__(kUnpackThreads, 16)
    k_unpack_forces(int n_atoms, int *__restrict__ counts, const int *__restrict__ inv, const long long *__restrict__ facc,
                    float *__restrict__ F, const float4 *__restrict__ xyzq, const int *__restrict__ atom_sys,
                    long long *__restrict__ sys_acc, int n_sys, double *__restrict__ energy,
                    double *__restrict__ virial, const long long *__restrict__ pme_f,
                    const long long *__restrict__ pme_s, double pme_self)
{
    const int stride = gridDim.x * blockDim.x;
    int a = blockIdx.x * blockDim.x + threadIdx.x;
    // of the kernels before the force kernel
    int s = a < n_atoms ? inv[a] : -1;
    float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int sys = -1;
    if (VIRIAL && s >= 0) {
        x = xyzq[s];
        sys = n_sys == 1 ? 0 : atom_sys[a];
    }
    pdl_entry();
    long long w[6] = {0, 0, 0, 0, 0, 0};
    int wsys = -1;
    for (int a0 = a - (int)threadIdx.x; a0 < n_atoms; a0 += stride) {
        if (VIRIAL) {
            // atoms come in system order: flush a lane's sums before it moves on
            if (__any_sync(kFull, sys >= 0 && wsys >= 0 && sys != wsys)) {
                flush_virial_warp(w, wsys, sys_acc);
                wsys = -1;
            }
        }
        if (s >= 0) {
            const long long v0 = facc[3ll * s], v1 = facc[3ll * s + 1], v2 = facc[3ll * s + 2];
            // PME forces (same slot order) join the sum before the one
            // rounding; the atom part of the virial is the short-range forces' alone
            const long long p0 = pme_f ? pme_f[3ll * s] : 0, p1 = pme_f ? pme_f[3ll * s + 1] : 0,
                            p2 = pme_f ? pme_f[3ll * s + 2] : 0;
            F[3ll * a] = fixed_to_float(v0 + p0);
            F[3ll * a + 1] = fixed_to_float(v1 + p1);
            F[3ll * a + 2] = fixed_to_float(v2 + p2);
            if (VIRIAL) {
                w[0] += virial_term(x.x, v0);
                w[1] += virial_term(x.y, v1);
                w[2] += virial_term(x.z, v2);
                w[3] += virial_term(x.x, v1);
                w[4] += virial_term(x.x, v2);
                w[5] += virial_term(x.y, v2);
                wsys = sys;
            }
        }
        a += stride;
        s = a < n_atoms ? inv[a] : -1;
        sys = -1;
        if (VIRIAL && s >= 0) {
            x = xyzq[s];
            sys = n_sys == 1 ? 0 : atom_sys[a];
        }
    }
    if (VIRIAL) flush_virial_warp(w, wsys, sys_acc);
    if (!energy && !virial) return;
    // the last block to finish converts the per-system sums (counts[2] is the
    // completion ticket: zero on entry, reset here)
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&counts[2], 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = threadIdx.x; i < n_sys * kTaskVals; i += blockDim.x) {
        const int sy = i / kTaskVals, k = i % kTaskVals;
        long long raw = __ldcg(&sys_acc[i]);
        if (pme_s) {  // single system: reciprocal + self + pair corrections join E_Coul and W
            if (k == 1)  // the self term from sum q^2 (scale 2^36) to the energy scale 2^32
                raw += __ldcg(&pme_s[0]) + __ldcg(&pme_s[2]) +
                       __double2ll_rn(pme_self * (double)__ldcg(&pme_s[1]) * (1.0 / 16.0));
            if (k >= 2) raw += __ldcg(&pme_s[1 + k]);
        }
        const double v = (double)raw * (k < 2 ? 1.0 / kFixScale : 1.0 / kVirScale);
        if (k < 2) {
            if (energy) energy[2 * sy + k] = v;
        } else if (virial) {
            virial[6 * sy + k - 2] = v;
        }
    }
    if (threadIdx.x == 0) counts[2] = 0;
}

// Adjoint sums (sorted order, fixed point) to FP32 dL/dx, dL/dq in the
// caller's order.
__global__ void k_unpack_adjoint(int slot_cap, const int *__restrict__ counts, const int *__restrict__ perm,
                                 const long long *__restrict__ gacc, float *__restrict__ dpos, float *__restrict__ dq)
{
    pdl_entry();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= slot_cap || s >= counts[0]) return;
    const int a = perm[s];
    if (a < 0) return;
    if (dpos) {
        dpos[3ll * a] = fixed_to_float(gacc[4ll * s]);
        dpos[3ll * a + 1] = fixed_to_float(gacc[4ll * s + 1]);
        dpos[3ll * a + 2] = fixed_to_float(gacc[4ll * s + 2]);
    }
    if (dq) dq[a] = fixed_to_float(gacc[4ll * s + 3]);
}

// Kernel function attributes belong to each device's context, so the
// shared-memory opt-in is made once per device (one bit per device in
// `done`; devices beyond 63 set it at every launch).  Concurrent first calls
// may both set it, which is harmless.
template <typename Kernel>
static void smem_optin_once(Kernel kernel, int device, int bytes, std::atomic<unsigned long long> &done)
{
    const unsigned long long bit = device >= 0 && device < 64 ? 1ull << device : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (bit) done.fetch_or(bit, std::memory_order_release);
}

size_t tile_smem_bytes(int T, int G) { return lj_table_bytes(T) + (size_t)kTileWarps * tile_warp_bytes(G); }

// beside_pme: the PME chain, forked before the list kernel, runs on its side
// stream during the list kernel and this one.  The persistent grid for groups of
// one cluster then leaves room for 8 warps per SM, so that the PME kernels run
// alongside instead of after it; the kernels for larger groups, which hold
// fewer warps anyway, take what the tuning asks for (23,500 atoms: 138 us a
// step with groups of 4, 151 with a block less; 180 and 210 with groups of 8).
// Which block takes which unit does not change any result.  (A second launch behind the PME chain that took units from the same
// counter made up for a chain that started late; now that the chain starts
// with the lists it costs 4 us of the PME step and 7 us of an MD step.)
template <int G, int RAD, bool VIRIAL, bool DEBUG>
static void launch_force_g(nb_ctx *ctx, const ForceArgs &A)
{
    const size_t smem = tile_smem_bytes(A.P.n_types, G);
    static std::atomic<unsigned long long> optin{0};
    smem_optin_once(k_force<G, RAD, VIRIAL, DEBUG>, ctx->device, 200 * 1024, optin);
    // persistent grid: never more blocks than can be resident at once
    int resident = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_force<G, RAD, VIRIAL, DEBUG>, kTileWarps * 32, smem);
    const int per_sm = std::max(1, std::min(ctx->tune.blocks_per_sm, resident));
    const int parts = ctx->tune.list_split > 0 ? ctx->tune.list_split : kDefaultListSplit;
    const int blocks = ctx->num_sms * per_sm;
    launch_pdl(k_force<G, RAD, VIRIAL, DEBUG>, dim3(blocks), dim3(kTileWarps * 32), smem, ctx->stream, A, parts,
               blocks * kTileWarps);
}

// Blocks of an instance of k_force1 that an SM holds (-1: not asked yet; the
// answer depends on the context's type count only and is kept there).
template <int W, int MB, int RAD, bool VIRIAL, bool DEBUG>
static int force1_resident(nb_ctx *ctx)
{
    int &r = ctx->force1_res[W == 8 ? 0 : (MB == 8 ? 2 : 1)][RAD][(VIRIAL ? 1 : 0) + (DEBUG ? 2 : 0)];
    if (r >= 0) return r;
    static std::atomic<unsigned long long> optin{0};
    smem_optin_once(k_force1<W, MB, RAD, VIRIAL, DEBUG>, ctx->device, 200 * 1024, optin);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_force1<W, MB, RAD, VIRIAL, DEBUG>, W * 32,
                                                  lj_table_bytes(ctx->pp.n_types) + W * tile1_warp_bytes());
    return r = n;
}

template <int W, int MB, int RAD, bool VIRIAL, bool DEBUG>
static void launch_force_1w(nb_ctx *ctx, const ForceArgs &A, bool beside_pme)
{
    constexpr int per = kTileWarps / W;  // blocks of W warps in the tuning's unit of kTileWarps warps
    const int resident = force1_resident<W, MB, RAD, VIRIAL, DEBUG>(ctx);
    // (the 64-register shape runs with blocks_per_sm 3, the default, or more: all that fit)
    const int want = W * MB > 24 ? MB : ctx->tune.blocks_per_sm * per;
    // beside PME 8 of the 24 warps' room is left: 109.4 us a step at 23,500
    // atoms (4: 110.2, 12: 116, none: 121).  A smaller grid leaves it as it
    // is: 8 and 16 warps asked for less another 8 took 199 and 134 us, as asked
    // for 137 and 107
    const int room = beside_pme ? std::max(resident - per, std::min(per, resident)) : resident;
    const int per_sm = std::max(1, std::min(want, room));
    const int parts = ctx->tune.list_split > 0 ? ctx->tune.list_split : kDefaultListSplit;
    const int blocks = ctx->num_sms * per_sm;
    launch_pdl(k_force1<W, MB, RAD, VIRIAL, DEBUG>, dim3(blocks), dim3(W * 32),
               lj_table_bytes(A.P.n_types) + W * tile1_warp_bytes(), ctx->stream, A, parts, blocks * W);
}

// Which instance.  Blocks of 4 warps start and end in smaller steps than
// blocks of 8 (the kernel before and the kernel after share the SM's registers
// with them sooner): rebuild + forces, with the unit claims as they are now,
// 93.4 -> 90.6 us at 23,500 atoms, 53.2 -> 51.2 us at 6,144.  Each block holds the type-pair table, so with many
// types (above about 26) an SM holds fewer warps in blocks of 4 than in blocks
// of 8, and blocks of 8 are taken.  So are they for a grid of 8 warps per SM
// (blocks_per_sm 1), whose blocks of 4 would not spread evenly over SMs that
// hold six of them (164 us at 23,500 atoms, 139 with blocks of 8; beside PME
// 137 and 141).  With 64 registers (a few spills) an SM
// holds 32 warps instead of 24, which, where the grid is to fill the SM (a
// smaller grid spreads unevenly here too: 2,875 us at 999,999 atoms with
// blocks_per_sm 2, 2,307 with 80 registers), pays once every warp has kMinRounds
// units (the longer units of fuller SMs make the end of a launch longer):
// 1976 -> 1928 us at 999,999 atoms, 511 -> 503 at 240,000, 914 -> 903 for 64
// boxes, 110.7 -> 109.2 at 39,003, but 90.6 -> 93.1 us at 23,500 (all water: an
// SM has to hold 8 blocks with their tables, so up to 17 types).  The
// tabulated form does not take it: 80.9 -> 83.3 us at 20,001 atoms, 129.0 ->
// 131.9 at 39,003, 262 -> 268 at 90,000 (its loads go to L1 and L2, which more
// warps share).
constexpr int kMinRounds = 4;

template <int RAD, bool VIRIAL, bool DEBUG>
static void launch_force_1(nb_ctx *ctx, const ForceArgs &A, bool beside_pme)
{
    if constexpr (!DEBUG) {
        if constexpr (RAD != 2) {
            const bool fill = !beside_pme && ctx->tune.blocks_per_sm >= 3 && force_rounds(ctx) >= kMinRounds;
            if (fill && force1_resident<4, 8, RAD, VIRIAL, DEBUG>(ctx) >= 8)
                return launch_force_1w<4, 8, RAD, VIRIAL, DEBUG>(ctx, A, beside_pme);
        }
        const bool fours = beside_pme || ctx->tune.blocks_per_sm > 1;
        if (fours && force1_resident<4, 6, RAD, VIRIAL, DEBUG>(ctx) >= 2 * force1_resident<8, 3, RAD, VIRIAL, DEBUG>(ctx))
            return launch_force_1w<4, 6, RAD, VIRIAL, DEBUG>(ctx, A, beside_pme);
    }
    launch_force_1w<8, 3, RAD, VIRIAL, DEBUG>(ctx, A, beside_pme);
}

template <int RAD, bool VIRIAL, bool DEBUG>
static void launch_force_t(nb_ctx *ctx, const ForceArgs &A, bool beside_pme)
{
    if (ctx->built_group == 1) launch_force_1<RAD, VIRIAL, DEBUG>(ctx, A, beside_pme);
    else if (ctx->built_group == 4) launch_force_g<4, RAD, VIRIAL, DEBUG>(ctx, A);
    else launch_force_g<8, RAD, VIRIAL, DEBUG>(ctx, A);
}

// The packed constants of a parameter block.
static PairConst2 make_const2(const PairParams &P)
{
    auto twice = [](float v) {
        uint32_t b;
        memcpy(&b, &v, sizeof(b));
        return (f32x2)b << 32 | b;
    };
    PairConst2 C;
    C.rc2 = twice(P.rc2);
    C.rs2 = twice(P.rs2);
    C.sw_a = twice(P.sw_a);
    C.sw_b = twice(P.sw_b);
    C.neg_sw_c = twice(-P.sw_c);
    C.neg_alpha_half = twice(-P.alpha_half);
    C.a2_hi = twice(P.neg_a2_log2e);
    C.neg_a2_hi = twice(-P.neg_a2_log2e);
    C.neg_a2_lo = twice(-P.neg_a2_log2e_lo);
    C.two_a_sqpi = twice(P.two_a_sqpi);
    C.magic = twice(12582912.0f);
    C.one = twice(1.0f);
    C.neg_one = twice(-1.0f);
    C.neg_half = twice(-0.5f);
    C.neg_zero = twice(-0.0f);
    for (int k = 0; k <= kErfcDeg; ++k) C.erfc_c[k] = twice(P.erfc_c[k]);
    for (int k = 0; k <= kExp2Deg; ++k) C.exp2_c[k] = twice(P.exp2_c[k]);
    return C;
}

static ForceArgs make_args(nb_ctx *ctx)
{
    auto &d = ctx->d;
    ForceArgs A;
    memset(&A, 0, sizeof(A));
    A.sys = d.sys;
    A.counts = d.counts;
    A.work = d.counts + 3;
    A.xyzq = d.xyzq;
    A.tslot = d.tslot;
    A.perm = d.perm;
    A.clus_sys = d.clus_sys;
    A.grp = d.grp;
    A.glist = d.glist;
    A.glist_n = d.glist_n;
    A.gmask = d.gmask;
    A.pool8 = d.gmask + (mask_pool_base(ctx->clus_cap) - kOwnRecs8) * 8;
    A.cap = ctx->list_cap;
    A.K = ctx->K;
    A.lj_tab = d.lj_tab;
    A.rtab = d.rtab;
    A.sys_acc = d.sys_acc;
    A.status = d.status;
    A.dbg_n = d.dbg_n;
    A.dbg_ij = d.dbg_ij;
    A.dbg_cap = d.dbg_cap;
    A.P = ctx->pp;
    return A;
}

cudaError_t launch_pack(nb_ctx *ctx, const float *d_pos, const float *d_q, const int32_t *d_type, bool zero_sums)
{
    auto &d = ctx->d;
    const int tb = 256;
    const int S = (int)ctx->slot_cap;
    return launch_pdl(k_pack, dim3((S + tb - 1) / tb), dim3(tb), 0, ctx->stream, S, d.counts, d.perm, d.xyzq,
                      d.tslot, d_pos, d_q, d_type, d.sys, d.atom_sys, ctx->pp.n_types, d.status,
                      zero_sums ? d.facc : nullptr, zero_sums ? d.sys_acc : nullptr, kTaskVals * ctx->n_sys,
                      d.counts + 3);
}

cudaError_t launch_forces(nb_ctx *ctx, const float *d_pos, const float *d_q, const int32_t *d_type, float *d_F,
                          double *d_energy, double *d_virial, bool debug_pairs)
{
    auto &d = ctx->d;
    if (d_pos) {  // packs and zeroes the fixed-point sums
        cudaError_t e = launch_pack(ctx, d_pos, d_q, d_type, true);
        if (e != cudaSuccess) return e;
    } else {  // the debug pair export reuses the last packed values
        cudaMemsetAsync(d.sys_acc, 0, sizeof(long long) * kTaskVals * ctx->n_sys, ctx->stream);
        cudaMemsetAsync(d.facc, 0, sizeof(long long) * 3 * ctx->slot_cap, ctx->stream);
        cudaMemsetAsync(d.counts + 3, 0, sizeof(int), ctx->stream);
    }
    // smooth PME: forked onto its own stream so that it overlaps the
    // short-range kernel; joined back before the unpack reads its sums
    const bool pme = ctx->pme && d_pos && !debug_pairs;
    if (pme) {
        cudaError_t e = launch_pme_fork(ctx, d_pos, d_q);
        if (e != cudaSuccess) return e;
    }
    return launch_forces_packed(ctx, d_F, d_energy, d_virial, debug_pairs, pme, false);
}

cudaError_t launch_forces_packed(nb_ctx *ctx, float *d_F, double *d_energy, double *d_virial, bool debug_pairs,
                                 bool pme, bool beside_pme)
{
    auto &d = ctx->d;
    ForceArgs A = make_args(ctx);
    A.C = make_const2(ctx->pp);
    A.facc = d.facc;
    const bool ewald = ctx->pp.ewald != 0;
    const bool virial = d_virial != nullptr;
    const bool prof = ctx->profiling && ctx->prof_n < (int)ctx->prof_ev.size() / 2;
    if (prof) cudaEventRecord(ctx->prof_ev[2 * ctx->prof_n], ctx->stream);
    if (debug_pairs) {  // the pair set does not depend on the radial functions
        if (ewald) launch_force_t<1, false, true>(ctx, A, beside_pme);
        else launch_force_t<0, false, true>(ctx, A, beside_pme);
    } else if (ctx->tab_n > 0) {
        if (virial) launch_force_t<2, true, false>(ctx, A, beside_pme);
        else launch_force_t<2, false, false>(ctx, A, beside_pme);
    } else if (ewald) {
        if (virial) launch_force_t<1, true, false>(ctx, A, beside_pme);
        else launch_force_t<1, false, false>(ctx, A, beside_pme);
    } else {
        if (virial) launch_force_t<0, true, false>(ctx, A, beside_pme);
        else launch_force_t<0, false, false>(ctx, A, beside_pme);
    }
    if (prof) {
        cudaEventRecord(ctx->prof_ev[2 * ctx->prof_n + 1], ctx->stream);
        ctx->prof_n++;
    }
    if (pme) {
        cudaError_t e = launch_pme_join(ctx);
        if (e != cudaSuccess) return e;
    }
    if (d_F) {  // else the caller's next kernel reads the fixed-point sums (the MD step)
        const int tb = kUnpackThreads;
        const int S = (int)ctx->n_atoms;
        const int blocks = std::max(1, std::min((S + tb - 1) / tb, 16 * ctx->num_sms));
        double *en = debug_pairs ? nullptr : d_energy;
        double *vi = debug_pairs ? nullptr : d_virial;
        const long long *pf = pme ? pme_forces_acc(ctx) : nullptr, *ps = pme ? pme_sums_acc(ctx) : nullptr;
        const double pself = pme ? pme_self_coef(ctx) : 0.0;
        if (virial)
            launch_pdl_split(pme_beside(ctx), k_unpack_forces<true>, dim3(blocks), dim3(tb), 0, ctx->stream, S, d.counts, d.inv, d.facc, d_F,
                       d.xyzq, d.atom_sys, d.sys_acc, ctx->n_sys, en, vi, pf, ps, pself);
        else
            launch_pdl_split(pme_beside(ctx), k_unpack_forces<false>, dim3(blocks), dim3(tb), 0, ctx->stream, S, d.counts, d.inv, d.facc,
                       d_F, d.xyzq, d.atom_sys, d.sys_acc, ctx->n_sys, en, vi, pf, ps, pself);
    }
    return cudaGetLastError();
}

size_t adjoint_smem_bytes(int T, int G)
{
    return (size_t)T * T * 32 + align16((size_t)T * T * 8) + (size_t)kAdjWarps * adj_warp_bytes(G);
}

template <int G, int RAD>
static void launch_adjoint_g(nb_ctx *ctx, const ForceArgs &A)
{
    const size_t smem = adjoint_smem_bytes(A.P.n_types, G);
    static std::atomic<unsigned long long> optin{0};
    smem_optin_once(k_adjoint<G, RAD>, ctx->device, 220 * 1024, optin);
    int resident = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_adjoint<G, RAD>, kAdjWarps * 32, smem);
    const int parts = ctx->tune.list_split > 0 ? ctx->tune.list_split : kDefaultListSplit;
    const int blocks = ctx->num_sms * std::max(1, resident);
    launch_pdl(k_adjoint<G, RAD>, dim3(blocks), dim3(kAdjWarps * 32), smem, ctx->stream, A, parts, blocks * kAdjWarps);
}

template <int RAD>
static void launch_adjoint_1(nb_ctx *ctx, const ForceArgs &A)
{
    const size_t smem = adjoint1_smem_bytes(A.P.n_types);
    static std::atomic<unsigned long long> optin{0};
    smem_optin_once(k_adjoint1<RAD>, ctx->device, 220 * 1024, optin);
    int resident = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_adjoint1<RAD>, kAdjWarps * 32, smem);
    const int parts = ctx->tune.list_split > 0 ? ctx->tune.list_split : kDefaultListSplit;
    const int blocks = ctx->num_sms * std::max(1, resident);
    launch_pdl(k_adjoint1<RAD>, dim3(blocks), dim3(kAdjWarps * 32), smem, ctx->stream, A, parts, blocks * kAdjWarps);
}

template <int RAD>
static void launch_adjoint_t(nb_ctx *ctx, const ForceArgs &A)
{
    if (ctx->built_group == 1) launch_adjoint_1<RAD>(ctx, A);
    else if (ctx->built_group == 4) launch_adjoint_g<4, RAD>(ctx, A);
    else launch_adjoint_g<8, RAD>(ctx, A);
}

size_t force_smem_for(int T, int scap, int K)
{
    (void)scap;  // unused: the kernels stage per batch of entries
    (void)K;     // the exclusion masks are built by the list kernel
    return std::max(tile_smem_bytes(T, kMaxGroup), adjoint_smem_bytes(T, kMaxGroup));
}

cudaError_t launch_adjoint_tile(nb_ctx *ctx, const double *d_dLdE, float *d_dpos, float *d_dq)
{
    auto &d = ctx->d;
    ForceArgs A = make_args(ctx);
    A.gslot = d.gslot;
    A.dLdE = d_dLdE;
    A.lj_d = d.lj_d;
    A.tab_acc = d.tab_grad;
    A.gacc = d.gacc;
    if (ctx->pp.ewald) launch_adjoint_t<1>(ctx, A);
    else launch_adjoint_t<0>(ctx, A);
    const int tb = 256;
    const int S = (int)ctx->slot_cap;
    return launch_pdl(k_unpack_adjoint, dim3((S + tb - 1) / tb), dim3(tb), 0, ctx->stream, S, d.counts, d.perm,
                      d.gacc, d_dpos, d_dq);
}

// Test export of the pair arithmetic (nb_debug_pair_terms): pair k of the
// given lists evaluated by eval_pair, as k_force<G> does it (k_force1's packed
// form has the same bits; unit weights, d = x_j - x_i as given); out[2k] = (E_LJ, E_Coul, r2, 0),
// out[2k + 1] = the force on j.
template <int RAD>
__global__ void k_debug_pair_terms(PairParams P, const float4 *__restrict__ lj_tab, const float4 *__restrict__ rtab,
                                   long long n, const float4 *__restrict__ xi, const float4 *__restrict__ xj,
                                   const int *__restrict__ ti, const int *__restrict__ tj, float4 *__restrict__ out)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float4 a = xi[k], b = xj[k];
    const float4 ab = lj_tab[ti[k] * P.n_types + tj[k]];
    float4 lj4[2];  // one type pair: (A, B, 12 A, 6 B), then the remainders at lj4 + n_types^2
    lj4[0] = make_float4(ab.x, ab.y, 12.0f * ab.x, 6.0f * ab.y);
    lj4[1] = make_float4(ab.z, ab.w, 0.0f, 0.0f);
    float dx, dy, dz;
    const float r2 = disp_r2(b.x, b.y, b.z, a.x, a.y, a.z, dx, dy, dz);
    Acc acc = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    float fjx = 0.0f, fjy = 0.0f, fjz = 0.0f;
    PairParams P1 = P;
    P1.n_types = 1;  // the one-pair table above
    eval_pair<RAD, false>(P1, lj4, rtab, 0, a.w * P.ke, true, dx, dy, dz, r2, b.w, 0, false, acc, fjx, fjy, fjz);
    out[2 * k] = make_float4(acc.elj, acc.ec, r2, 0.0f);
    out[2 * k + 1] = make_float4(fjx, fjy, fjz, 0.0f);
}

cudaError_t launch_debug_pair_terms(nb_ctx *ctx, long long n, const float4 *xi, const float4 *xj, const int *ti,
                                    const int *tj, float4 *out)
{
    const int tb = 128;
    const unsigned g = (unsigned)((n + tb - 1) / tb);
    const PairParams &P = ctx->pp;
    if (ctx->tab_n > 0)
        k_debug_pair_terms<2><<<g, tb, 0, ctx->stream>>>(P, ctx->d.lj_tab, ctx->d.rtab, n, xi, xj, ti, tj, out);
    else if (P.ewald)
        k_debug_pair_terms<1><<<g, tb, 0, ctx->stream>>>(P, ctx->d.lj_tab, ctx->d.rtab, n, xi, xj, ti, tj, out);
    else
        k_debug_pair_terms<0><<<g, tb, 0, ctx->stream>>>(P, ctx->d.lj_tab, ctx->d.rtab, n, xi, xj, ti, tj, out);
    return cudaGetLastError();
}

}  // namespace acenb
