// Short-range non-bonded forces: Debye-screened Coulomb (Sec. II.A, Eq. 2)
// plus screened LJ (Sec. II.B, Eq. 8) with charge-scaled LJ sizes (Eq. 11),
// LJ excluded inside a native fragment (Sec. II.B), cut off at r_cut with the
// energy shifted to zero there.
//
// Work decomposition (Newton's third law, every unordered pair once):
//   * atoms are cell-sorted into clusters of 8; up to 8 consecutive clusters
//     of one cell form a super-cluster (SC);
//   * a list kernel tests, per SC and half-shell cell, every j-cluster's
//     bounding box against the SC's 8 i-cluster boxes, and for the clusters
//     in range every i-atom against the j-cluster's box; each j-cluster with
//     an i-atom in range becomes an entry (j-cluster, shift, 64-bit i-atom
//     mask), contiguous per SC and cut into chunks of kChunk entries;
//   * a warp of the force kernel owns one chunk at a time (dynamic scheduling
//     through an atomic counter);
//   * mixed precision (k_pair): lane (tx = lane & 7, ty = lane >> 3) keeps the
//     force of atom tx of every i-cluster of the SC in registers and evaluates
//     it against j-atoms ty and ty + 4 of the entry's j-cluster in the two
//     halves of packed FP32 operations, one 8 x 8 cluster tile at a time;
//   * FP64 (k_pair64) and the analyses (k_walk): the SC's atoms (and, in
//     k_pair64, per-(atom, lane row) i-force partials) live in shared memory;
//     a lane takes atoms ty, ty+4 of the entry's j-cluster and, tile by tile,
//     the next i-cluster whose atom tx is in the mask (its own queue), so a lane
//     column always sees the same slots in the same order and the rows it
//     touches never share a bank with another column's;
//   * at the step of a Verlet-buffered build the evaluation also tests every
//     pair against r_cut + skin and drops from the mask the i-clusters (FP64:
//     i-atoms) with no j-atom in range (exact for the list's lifetime), and
//     clears the entry's fragment flag when no pair in range lies within one
//     fragment;
//   * forces are summed in FP32 (or FP64) within one chunk for the i side
//     and one (SC, j-cluster) entry for the j side, then converted
//     once to 64-bit fixed point (2^-32 kJ/mol/nm): the per-atom totals are
//     exact integer sums, identical for every launch shape and schedule.
#include <algorithm>
#include <type_traits>

#include "bonded_terms.cuh"
#include "md_internal.cuh"

namespace mdg {

template <bool FP64>
struct Prec;

template <>
struct Prec<false> {
    using T = float;
    using T4 = float4;         // global packed position + charge
    using S4 = float4;         // shared-memory copy
    using C2 = float2;         // 6 c6, 6 c12
    static __device__ __forceinline__ T4 pos(const Params& p, int slot) { return p.xq[slot]; }
    // single MUFU operations (arguments are far from the denormal range)
    static __device__ __forceinline__ T rsq(T x)
    {
        T y;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
        return y;
    }
    static __device__ __forceinline__ T expneg(T x)
    {
        T y;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * -1.4426950408889634f));
        return y;
    }
    static __device__ __forceinline__ T exp2_(T x)
    {
        T y;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
        return y;
    }
    static __device__ __forceinline__ long long fix(T v) { return __float2ll_rn(v * 4294967296.0f); }
    static __device__ __forceinline__ bool fix_ok(T v) { return fabsf(v) < 1.0737418e9f; }
    static __device__ __forceinline__ const C2* table(const Params& p) { return p.lj_f; }
    static __device__ __forceinline__ S4 mk(T a, T b, T c, T d) { return make_float4(a, b, c, d); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return __fmaf_rn(a, b, c); }
};

template <>
struct Prec<true> {
    using T = double;
    using T4 = double4_32a;
    using S4 = double4_16a;
    using C2 = double2;        // -6 c6, -ln2 c12
    static __device__ __forceinline__ T4 pos(const Params& p, int slot) { return p.xq64[slot]; }
    static __device__ __forceinline__ T rsq(T x) { return rsqrt(x); }   // within 1 ulp, without a division
    static __device__ __forceinline__ T expneg(T x) { return exp(-x); }
    static __device__ __forceinline__ T exp2_(T x) { return exp2(x); }
    static __device__ __forceinline__ long long fix(T v) { return __double2ll_rn(v * 4294967296.0); }
    static __device__ __forceinline__ bool fix_ok(T v) { return fabs(v) < 1.073741824e9; }
    static __device__ __forceinline__ const C2* table(const Params& p) { return p.lj_d; }
    static __device__ __forceinline__ S4 mk(T a, T b, T c, T d) { S4 s; s.x = a; s.y = b; s.z = c; s.w = d; return s; }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return __fma_rn(a, b, c); }
};

// Rows kSCAtoms + tx are far-away stand-ins for lane column tx once its queue of
// i-clusters is used up (FP64 kernel and analyses).
constexpr int kFiRow = kSCAtoms + kClusterSize;
// per-warp shared-memory layout of the FP64 kernel
constexpr int kGroup64 = 4;                  // entries whose pairs in range are evaluated together
template <bool HYB>
struct Hyb64 {};
template <>
struct Hyb64<true> {                         // hybrid electrostatics (Eqs. 4-7)
    double4_16a ih[kSCAtoms];                // (f/2) G_i, (f/2) q_i, q_i of the SC atoms
    double jG[kChunk * kClusterSize];        // G_j of the chunk's j-atoms
};
template <bool HYB>
struct Warp64 {
    double4_16a ix[kSCAtoms];                // x, y, z, f*q of the SC atoms
    double4_16a fi[4 * kSCAtoms];            // [ty][atom] force (+energy)
    double4_16a jx[kChunk * kClusterSize];   // the chunk's j-atoms, shifted: x, y, z, q
    float4 ixf[kFiRow];                      // FP32 positions of the SC atoms (and stand-ins)
    float4 jxf[kChunk * kClusterSize];       // and of the j-atoms
    double fj[6 * kGroup64][32];             // j forces of each lane: [entry of the group][j-atom of the lane][component]
    double jqk[kChunk * kClusterSize];       // q kappa of the j-atoms
    int2 it[kFiRow];                         // LJ row byte offset, fragment
    int2 jt[kChunk * kClusterSize];          // LJ column byte offset, fragment of the j-atoms
    unsigned kq[kGroup64][32];               // each lane's queue of i-clusters
    PairEntry ent[kChunk];                   // the chunk's list entries
    Hyb64<HYB> hy;
};

// Hybrid electrostatics of one pair (Sec. II.A, Eqs. 4-7; the reading is in
// include/md.h): an ion's potential is q/r + c1 - c2 r^2 inside its
// transition radius r' and G e^{-kappa r}/r outside, and the pair's Coulomb
// energy f (q_j phi_i + q_i phi_j) / 2.
template <typename T>
struct HybArg {
    T hGi, hqi, qi;          // (f/2) G_i, (f/2) q_i, q_i
    T Gj, Gjk;               // G_j, G_j kappa
    T kap, c2, rpm2, hf;     // kappa, c2, (largest r')^2 of the replica, f/2
    const HybQ* rows;        // the replica's charge states
};

template <bool FP64>
__device__ __forceinline__ void red_fix(long long* dst, typename Prec<FP64>::T v, unsigned* err)
{
    if (!Prec<FP64>::fix_ok(v)) {
        atomicOr(err, ERR_OVERFLOW);
        return;
    }
    atomicAdd((unsigned long long*)dst, (unsigned long long)Prec<FP64>::fix(v));
}

// One FP64 pair, d = x_i - x_j; equal fragments drop the LJ part.  qjk = q_j *
// kappa, kl = -kappa log2(e).  The LJ table holds (-6 c6, -ln2 c12), so that
// t = kl r serves both the screening factor e^{-kappa r} = 2^t and the kappa r
// term of the LJ force (kappa r = -ln2 t).  The force on i is accumulated into
// (fx, fy, fz), the force on j into (fjx, fjy, fjz); with ENERGY the
// cutoff-shifted pair energy into u.
template <bool ENERGY, bool HYB>
__device__ __forceinline__ void pair64(const double4_16a& xi, int row_off, int fri, double xj, double yj, double zj, double qj,
                                       double qjk, int tsj_off, int frj, const unsigned char* __restrict__ lj_bytes, double kl,
                                       double rc2, double& fx, double& fy, double& fz, double& fjx, double& fjy, double& fjz,
                                       double& u, int& npair, double erc, double irc, const HybArg<double>& ha)
{
    using P = Prec<true>;
    using T = double;
    constexpr T kLn2 = T(0.69314718055994530942);
    const T dx = xi.x - xj, dy = xi.y - yj, dz = xi.z - zj;
    const T r2 = P::fma(dz, dz, P::fma(dy, dy, dx * dx));
    const bool in = r2 < rc2;
    const T rinv = in ? P::rsq(r2) : T(0);
    const double2 c = *reinterpret_cast<const double2*>(lj_bytes + row_off + tsj_off);
    const T rinv2 = rinv * rinv;
    const T rinv6 = rinv2 * rinv2 * rinv2;
    const T lj6 = fri == frj ? T(0) : rinv6;   // bonded in the native structure: no LJ
    const T r = r2 * rinv;
    const T t = kl * r;                         // -kappa r log2(e)
    const T e = P::exp2_(t);                    // e^{-kappa r}
    const T An = c.y * rinv6;                   // -ln2 c12/r^6
    const T Bn = P::fma(c.x, T(-kLn2 / 6), An); // -ln2 (c12/r^6 - c6)
    const T D6 = P::fma(An, T(-12 / kLn2), c.x);  // 12 c12/r^6 - 6 c6
    const T E1 = P::fma(t, Bn, D6);             // D6 + kappa r (c12/r^6 - c6)
    // f q_i q_j (1/r + kappa); hybrid, outside both transition radii:
    // (f/2)(G_i q_j + q_i G_j)(1/r + kappa)
    const T Cc = HYB ? P::fma(ha.hGi, P::fma(qj, rinv, qjk), ha.hqi * P::fma(ha.Gj, rinv, ha.Gjk))
                     : xi.w * P::fma(qj, rinv, qjk);
    const T S = P::fma(lj6, E1, Cc);
    T fs = S * (rinv2 * e);                     // F(r)/r
    if (HYB && in && r2 < ha.rpm2) {
        // inside some ion's transition radius: each ion's -phi' from its own form
        const HybQ& Ri = ha.rows[(int)ha.qi];
        const HybQ& Rj = ha.rows[(int)qj];
        const T rpi = Ri.rp, rpj = Rj.rp;
        const T Gj = ha.Gj;
        const T outf = e * P::fma(ha.kap, r, T(1)) * rinv2;   // e^{-kappa r} (1 + kappa r) / r^2
        const T fc2r = T(2) * ha.hf * ha.c2 * r;                // (f/2) 2 c2 r
        const T hmi = r < rpi ? P::fma(ha.hqi, rinv2, fc2r) : ha.hGi * outf;            // (f/2)(-phi_i')
        const T hmj = r < rpj ? P::fma(ha.hf * qj, rinv2, fc2r) : (ha.hf * Gj) * outf;  // (f/2)(-phi_j')
        fs = P::fma(lj6 * E1, rinv2 * e, P::fma(qj, hmi, ha.qi * hmj) * rinv);
    }
    const T nfs = -fs;
    fx = P::fma(fs, dx, fx); fy = P::fma(fs, dy, fy); fz = P::fma(fs, dz, fz);
    fjx = P::fma(nfs, dx, fjx); fjy = P::fma(nfs, dy, fjy); fjz = P::fma(nfs, dz, fjz);
    if (ENERGY) {
        if (in) {
            const T irc6 = irc * irc * irc * irc * irc * irc;
            const T lj_on = fri == frj ? T(0) : T(1);
            const T ulj = e * (lj6 * (Bn * T(-1 / kLn2))) - erc * lj_on * (c.y * T(-1 / kLn2) * irc6 + c.x * T(1.0 / 6.0)) * irc6;
            if (HYB) {
                const HybQ& Ri = ha.rows[(int)ha.qi];
                const HybQ& Rj = ha.rows[(int)qj];
                const T rpi = Ri.rp, rpj = Rj.rp;
                const T c1i = Ri.c1, c1j = Rj.c1;
                const T Gi = Ri.G;
                const T pci = Ri.phirc, pcj = Rj.phirc;
                const T cr2 = ha.c2 * r2;
                const T phi_i = r < rpi ? ha.qi * rinv + c1i - cr2 : Gi * e * rinv;
                const T phi_j = r < rpj ? qj * rinv + c1j - cr2 : ha.Gj * e * rinv;
                u += ulj + ha.hf * (qj * (phi_i - pci) + ha.qi * (phi_j - pcj));
            } else {
                const T qq = xi.w * qj;
                u += ulj + e * qq * rinv - erc * qq * irc;
            }
            npair += 1;
        }
    }
}

// Cluster-pair list.  Every j-cluster whose bounding box comes within
// r_cut + skin of at least one of a super-cluster's (SC's) i-cluster boxes gets
// an entry (j-cluster, half-shell index, mask of the i-atoms of those clusters
// that lie within r_cut + skin of the j-cluster's box).  An SC's entries are
// contiguous, in half-shell order and by j-cluster within a cell, and cut into
// chunks of kChunk, the work items of the force kernel.  The j-clusters of an
// SC's 14 half-shell cells form one index range, swept 32 at a time with every
// lane busy (cell by cell would leave lanes idle and chain one load latency per
// cell).  Five kernels, the box tests with no block-level barrier:
//   k_list_count  a warp per (SC, part of its index range) item counts the
//                 entries of its part;
//   k_list_scan_* three kernels sum each SC's parts and scan the totals into
//                 entry and chunk offsets (and flag a list too small for them);
//   k_list_write  a warp per item repeats the box tests in the same rounding
//                 and writes its entries from its offset (the SC's plus the
//                 counts of the SC's earlier parts); the SC's first item writes
//                 the SC's chunk descriptors.
// An SC's range is split into 1, 2, 7 or 14 parts (list_parts): as few as keep
// every warp of the grid busy, so that a system of many SCs stages each SC once
// and a smaller one still spreads over the GPU.  Systems of few SCs take
// k_list_fused below instead (list_in_one_kernel).
// Whether the list of these parameters holds light chunks apart (k_list_fused, lists
// that serve several steps).  The kernels that find them (LIGHT) cost large systems
// and single calls more than they give: 500,001 atoms 768 us without, 786 with.
constexpr int kLightScs = 8192;
__host__ __forceinline__ bool has_light(const Params& p) { return p.list_fused && p.sc_cap <= kLightScs && p.xr != nullptr; }
// The list's chunks and how many of them are heavy.
__device__ __forceinline__ int2 chunk_counts(const Params& p)
{
    const int n = min(p.counters[7], p.chunk_cap);
    return make_int2(n, max(n - p.counters[5], 0));
}
// Where chunk `item` of the list is: the heavy ones from the start of the table, the
// light ones (k_list_fused) from its end; -1 beyond the last.
__device__ __forceinline__ int chunk_at(const Params& p, int item, int2 n)
{
    return item >= n.x ? -1 : (item < n.y ? item : p.chunk_cap - 1 - (item - n.y));
}

struct ListWarp {
    float4 lo[kSuperClusters], hi[kSuperClusters];   // the SC's i-cluster boxes (cell frame)
    int2 fr[kSuperClusters];                          // fragment range of each i-cluster
    float4 ip[kSCAtoms];                              // the SC's atoms, [cluster k][atom a] (write pass)
};

// An SC's cell, in the grid of its replica.
struct ListSC {
    int sc, fc, ncl, rr, cx, cy, cz;
};
__device__ __forceinline__ ListSC list_sc(const Params& p, int sc)
{
    ListSC s;
    s.sc = sc;
    const int c = p.sc_cell[sc];
    s.fc = p.sc_first[sc];
    s.ncl = p.sc_ncl[sc];
    int lo = 0, hi = p.n_rep - 1;   // replicas own contiguous cell ranges
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.grid_b[mid].cell_off <= c) lo = mid; else hi = mid - 1;
    }
    s.rr = lo;
    const Grid& g = p.grid_b[lo];
    const int local = c - g.cell_off;
    s.cx = local % g.dims[0];
    s.cy = (local / g.dims[0]) % g.dims[1];
    s.cz = local / (g.dims[0] * g.dims[1]);
    return s;
}

// Lane nb < 14: half-shell cell nb of the SC (its first j-cluster, its number
// of j-clusters, the clusters of the cells before it, its shift into the SC
// cell's frame); *total: the SC's j-clusters over the 14 cells.
struct ListCell {
    int jr0, n, pre;
    float Dx, Dy, Dz;
};
__device__ __forceinline__ ListCell list_cells(const Params& p, const ListSC& s, int lane, int* total)
{
    ListCell c{};
    if (lane < kHalfShell) {
        const Grid& g = p.grid_b[s.rr];
        int dx, dy, dz;
        half_shell(lane, dx, dy, dz);
        int ncx = s.cx + dx, ncy = s.cy + dy, ncz = s.cz + dz;
        bool valid = true;
        if (g.periodic) {
            ncx = ncx < 0 ? ncx + g.dims[0] : (ncx >= g.dims[0] ? ncx - g.dims[0] : ncx);
            ncy = ncy < 0 ? ncy + g.dims[1] : (ncy >= g.dims[1] ? ncy - g.dims[1] : ncy);
            ncz = ncz < 0 ? ncz + g.dims[2] : (ncz >= g.dims[2] ? ncz - g.dims[2] : ncz);
        } else {
            valid = ncx >= 0 && ncy >= 0 && ncz >= 0 && ncx < g.dims[0] && ncy < g.dims[1] && ncz < g.dims[2];
        }
        if (valid) {
            const int c2 = g.cell_off + ncx + g.dims[0] * (ncy + g.dims[1] * ncz);
            c.jr0 = lane == 0 ? s.fc : p.cell_pstart[c2] / kClusterSize;
            c.n = p.cell_pstart[c2 + 1] / kClusterSize - c.jr0;
        }
        c.Dx = (float)dx * g.edge_f[0];
        c.Dy = (float)dy * g.edge_f[1];
        c.Dz = (float)dz * g.edge_f[2];
    }
    int inc = c.n;   // inclusive scan over the 14 cells
    for (int o = 1; o < 16; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    c.pre = inc - c.n;
    *total = __shfl_sync(0xffffffffu, inc, kHalfShell - 1);
    return c;
}

// The cell (nb) and j-cluster of flat index idx of the SC's range (every lane
// takes part; lanes with idx out of range get some cell, unused).
__device__ __forceinline__ void list_locate(const ListCell& c, int idx, int& nb, int& jc, float& Dx, float& Dy,
                                            float& Dz)
{
    int lo = 0;   // the last cell whose first index is <= idx (cells of no cluster are skipped)
#pragma unroll
    for (int step = 8; step; step >>= 1) {
        const int cand = min(lo + step, kHalfShell - 1);
        if (__shfl_sync(0xffffffffu, c.pre, cand) <= idx) lo = cand;
    }
    nb = lo;
    jc = __shfl_sync(0xffffffffu, c.jr0, lo) + idx - __shfl_sync(0xffffffffu, c.pre, lo);
    Dx = __shfl_sync(0xffffffffu, c.Dx, lo);
    Dy = __shfl_sync(0xffffffffu, c.Dy, lo);
    Dz = __shfl_sync(0xffffffffu, c.Dz, lo);
}

// Largest of three floats in one instruction (max selects, so this equals
// fmaxf(c, fmaxf(a, b)) for the finite operands of the box tests).
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Mask of the SC's i-clusters whose boxes come within r_cut + skin of the
// j-cluster box [jl, jh] (already shifted into the SC's frame); in the SC's own
// cell (nb = 0) only i-clusters up to the j-cluster.  Explicit roundings, so
// that the count and the write pass reach the same masks.
__device__ __forceinline__ unsigned list_test(const ListWarp& w, int nb, int fc, int ncl, int jc, float4 jl,
                                              float4 jh, float rcb2)
{
    unsigned m = 0;
    const int kmax = nb == 0 ? min(ncl, jc - fc + 1) : ncl;
#pragma unroll 2
    for (int k = 0; k < kmax; ++k) {
        const float4 il = w.lo[k], ih = w.hi[k];
        const float gx = max3f(il.x - jh.x, jl.x - ih.x, 0.0f);
        const float gy = max3f(il.y - jh.y, jl.y - ih.y, 0.0f);
        const float gz = max3f(il.z - jh.z, jl.z - ih.z, 0.0f);
        if (__fmaf_rn(gz, gz, __fmaf_rn(gy, gy, __fmul_rn(gx, gx))) < rcb2) m |= 1u << k;
    }
    return m;
}

// Parts of an SC's index range: the fewest of 1, 2, 7, 14 with at least as
// many (SC, part) items as the grid has warps.
__device__ __forceinline__ int list_parts(int n_sc)
{
    const long long warps = (long long)gridDim.x * kListWarps;
    if ((long long)n_sc >= warps) return 1;
    if (2LL * n_sc >= warps) return 2;
    if (7LL * n_sc >= warps) return 7;
    return 14;
}

// The box of flat index idx (when idx < i1), shifted into the SC's frame.
struct ListJ {
    int nb, jc;
    unsigned m;
    float4 jl, jh;
};
__device__ __forceinline__ ListJ list_j(const Params& p, const ListWarp& w, const ListSC& s, const ListCell& c,
                                        int idx, int i1, float rcb2)
{
    ListJ j;
    float Dx, Dy, Dz;
    list_locate(c, idx, j.nb, j.jc, Dx, Dy, Dz);
    j.m = 0u;
    j.jl = j.jh = make_float4(0.f, 0.f, 0.f, 0.f);
    if (idx < i1) {
        const float4 lo = p.bb_lo[j.jc], hi = p.bb_hi[j.jc];
        j.jl = make_float4(lo.x + Dx, lo.y + Dy, lo.z + Dz, 0.0f);
        j.jh = make_float4(hi.x + Dx, hi.y + Dy, hi.z + Dz, 0.0f);
        j.m = list_test(w, j.nb, s.fc, s.ncl, j.jc, j.jl, j.jh, rcb2);
    }
    return j;
}

__global__ void __launch_bounds__(kListWarps * 32, 4) k_list_count(Params p)
{
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ ListWarp s_w[kListWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ListWarp& w = s_w[warp];
    if (*p.err & ERR_CELL) return;
    const int n_sc = p.counters[0];
    const int G = list_parts(n_sc);
    const float rcb = list_rlist_f(p) + kBBoxMargin;   // r_cut + Verlet skin
    const float rcb2 = rcb * rcb;
    for (int item = blockIdx.x * kListWarps + warp; item < n_sc * G; item += gridDim.x * kListWarps) {
        const int sc = item / G, gr = item - sc * G;
        const ListSC s = list_sc(p, sc);
        int total;
        const ListCell c = list_cells(p, s, lane, &total);
        const int i0 = (int)((long long)total * gr / G), i1 = (int)((long long)total * (gr + 1) / G);
        __syncwarp();
        if (lane < s.ncl) {
            w.lo[lane] = p.bb_lo[s.fc + lane];
            w.hi[lane] = p.bb_hi[s.fc + lane];
        }
        __syncwarp();
        int cnt = 0;
        for (int base = i0; base < i1; base += 64) {   // two batches in flight
            const ListJ ja = list_j(p, w, s, c, base + lane, i1, rcb2);
            const ListJ jb = list_j(p, w, s, c, base + 32 + lane, i1, rcb2);
            cnt += __popc(__ballot_sync(kFull, ja.m != 0u)) + __popc(__ballot_sync(kFull, jb.m != 0u));
        }
        if (lane == 0) p.list_cnt[sc * kHalfShell + gr] = cnt;
        if (gr == 0 && lane >= G && lane < kHalfShell) p.list_cnt[sc * kHalfShell + lane] = 0;   // unused parts
    }
}

// Exclusive scans of the SCs' entry counts and chunk counts, each SC's total
// summed over its parts first (stored in sc_tot).  One block's part: SCs
// [lo, hi) from the running totals base[0..1] of the SCs before lo; each warp
// owns a contiguous run of SCs and reads it 32 at a time.  Leaves the block's
// totals in s_tot / s_base (warp 31's base plus total).  WRITE = false: the
// totals (and sc_tot) only.
template <bool WRITE>
__device__ __forceinline__ void scan_scs(const Params& p, int lo, int hi, const int base[2], int (*s_tot)[2],
                                         int (*s_base)[2])
{
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int kWarps = 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int run = ((hi - lo + kWarps - 1) / kWarps + 31) & ~31;
    const int s_lo = min(lo + warp * run, hi), s_hi = min(s_lo + run, hi);
    int te = 0, tc = 0;
    for (int s = s_lo + lane; s < s_hi; s += 32) {
        int t = 0;
        if (!WRITE) {
#pragma unroll
            for (int k = 0; k < kHalfShell; ++k) t += p.list_cnt[s * kHalfShell + k];
            p.sc_tot[s] = t;
        } else {
            t = p.sc_tot[s];
        }
        te += t;
        tc += (t + kChunk - 1) / kChunk;
    }
    for (int o = 16; o; o >>= 1) {
        te += __shfl_xor_sync(kFull, te, o);
        tc += __shfl_xor_sync(kFull, tc, o);
    }
    if (lane == 0) { s_tot[warp][0] = te; s_tot[warp][1] = tc; }
    __syncthreads();
    if (warp == 0) {
        int ie = s_tot[lane][0], ic = s_tot[lane][1];
        for (int o = 1; o < 32; o <<= 1) {
            const int ue = __shfl_up_sync(kFull, ie, o), uc = __shfl_up_sync(kFull, ic, o);
            if (lane >= o) { ie += ue; ic += uc; }
        }
        s_base[lane][0] = base[0] + ie - s_tot[lane][0];
        s_base[lane][1] = base[1] + ic - s_tot[lane][1];
    }
    __syncthreads();
    if (!WRITE) return;
    int be = s_base[warp][0], bc = s_base[warp][1];
    for (int g0 = s_lo; g0 < s_hi; g0 += 32) {
        const int s = g0 + lane;
        const int t = s < s_hi ? p.sc_tot[s] : 0;
        const int ch = (t + kChunk - 1) / kChunk;
        int ie = t, ic = ch;
        for (int o = 1; o < 32; o <<= 1) {
            const int ue = __shfl_up_sync(kFull, ie, o), uc = __shfl_up_sync(kFull, ic, o);
            if (lane >= o) { ie += ue; ic += uc; }
        }
        if (s < s_hi) {
            p.sc_eoff[s] = be + ie - t;
            p.sc_coff[s] = bc + ic - ch;
        }
        be += __shfl_sync(kFull, ie, 31);
        bc += __shfl_sync(kFull, ic, 31);
    }
}

// The list's totals into counters[6] (entries) and counters[7] (chunks),
// ERR_LIST when the list is too small for them.
__device__ __forceinline__ void scan_scs_finish(const Params& p, long long E, long long Cn)
{
    p.counters[6] = (int)min(E, (long long)0x7fffffff);
    p.counters[7] = (int)min(Cn, (long long)0x7fffffff);
    p.counters[2] = 0;   // work counter of the force kernel
    if (E > p.pl_cap || Cn > p.chunk_cap) atomicOr(p.err, ERR_LIST);
}

// Each CTA sums its range; one CTA scans the sums (and finishes);
// each CTA scans its range from its base (p.scan_tmp: [CTA][2]).
__device__ __forceinline__ void sc_cta_range(int n, int& lo, int& hi)
{
    const int per = ((n + (int)gridDim.x - 1) / (int)gridDim.x + 31) & ~31;
    lo = min((int)blockIdx.x * per, n);
    hi = min(lo + per, n);
}
__global__ void __launch_bounds__(1024) k_list_scan_sums(Params p)
{
    __shared__ int s_tot[32][2], s_base[32][2];
    const int n = (*p.err & ERR_CELL) ? 0 : p.counters[0];
    int lo, hi;
    sc_cta_range(n, lo, hi);
    const int zero[2] = {0, 0};
    scan_scs<false>(p, lo, hi, zero, s_tot, s_base);
    if (threadIdx.x == 0)
        for (int k = 0; k < 2; ++k) p.scan_tmp[2 * blockIdx.x + k] = s_base[31][k] + s_tot[31][k];
}
__global__ void __launch_bounds__(1024) k_list_scan_top(Params p, int n_ctas)
{
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ long long s_w[32][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    long long v[2] = {0, 0}, inc[2];
    if ((int)threadIdx.x < n_ctas)
        for (int k = 0; k < 2; ++k) v[k] = p.scan_tmp[2 * threadIdx.x + k];
    for (int k = 0; k < 2; ++k) inc[k] = v[k];
    for (int o = 1; o < 32; o <<= 1)
        for (int k = 0; k < 2; ++k) {
            const long long u = __shfl_up_sync(kFull, inc[k], o);
            if (lane >= o) inc[k] += u;
        }
    if (lane == 31)
        for (int k = 0; k < 2; ++k) s_w[warp][k] = inc[k];
    __syncthreads();
    if (warp == 0) {
        long long w[2], wi[2];
        for (int k = 0; k < 2; ++k) w[k] = wi[k] = s_w[lane][k];
        for (int o = 1; o < 32; o <<= 1)
            for (int k = 0; k < 2; ++k) {
                const long long u = __shfl_up_sync(kFull, wi[k], o);
                if (lane >= o) wi[k] += u;
            }
        for (int k = 0; k < 2; ++k) s_w[lane][k] = wi[k] - w[k];
        if (lane == 31) scan_scs_finish(p, wi[0], wi[1]);
    }
    __syncthreads();
    if ((int)threadIdx.x < n_ctas)
        for (int k = 0; k < 2; ++k) p.scan_tmp[2 * threadIdx.x + k] = (int)min(s_w[warp][k] + inc[k] - v[k], (long long)0x7fffffff);
}
__global__ void __launch_bounds__(1024) k_list_scan_apply(Params p)
{
    __shared__ int s_tot[32][2], s_base[32][2];
    const int n = (*p.err & ERR_CELL) ? 0 : p.counters[0];
    int lo, hi;
    sc_cta_range(n, lo, hi);
    const int base[2] = {p.scan_tmp[2 * blockIdx.x], p.scan_tmp[2 * blockIdx.x + 1]};
    scan_scs<true>(p, lo, hi, base, s_tot, s_base);
}

// Entry of one j-cluster: the i-atoms of the clusters in range that lie within
// r_cut + skin of the j-cluster's box (padding slots are far away), as a
// column-major mask (bit a*8 + k: atom a of i-cluster k), and whether an
// i-cluster in range may share a fragment with it.  The i-atoms are broadcast
// reads of the staged SC.
__device__ __forceinline__ uint4 list_entry(const Params& p, const ListWarp& w, const ListJ& j, unsigned any_m,
                                            float rcb2)
{
    const int2 jfr = j.m ? p.bb_frag[j.jc] : make_int2(0, 0);
    unsigned mlo = 0u, mhi = 0u;
    bool share = false;
#pragma unroll
    for (int k = 0; k < kSuperClusters; ++k) {
        if (!((any_m >> k) & 1u)) continue;   // no lane has i-cluster k in range
        const bool kin = (j.m >> k) & 1u;
        unsigned klo = 0u, khi = 0u;   // column k's bits, kept only if cluster k is in range
#pragma unroll
        for (int a = 0; a < kClusterSize; ++a) {
            const float4 xi = w.ip[k * kClusterSize + a];
            const float gx = max3f(xi.x - j.jh.x, j.jl.x - xi.x, 0.0f);
            const float gy = max3f(xi.y - j.jh.y, j.jl.y - xi.y, 0.0f);
            const float gz = max3f(xi.z - j.jh.z, j.jl.z - xi.z, 0.0f);
            const bool in = __fmaf_rn(gz, gz, __fmaf_rn(gy, gy, __fmul_rn(gx, gx))) < rcb2;
            if (a < 4) klo |= (in ? 1u : 0u) << (a * 8 + k);
            else khi |= (in ? 1u : 0u) << ((a - 4) * 8 + k);
        }
        if (kin) {
            mlo |= klo;
            mhi |= khi;
        }
        const int2 ifr = w.fr[k];
        share |= kin && !(ifr.y < jfr.x || jfr.y < ifr.x);
    }
    return make_uint4((unsigned)j.jc, (unsigned)j.nb | (share ? kEntryExcl : 0u), mlo, mhi);
}

// The SC's atoms in slot order (cluster k, atom a); absent clusters far away.
__device__ __forceinline__ void list_stage_atoms(const Params& p, ListWarp& w, const ListSC& s, int t, int n_threads)
{
    for (int a = t; a < kSCAtoms; a += n_threads) {
        float4 v = make_float4(1.0e6f, 1.0e6f, 1.0e6f, 0.0f);
        if ((a >> 3) < s.ncl) {
            const int slot = s.fc * kClusterSize + a;
            if (p.precision == 0) {
                v = p.xq[slot];
            } else {
                const double4_32a x = p.xq64[slot];
                v = make_float4((float)x.x, (float)x.y, (float)x.z, 0.0f);
            }
        }
        w.ip[a] = v;
    }
}

__global__ void __launch_bounds__(kListWarps * 32, 4) k_list_write(Params p)
{
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ ListWarp s_w[kListWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ListWarp& w = s_w[warp];
    if (*p.err & (ERR_CELL | ERR_LIST)) return;
    const int n_sc = p.counters[0];
    const int G = list_parts(n_sc);
    const float rcb = list_rlist_f(p) + kBBoxMargin;
    const float rcb2 = rcb * rcb;
    for (int item = blockIdx.x * kListWarps + warp; item < n_sc * G; item += gridDim.x * kListWarps) {
        const int sc = item / G, gr = item - sc * G;
        const int tot = p.sc_tot[sc];
        if (tot == 0) continue;
        const ListSC s = list_sc(p, sc);
        const int e0 = p.sc_eoff[sc], c0 = p.sc_coff[sc];
        if (gr == 0)
            for (int t = lane; t * kChunk < tot; t += 32)
                p.pl_chunk[c0 + t] = make_int4(s.fc, e0 + t * kChunk, min(kChunk, tot - t * kChunk) | (s.ncl << 16), s.rr);
        // this item's first entry: the SC's offset plus the counts of its earlier parts
        const int cnt_l = lane < G ? p.list_cnt[sc * kHalfShell + lane] : 0;
        int pre = lane < gr ? cnt_l : 0;
        for (int o = 16; o; o >>= 1) pre += __shfl_xor_sync(kFull, pre, o);
        const int mine = __shfl_sync(kFull, cnt_l, gr);
        if (mine == 0) continue;
        int total;
        const ListCell c = list_cells(p, s, lane, &total);
        const int i0 = (int)((long long)total * gr / G), i1 = (int)((long long)total * (gr + 1) / G);
        __syncwarp();
        if (lane < s.ncl) {
            w.lo[lane] = p.bb_lo[s.fc + lane];
            w.hi[lane] = p.bb_hi[s.fc + lane];
            w.fr[lane] = p.bb_frag[s.fc + lane];
        }
        list_stage_atoms(p, w, s, lane, 32);
        __syncwarp();
        int off = e0 + pre;
        const int end = off + mine;
        for (int base = i0; base < i1; base += 32) {
            const ListJ j = list_j(p, w, s, c, base + lane, i1, rcb2);
            const unsigned bal = __ballot_sync(kFull, j.m != 0u);
            const int at = off + __popc(bal & ((1u << lane) - 1u));
            const uint4 e = list_entry(p, w, j, __reduce_or_sync(kFull, j.m), rcb2);
            if (j.m && at < end) p.pl[at] = e;
            off += __popc(bal);
        }
        // both passes see the same boxes and round identically, so `off` ends at
        // `end`; should it fall short, pad with empty entries (a real cluster, no
        // i-atom in range) rather than leave slots unwritten
        for (int at = off + lane; at < end; at += 32) p.pl[at] = make_uint4((unsigned)s.fc, 0u, 0u, 0u);
    }
}

// The same list in one kernel, for systems of few SCs (list_in_one_kernel): a block
// per SC, its 8 warps sharing the SC's index range.  Each warp keeps the
// j-clusters it found in range (compacted in shared memory, kFound of them; a
// warp that finds more repeats the box tests), the block adds up its warps'
// counts and reserves the SC's entries and chunks with one atomic each.  An
// SC's entries and chunks are those of the kernels above; only where they
// lie in the list follows the order of the atomics, which no sum depends on.
// Latency-bound: what the kernels above spend on their launches, on staging the
// SC once per part and pass, and on entries of j-clusters out of range is saved.
// Count, scan and write against this kernel, per build: 8,005 atoms (unbuffered)
// 20.1 -> 8.9 us, 12,297 atoms 23.6 -> 11.6, 30,000 atoms 31.9 -> 17.3, 199,773 atoms
// of protein crystal 111 -> 80.
//
// ORDER (buffered lists of up to kLightScs): the chunks of fewer than kLightTiles
// tiles (i-clusters in range of an entry, before trimming) go to the end of the chunk
// table, from its last element down, and are taken last (chunk_at): a force kernel's
// warps then end within a light chunk's time of one another instead of a heavy
// chunk's (of 63 us for 30,000 atoms the warps idled 11 on average).  Per launch
// 30,000 atoms 63.0 -> 60.0 us, 45,005 atoms 66.6 -> 63.2, 12,003 with hybrid
// screening 41.1 -> 39.1, FP64 forces of 30,000 atoms 1,628 -> 1,550, for 0.5 us more
// of list building; with 24, 40 and 48 tiles 30,000 atoms take 61, 60.8 and 61.2.  A
// list used once does not pay for it: of the 1.0 us that 8,005 atoms gain per launch
// a build at every step takes 0.6, and a single call on 12,297 atoms is 2 % slower.
constexpr int kLightTiles = 32;
constexpr int kTileChunks = 256;   // chunks of an SC whose tiles are counted; later ones count as heavy
constexpr int kFound = 128;
template <bool ORDER>
__global__ void __launch_bounds__(kListWarps * 32, 4) k_list_fused(Params p)
{
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ ListWarp w;
    __shared__ uint2 s_found[kListWarps][kFound];   // (j-cluster, half-shell index | i-cluster mask << 8)
    __shared__ int s_cnt[kListWarps], s_e0, s_c0, s_tiles[ORDER ? kTileChunks : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (*p.err & ERR_CELL) return;
    const int n_sc = p.counters[0];
    const float rcb = list_rlist_f(p) + kBBoxMargin;
    const float rcb2 = rcb * rcb;
    if (blockIdx.x == 0 && threadIdx.x == 0) p.counters[2] = 0;   // work counter of the force kernel
    for (int sc = blockIdx.x; sc < n_sc; sc += gridDim.x) {
        const ListSC s = list_sc(p, sc);
        int total;
        const ListCell c = list_cells(p, s, lane, &total);
        __syncthreads();   // the previous SC's reads are done
        if ((int)threadIdx.x < s.ncl) {
            w.lo[threadIdx.x] = p.bb_lo[s.fc + threadIdx.x];
            w.hi[threadIdx.x] = p.bb_hi[s.fc + threadIdx.x];
            w.fr[threadIdx.x] = p.bb_frag[s.fc + threadIdx.x];
        }
        list_stage_atoms(p, w, s, threadIdx.x, blockDim.x);
        if constexpr (ORDER)
            for (int t = threadIdx.x; t < kTileChunks; t += blockDim.x) s_tiles[t] = 0;
        __syncthreads();
        const int i0 = (int)((long long)total * warp / kListWarps), i1 = (int)((long long)total * (warp + 1) / kListWarps);
        int cnt = 0;
        for (int base = i0; base < i1; base += 32) {
            const ListJ j = list_j(p, w, s, c, base + lane, i1, rcb2);
            const unsigned bal = __ballot_sync(kFull, j.m != 0u);
            const int at = cnt + __popc(bal & ((1u << lane) - 1u));
            if (j.m && at < kFound) s_found[warp][at] = make_uint2((unsigned)j.jc, (unsigned)j.nb | (j.m << 8));
            cnt += __popc(bal);
        }
        if (lane == 0) s_cnt[warp] = cnt;
        __syncthreads();
        if constexpr (ORDER) {
            int pre = 0, tot = 0;
            bool counted = true;
            for (int k = 0; k < kListWarps; ++k) {
                if (k < warp) pre += s_cnt[k];
                tot += s_cnt[k];
                counted &= s_cnt[k] <= kFound;
            }
            for (int k = lane; k < min(cnt, kFound); k += 32) {   // the chunks' tiles
                const int t = (pre + k) / kChunk;
                if (t < kTileChunks) atomicAdd(&s_tiles[t], __popc(s_found[warp][k].y >> 8));
            }
            __syncthreads();
            if (warp == 0) {   // the SC's entries and chunks: four reservations at once
                const int nch = (tot + kChunk - 1) / kChunk;
                auto light = [&](int t) { return counted && t < min(nch, kTileChunks) && s_tiles[t] < kLightTiles; };
                int nl = 0;
                for (int t = lane; t - lane < nch; t += 32) nl += __popc(__ballot_sync(kFull, light(t)));
                const int slot = lane == 0 ? 6 : (lane == 1 ? 7 : (lane == 2 ? 8 : 5));
                int got = 0;
                if (lane < 4) got = atomicAdd(&p.counters[slot], lane == 0 ? tot : (lane == 1 ? nch : (lane == 2 ? nch - nl : nl)));
                const int e0 = __shfl_sync(kFull, got, 0), c0 = __shfl_sync(kFull, got, 1);
                int h0 = __shfl_sync(kFull, got, 2), l0 = __shfl_sync(kFull, got, 3);
                const bool fits = (long long)e0 + tot <= p.pl_cap && (long long)c0 + nch <= p.chunk_cap;
                if (lane == 0) {
                    if (!fits) atomicOr(p.err, ERR_LIST);
                    s_e0 = fits ? e0 : -1;
                }
                for (int t = lane; fits && t - lane < nch; t += 32) {
                    const bool on = t < nch, lt = light(t);
                    const unsigned bl = __ballot_sync(kFull, lt), bh = __ballot_sync(kFull, on && !lt), before = (1u << lane) - 1u;
                    const int at = lt ? p.chunk_cap - 1 - (l0 + __popc(bl & before)) : h0 + __popc(bh & before);
                    // (where some SC did not fit, the reservations may run past the table)
                    if (on && at >= 0 && at < p.chunk_cap)
                        p.pl_chunk[at] = make_int4(s.fc, e0 + t * kChunk, min(kChunk, tot - t * kChunk) | (s.ncl << 16), s.rr);
                    l0 += __popc(bl);
                    h0 += __popc(bh);
                }
            }
        } else if (threadIdx.x == 0) {
            int tot = 0;
            for (int k = 0; k < kListWarps; ++k) tot += s_cnt[k];
            const int nch = (tot + kChunk - 1) / kChunk;
            int e0 = atomicAdd(&p.counters[6], tot), c0 = atomicAdd(&p.counters[7], nch);
            if ((long long)e0 + tot > p.pl_cap || (long long)c0 + nch > p.chunk_cap) {
                atomicOr(p.err, ERR_LIST);
                e0 = -1;
            }
            s_e0 = e0;
            s_c0 = c0;
        }
        __syncthreads();
        const int e0 = s_e0;
        if (e0 < 0) continue;   // uniform across the block
        int off = e0, tot = 0;
        for (int k = 0; k < kListWarps; ++k) {
            if (k < warp) off += s_cnt[k];
            tot += s_cnt[k];
        }
        if constexpr (!ORDER)
            for (int t = threadIdx.x; t * kChunk < tot; t += blockDim.x)
                p.pl_chunk[s_c0 + t] = make_int4(s.fc, e0 + t * kChunk, min(kChunk, tot - t * kChunk) | (s.ncl << 16), s.rr);
        if (cnt <= kFound) {
            for (int b = 0; b < cnt; b += 32) {
                ListJ j;
                j.jc = 0;
                j.nb = 0;
                j.m = 0u;
                j.jl = j.jh = make_float4(0.f, 0.f, 0.f, 0.f);
                if (b + lane < cnt) {
                    const uint2 f = s_found[warp][b + lane];
                    j.jc = (int)f.x;
                    j.nb = (int)(f.y & 0xffu);
                    j.m = f.y >> 8;
                }
                const float Dx = __shfl_sync(kFull, c.Dx, j.nb), Dy = __shfl_sync(kFull, c.Dy, j.nb),
                            Dz = __shfl_sync(kFull, c.Dz, j.nb);
                if (j.m) {
                    const float4 lo = p.bb_lo[j.jc], hi = p.bb_hi[j.jc];
                    j.jl = make_float4(lo.x + Dx, lo.y + Dy, lo.z + Dz, 0.0f);
                    j.jh = make_float4(hi.x + Dx, hi.y + Dy, hi.z + Dz, 0.0f);
                }
                const uint4 e = list_entry(p, w, j, __reduce_or_sync(kFull, j.m), rcb2);
                if (j.m) p.pl[off + b + lane] = e;
            }
        } else {
            for (int base = i0; base < i1; base += 32) {
                const ListJ j = list_j(p, w, s, c, base + lane, i1, rcb2);
                const unsigned bal = __ballot_sync(kFull, j.m != 0u);
                const uint4 e = list_entry(p, w, j, __reduce_or_sync(kFull, j.m), rcb2);
                if (j.m) p.pl[off + __popc(bal & ((1u << lane) - 1u))] = e;
                off += __popc(bal);
            }
        }
    }
}

// Bonded terms (Sec. II.B, Eqs. 9-10), one per thread over the grid before the
// chunks: their dependent loads overlap the other warps' pair work, and they
// add to the same fixed-point sums.
template <bool FP64, bool ENERGY>
__device__ __forceinline__ void bonded_prologue(const Params& p)
{
    if (p.n_bonds + p.n_angles == 0) return;
    using T = typename Prec<FP64>::T;
    const T* bp;
    const T* ap;
    if constexpr (FP64) { bp = p.bond_pd; ap = p.angle_pd; }
    else { bp = p.bond_pf; ap = p.angle_pf; }
    const int nb = p.n_bonds, nt = p.n_bonds + p.n_angles;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        if (t < nb) bonded::bond_term<T, ENERGY>(p, bp, t);
        else bonded::angle_term<T, ENERGY>(p, ap, t - nb);
    }
}

// ---------------------------------------------------------------------------
// Mixed-precision force kernel.  A warp takes one chunk (up to kChunk entries
// of one SC) at a time from an atomic counter.  Lane (tx, ty) keeps the force
// of atom tx of each i-cluster in registers for the whole chunk; an entry's
// tiles are the i-clusters of its mask, a warp-uniform branch each, and the
// lane's two j-atoms fill the halves of packed FP32 operations.  j forces go to
// shared memory per lane and are summed over the i-lanes once per chunk.
//
// Bound: instruction issue, with the FMA pipe next.  The kernel it replaced (per-atom
// queues, scalar arithmetic, i forces read and written in shared memory per
// tile, a shuffle reduction per entry) issued 1.66 G warp instructions for a
// million droplet atoms at 80 % issue with the shared-memory pipe 73 % busy;
// this one issues 1.28 G at 68 %, the FMA pipe 48 % busy.  Cluster masks evaluate 14 %
// more pairs than per-atom queues did (33 against 38 % of the evaluations
// within r_cut, water at a 0.12 nm skin), which the cheaper tiles more than
// pay for.  Per launch, 500,001-atom droplet 851 -> 768 us, water box of
// 30,000 atoms 68.9 -> 60.1, 1,500 atoms 19.0 -> 10.5; hybrid screening, 12,003
// atoms, 46.2 -> 39.1.  96 registers (20 warps per SM): with 80 (24 warps) the
// compiler recomputes and spills (963 us), with 128 (16 warps) too few warps
// cover the latencies (947 us before the j sums moved to shared memory).
// Two tiles per branch for more independent work: 852 us, the longer code is
// slower.  The hybrid instance needs 128 registers (112: 45.1 us, 96: 50.9).
// ---------------------------------------------------------------------------
// MODE: 0 Debye, 1 hybrid electrostatics, 2 hybrid with energies
template <int MODE>
struct JHyb {};
template <>
struct JHyb<1> {
    float4 Gr[kChunk * 4];         // G and r' of the two j-atoms: G0 G1 r'0 r'1
    float2 iGr[kSCAtoms];          // (f/2) G_i and r'_i of the SC's atoms
};
template <>
struct JHyb<2> : JHyb<1> {
    float4 ce[kChunk * 4];         // c1 and phi(r_cut) of the two j-atoms: c1_0 c1_1 phi_0 phi_1
    float2 ice[kSCAtoms];          // (f/2) c1_i and (f/2) phi_i(r_cut) of the SC's atoms
};
constexpr int kJpRow = 52;         // floats per lane row of the j-force parts (padded: rows start on different banks)
template <int MODE>
struct WarpF32 {
    float4 xy[kChunk * 4];         // j-atom pairs of the chunk, [entry][ty]: x0 x1 y0 y1 (shifted)
    float4 zq[kChunk * 4];         // z0 z1 q0 q1
    float4 ix[kSCAtoms];           // the SC's atoms: x, y, z, f q (hybrid: (f/2) q)
    int2 off[kChunk * 4];          // LJ column byte offsets of the j-atom pairs
    int2 jfr[kChunk * 4];          // and their fragments
    int irow[kSCAtoms];            // shared-memory address of the SC atoms' LJ rows
    int ifr[kSCAtoms];             // and their fragments
    float jp[kChunk * 4 * kJpRow]; // j-force parts [entry][ty][component][tx]
    int2 counts;                   // the list's chunks, and the heavy ones among them
    uint2 ent[kChunk];             // first slot of the j-cluster; i-cluster mask | kEntGen | kEntShare | cluster of the SC << 16
    JHyb<MODE> hy;
};
constexpr unsigned kEntGen = 0x100u;     // the self-cluster diagonal or pairs within one fragment are possible
constexpr unsigned kEntShare = 0x200u;   // the entry's fragment flag

// What a pair needs besides its two atoms (per chunk).
struct PairCtx {
    float rc2, kl, kap, erc, irc;  // kl = -kappa log2(e)
    float rl2;                     // PRUNE: squared list radius
    float irc6, sh6, sh1;          // ENERGY: r_c^-6, and the shift's e^{-kappa r_c} r_c^-6 / 6 and e^{-kappa r_c} / r_c
    float c2, hf;                  // hybrid: c2 of the replica, f/2
};

__device__ __forceinline__ float2 lds_f2(int addr)
{
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// Atom i against j-atoms 0 and 1.  r^-6 (12 c12 r^-6 - 6 c6 + kappa r (c12 r^-6
// - c6)) is r^-6 ((2 + kappa r / 6) P + 6 c6) with P = 6 c12 r^-6 - 6 c6.
// GEN: pairs may be dropped (ok) or lie within one fragment (no LJ).  iGr, jGr, iCe and
// jCe: the hybrid constants of the atoms (JHyb).
template <bool GEN, bool ENERGY, bool HYB>
__device__ __forceinline__ void pair2(const PairCtx& c, const float4& xi, const float2& iGr, int row, int fri, const float4& xy,
                                      const float4& zq, const int2& off, const int2& frj, const float4& jGr,
                                      const float2& iCe, const float4& jCe, bool ok0, bool ok1, float& fx, float& fy, float& fz, float& u, int& npair, float2& fjx,
                                      float2& fjy, float2& fjz, float2& r2)
{
    using P = Prec<false>;
    constexpr float kL = 0.69314718055994530942f;
    const float2 l0 = lds_f2(row + off.x), l1 = lds_f2(row + off.y);   // (6 c6, 6 c12)
    const float2 dx = make_float2(xi.x - xy.x, xi.x - xy.y);
    const float2 dy = make_float2(xi.y - xy.z, xi.y - xy.w);
    const float2 dz = make_float2(xi.z - zq.x, xi.z - zq.y);
    r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    const bool in0 = r2.x < c.rc2 && (!GEN || ok0), in1 = r2.y < c.rc2 && (!GEN || ok1);
    const float y0 = P::rsq(r2.x), y1 = P::rsq(r2.y);
    const float2 rinv = make_float2(in0 ? y0 : 0.0f, in1 ? y1 : 0.0f);
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    const float2 u6 = __fmul2_rn(__fmul2_rn(rinv2, rinv2), rinv2);
    const float2 r = __fmul2_rn(r2, rinv);
    const float2 t = __fmul2_rn(make_float2(c.kl, c.kl), r);              // -kappa r log2(e)
    const float2 e = make_float2(P::exp2_(t.x), P::exp2_(t.y));           // e^{-kappa r}
    const float2 w6 = __ffma2_rn(t, make_float2(-kL / 6.0f, -kL / 6.0f), make_float2(2.0f, 2.0f));
    const float P0 = __fmaf_rn(l0.y, u6.x, -l0.x), P1 = __fmaf_rn(l1.y, u6.y, -l1.x);
    const float E0 = __fmaf_rn(w6.x, P0, l0.x), E1 = __fmaf_rn(w6.y, P1, l1.x);
    const bool same0 = GEN && fri == frj.x, same1 = GEN && fri == frj.y;   // bonded in the native structure: no LJ
    const float lj0 = same0 ? 0.0f : u6.x, lj1 = same1 ? 0.0f : u6.y;
    const float2 w = __fmul2_rn(rinv2, e);
    float2 fs;   // F(r)/r
    if constexpr (HYB) {
        // each ion's -phi' from its own form, the ion sphere's inside its r' and the
        // Debye form's outside; xi.w = (f/2) q_i
        const float2 q2 = make_float2(zq.z, zq.w);
        const float2 outf = __fmul2_rn(__ffma2_rn(make_float2(c.kap, c.kap), r, make_float2(1.0f, 1.0f)), w);   // e^{-kappa r} (1 + kappa r) / r^2
        const float2 cr = __fmul2_rn(make_float2(2.0f * c.c2, 2.0f * c.c2), r);
        const float2 ii = __ffma2_rn(make_float2(xi.w, xi.w), rinv2, __fmul2_rn(make_float2(c.hf, c.hf), cr));
        const float2 io = __fmul2_rn(make_float2(iGr.x, iGr.x), outf);
        const float2 ji = __ffma2_rn(q2, rinv2, cr), jo = __fmul2_rn(make_float2(jGr.x, jGr.y), outf);
        const float2 mi = make_float2(r.x < iGr.y ? ii.x : io.x, r.y < iGr.y ? ii.y : io.y);     // (f/2)(-phi_i')
        const float2 mj = make_float2(r.x < jGr.z ? ji.x : jo.x, r.y < jGr.w ? ji.y : jo.y);     // -phi_j'
        const float2 cl = __ffma2_rn(make_float2(xi.w, xi.w), mj, __fmul2_rn(q2, mi));
        const float2 lw = __fmul2_rn(make_float2(lj0 * E0, lj1 * E1), w);
        fs = __ffma2_rn(cl, rinv, lw);
    } else {
        // f q_i q_j (1/r + kappa)
        const float2 rk = __fadd2_rn(rinv, make_float2(c.kap, c.kap));
        const float2 qr = __fmul2_rn(make_float2(zq.z, zq.w), rk);
        fs = __fmul2_rn(make_float2(__fmaf_rn(lj0, E0, xi.w * qr.x), __fmaf_rn(lj1, E1, xi.w * qr.y)), w);
    }
    fx = __fmaf_rn(fs.y, dx.y, __fmaf_rn(fs.x, dx.x, fx));
    fy = __fmaf_rn(fs.y, dy.y, __fmaf_rn(fs.x, dy.x, fy));
    fz = __fmaf_rn(fs.y, dz.y, __fmaf_rn(fs.x, dz.x, fz));
    fjx = __ffma2_rn(fs, dx, fjx);
    fjy = __ffma2_rn(fs, dy, fjy);
    fjz = __ffma2_rn(fs, dz, fjz);
    if constexpr (ENERGY) {
        // out of range rinv and lj are zero, and the rest is left out: selects instead of
        // two branches a tile, the shift's constants once per chunk (million-atom frame
        // 2,280 -> 2,032 us)
        const float2 lp = __fmul2_rn(make_float2(lj0, lj1), make_float2(P0, P1));
        const float s0 = same0 ? 0.0f : __fmaf_rn(l0.y, c.irc6, -l0.x), s1 = same1 ? 0.0f : __fmaf_rn(l1.y, c.irc6, -l1.x);
        const float2 six = make_float2(1.0f / 6.0f, 1.0f / 6.0f);
        if constexpr (HYB) {
            // each ion's phi - phi(r_cut) from its own form, the constants staged with the
            // atoms (read from the replica's table per pair in range, in a branch each,
            // they took md_get_energies of 30,000 atoms 641 us; 269 this way)
            const float2 q2 = make_float2(zq.z, zq.w), er = __fmul2_rn(e, rinv);
            const float2 ii = __ffma2_rn(make_float2(xi.w, xi.w), rinv,
                                         __ffma2_rn(make_float2(-c.hf * c.c2, -c.hf * c.c2), r2, make_float2(iCe.x, iCe.x)));
            const float2 io = __fmul2_rn(make_float2(iGr.x, iGr.x), er);
            const float2 ji = __ffma2_rn(q2, rinv, __ffma2_rn(make_float2(-c.c2, -c.c2), r2, make_float2(jCe.x, jCe.y)));
            const float2 jo = __fmul2_rn(make_float2(jGr.x, jGr.y), er);
            const float2 pi = make_float2((r.x < iGr.y ? ii.x : io.x) - iCe.y, (r.y < iGr.y ? ii.y : io.y) - iCe.y);
            const float2 pj = make_float2((r.x < jGr.z ? ji.x : jo.x) - jCe.z, (r.y < jGr.w ? ji.y : jo.y) - jCe.w);
            const float2 cl = __ffma2_rn(q2, pi, __fmul2_rn(make_float2(xi.w, xi.w), pj));
            const float2 v = __ffma2_rn(__fmul2_rn(e, lp), six, cl);
            u += in0 ? __fmaf_rn(-s0, c.sh6, v.x) : 0.0f;
            u += in1 ? __fmaf_rn(-s1, c.sh6, v.y) : 0.0f;
        } else {
            const float2 qq = __fmul2_rn(make_float2(xi.w, xi.w), make_float2(zq.z, zq.w));
            const float2 v = __fmul2_rn(e, __ffma2_rn(lp, six, __fmul2_rn(qq, rinv)));
            const float h0 = __fmaf_rn(s0, c.sh6, qq.x * c.sh1), h1 = __fmaf_rn(s1, c.sh6, qq.y * c.sh1);
            u += v.x - (in0 ? h0 : 0.0f);
            u += v.y - (in1 ? h1 : 0.0f);
        }
        npair += (in0 ? 1 : 0) + (in1 ? 1 : 0);
    }
}

// Adds v to a fixed-point sum when `on`; a value beyond 2^30 (or not finite)
// is left out and noted in bad.
__device__ __forceinline__ void red_fix_if(long long* dst, float v, bool on, bool& bad)
{
    const bool ok = Prec<false>::fix_ok(v);
    if (on && ok) atomicAdd((unsigned long long*)dst, (unsigned long long)Prec<false>::fix(v));
    bad |= on && !ok;
}

template <bool ENERGY, bool HYB, bool LIGHT, int REGS>
__global__ void __maxnreg__(REGS) k_pair(Params p)
{
    using P = Prec<false>;
    using WF = WarpF32<HYB ? (ENERGY ? 2 : 1) : 0>;
    constexpr unsigned kFull = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nts = p.n_ts_lj;
    float2* s_lj = reinterpret_cast<float2*>(smem);
    const size_t tab = ((size_t)nts * nts * sizeof(float2) + 127) / 128 * 128;
    const int warp = threadIdx.x >> 5;
    int lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    WF& w = reinterpret_cast<WF*>(smem + tab)[warp];
    // A warp's first chunk is its own index (neighbours in the list on different
    // blocks), the rest come from the counter; its descriptor and entries are on
    // their way while the block copies the LJ table.  With every warp's first
    // chunk from the counter, 2,432 warps queued for one address, and the early
    // ones took second chunks before the late ones had asked for a first: 1,500
    // atoms 15.4 us against 10.5 now, 8,005 atoms (2,296 chunks) 21.8 against 15.4,
    // 30,000 atoms 64.7 against 62.9.
    const unsigned err = *p.err;
    const int n_chunks = min(p.counters[7], p.chunk_cap);
    const int n_warps = gridDim.x * (blockDim.x >> 5);
    int item = warp * gridDim.x + blockIdx.x;
    if constexpr (LIGHT) {
        const int2 counts = chunk_counts(p);
        item = chunk_at(p, item, counts);
        if (lane == 0) w.counts = counts;   // (registers are short, and the counters' line is busy with the work counter)
    }
    auto any = [&](int it) { return LIGHT ? it >= 0 : it < n_chunks; };
    int4 ch = make_int4(0, 0, 0, 0);   // (first cluster, first entry, entries | clusters << 16, replica)
    if (any(item)) ch = p.pl_chunk[item];
    for (int k = threadIdx.x; k < nts * nts; k += blockDim.x) s_lj[k] = p.lj_f[k];
    PairEntry e4 = make_uint4(0u, 0u, 0u, 0u);
    if (!(err & (ERR_CELL | ERR_LIST)) && any(item) && lane < (ch.z & 0xffff)) e4 = p.pl[ch.y + lane];
    __syncthreads();
    if (err & (ERR_CELL | ERR_LIST)) return;
    bonded_prologue<false, ENERGY>(p);

    const int tx = lane & 7, ty = lane >> 3;
    const int lj_addr = (int)__cvta_generic_to_shared(smem);
    // In the step of a Verlet-buffered build the positions are the build's:
    // i-clusters with no pair within r_cut + skin are dropped from an entry's
    // mask for the list's lifetime (they cannot come within r_cut before the
    // next build), and so is the fragment flag of an entry with no pair in
    // range inside one fragment.  A dropped tile only ever added exact zeros,
    // in the same order: every sum comes out bit-identical with either mask.
    const bool prune = p.builds != nullptr && list_half_skin2(p) > 0.0f && p.builds[1] != 0;
    const float rlb = list_rlist_f(p) + kBBoxMargin;
    const float coulf = (float)p.coulomb_f;
    PairCtx c;
    c.rc2 = p.rc2_f;
    c.irc = (float)(1.0 / p.r_cut);
    c.rl2 = rlb * rlb;
    c.hf = 0.5f * coulf;
    c.c2 = 0.0f;
    bool bad = false;

    // The work items are fetched ahead: while a chunk is evaluated, the counter's
    // answer and the descriptor of the next one are on their way, and its entries
    // are asked for before the i forces of this one are summed.
    while (any(item)) {
        int next = LIGHT ? -1 : n_chunks;
        if constexpr (LIGHT) {
            if (lane == 0) {
                const int warps = gridDim.x * (blockDim.x >> 5);
                if (w.counts.x > warps) next = warps + atomicAdd(&p.counters[2], 1);
            }
        } else {
            if (n_chunks > n_warps && lane == 0) next = n_warps + atomicAdd(&p.counters[2], 1);
        }
        const int fc = ch.x, ent0 = ch.y, n_ent = ch.z & 0xffff, ncl = ch.z >> 16, rr = ch.w;
        const Grid& g = p.grid_b[rr];
        c.kap = p.rs[rr].kappa_f;
        c.kl = c.kap * -1.4426950408889634f;
        c.erc = ENERGY ? P::expneg(c.kap * (float)p.r_cut) : 0.0f;
        if constexpr (ENERGY) {
            c.irc6 = c.irc * c.irc * c.irc * c.irc * c.irc * c.irc;
            c.sh6 = c.erc * c.irc6 * (1.0f / 6.0f);
            c.sh1 = c.erc * c.irc;
        }
        const HybQ* rows = nullptr;            // hybrid: the replica's charge states
        if constexpr (HYB) {
            rows = p.hq + (size_t)rr * kHybQ;
            const HybRep hr = p.hrep[rr];
            c.c2 = hr.c2f;
        }
        __syncwarp();                              // the previous chunk's reads are done
        if (lane < kChunk) {
            unsigned im = e4.z | e4.w;             // i-clusters with some atom in the mask
            im |= im >> 16;
            im = (im | (im >> 8)) & 0xffu;
            const unsigned kd = self_cluster((e4.y & 0xffu) == 0u, e4.x, (unsigned)fc);   // i-cluster equal to the j-cluster
            const bool share = (e4.y & kEntryExcl) != 0u;
            w.ent[lane] = make_uint2(e4.x * kClusterSize, im | (kd < (unsigned)ncl || share ? kEntGen : 0u) |
                                                              (share ? kEntShare : 0u) | (kd << 16));
        }
        // the chunk's j-atoms, one pair per lane, shifted into the SC's cell frame
        {
            const int e = lane >> 2;
            const unsigned jc = __shfl_sync(kFull, e4.x, e), cd = __shfl_sync(kFull, e4.y, e);
            if (e < n_ent) {
                int sx, sy, sz;
                half_shell((int)(cd & 0xffu), sx, sy, sz);
                const float Dx = (float)sx * g.edge_f[0], Dy = (float)sy * g.edge_f[1], Dz = (float)sz * g.edge_f[2];
                const int slot = (int)jc * kClusterSize + (lane & 3);
                const float4 a = p.xq[slot], b = p.xq[slot + 4];
                const int2 ta = p.tf[slot], tb = p.tf[slot + 4];
                const int4 t = make_int4(ta.x, ta.y, tb.x, tb.y);
                w.xy[lane] = make_float4(a.x + Dx, b.x + Dx, a.y + Dy, b.y + Dy);
                w.zq[lane] = make_float4(a.z + Dz, b.z + Dz, a.w, b.w);
                w.off[lane] = make_int2(t.x * (int)sizeof(float2), t.z * (int)sizeof(float2));
                w.jfr[lane] = make_int2(t.y, t.w);
                if constexpr (HYB) {
                    const HybQ& Ra = rows[(int)a.w];
                    const HybQ& Rb = rows[(int)b.w];
                    w.hy.Gr[lane] = make_float4(Ra.Gf, Rb.Gf, Ra.rpf, Rb.rpf);
                    if constexpr (ENERGY) w.hy.ce[lane] = make_float4(Ra.c1f, Rb.c1f, Ra.phircf, Rb.phircf);
                }
            }
        }
        // the SC's atoms
#pragma unroll
        for (int a = lane; a < kSCAtoms; a += 32)
            if (a < ncl * kClusterSize) {
                const float4 v = p.xq[fc * kClusterSize + a];
                const int2 t = p.tf[fc * kClusterSize + a];
                w.ix[a] = make_float4(staged_x(v.x, v.w), v.y, v.z, (HYB ? c.hf : coulf) * v.w);
                w.irow[a] = lj_addr + t.x * nts * (int)sizeof(float2);
                w.ifr[a] = t.y;
                if constexpr (HYB) {
                    const HybQ& Ri = rows[(int)v.w];
                    w.hy.iGr[a] = make_float2(c.hf * Ri.Gf, Ri.rpf);
                    if constexpr (ENERGY) w.hy.ice[a] = make_float2(c.hf * Ri.c1f, c.hf * Ri.phircf);
                }
            }
        float ue[ENERGY ? kSuperClusters : 1];
        float fx[kSuperClusters], fy[kSuperClusters], fz[kSuperClusters];
        int npair = 0;
#pragma unroll
        for (int k = 0; k < kSuperClusters; ++k) {
            fx[k] = fy[k] = fz[k] = 0.0f;
            if constexpr (ENERGY) ue[k] = 0.0f;
        }
        if constexpr (LIGHT)
            if (lane == 0 && next >= 0) next = chunk_at(p, next, w.counts);
        next = __shfl_sync(kFull, next, 0);
        if (any(next)) ch = p.pl_chunk[next];
        __syncwarp();

#pragma unroll 1
        for (int v = 0; v < n_ent; ++v) {
            const uint2 en = w.ent[v];
            // through a warp reduction, so that the branches on it are known to be uniform
            const unsigned um = __reduce_or_sync(kFull, en.y);
            if ((um & 0xffu) == 0u) continue;      // no i-cluster in range (or emptied by pruning)
            const float4 xy = w.xy[4 * v + ty], zq = w.zq[4 * v + ty];
            const int2 off = w.off[4 * v + ty];
            float4 jGr = make_float4(0.f, 0.f, 0.f, 0.f), jCe = jGr;
            if constexpr (HYB) jGr = w.hy.Gr[4 * v + ty];
            if constexpr (HYB && ENERGY) jCe = w.hy.ce[4 * v + ty];
            float2 fjx = make_float2(0.f, 0.f), fjy = fjx, fjz = fjx, r2;
            // GEN: the self-cluster diagonal (i < j) or pairs within one fragment are
            // possible; PRUNE: build step
            auto tiles = [&](auto gen, auto pr) {
                constexpr bool GEN = decltype(gen)::value, PRUNE = decltype(pr)::value;
                int2 frj = make_int2(0, 0);
                if constexpr (GEN) frj = w.jfr[4 * v + ty];
                bool share = false;   // a pair in range within one fragment
                unsigned keep = 0u;   // i-clusters with a pair in range
#pragma unroll
                for (int k = 0; k < kSuperClusters; ++k) {
                    if (um & (1u << k)) {
                        const float4 xi = w.ix[k * kClusterSize + tx];
                        const int row = w.irow[k * kClusterSize + tx];
                        float2 iGr = make_float2(0.f, 0.f), iCe = iGr;
                        if constexpr (HYB) iGr = w.hy.iGr[k * kClusterSize + tx];
                        if constexpr (HYB && ENERGY) iCe = w.hy.ice[k * kClusterSize + tx];
                        int fri = 0;
                        bool ok0 = true, ok1 = true;
                        if constexpr (GEN) {
                            fri = w.ifr[k * kClusterSize + tx];
                            const bool dg = (um >> 16) == (unsigned)k;
                            ok0 = !dg || tx < ty;
                            ok1 = !dg || tx < ty + 4;
                        }
                        pair2<GEN, ENERGY, HYB>(c, xi, iGr, row, fri, xy, zq, off, frj, jGr, iCe, jCe, ok0, ok1, fx[k], fy[k], fz[k],
                                                ue[ENERGY ? k : 0], npair, fjx, fjy, fjz, r2);
                        if constexpr (PRUNE) {
                            const bool n0 = ok0 && r2.x < c.rl2, n1 = ok1 && r2.y < c.rl2;
                            if (__any_sync(kFull, n0 || n1)) keep |= 1u << k;
                            if constexpr (GEN) share |= (n0 && fri == frj.x) || (n1 && fri == frj.y);
                        }
                    }
                }
                if constexpr (PRUNE) {
                    share = __any_sync(kFull, share);
                    if (lane == 0) {
                        PairEntry& out = p.pl[ent0 + v];
                        if (keep != (um & 0xffu)) {
                            const unsigned m4 = keep * 0x01010101u;
                            out.z &= m4;
                            out.w &= m4;
                        }
                        if (share != ((um & kEntShare) != 0u)) out.y ^= kEntryExcl;
                    }
                }
            };
            if (um & kEntGen) {
                if (prune) tiles(std::true_type{}, std::true_type{});
                else tiles(std::true_type{}, std::false_type{});
            } else {
                if (prune) tiles(std::false_type{}, std::true_type{});
                else tiles(std::false_type{}, std::false_type{});
            }
            // the lane's j forces, summed over the 8 i-lanes after the chunk
            float* jp = &w.jp[(4 * v + ty) * kJpRow + tx];
            jp[0] = fjx.x; jp[8] = fjy.x; jp[16] = fjz.x;
            jp[24] = fjx.y; jp[32] = fjy.y; jp[40] = fjz.y;
        }
        __syncwarp();
        // j forces: lane (entry, ty) sums the 8 lanes' parts of its pair's six components
        {
            const int slot = (int)w.ent[lane >> 2].x + (lane & 3);
            if (lane < 4 * n_ent && (w.ent[lane >> 2].y & 0xffu)) {
                const float* jp = &w.jp[lane * kJpRow];
                // (padding takes no force; where the pair's second atom is, its sums are
                // mostly a memory sector each: a gas of one atom a cell, 262,144 atoms, takes
                // 1,290 us per step without them and 1,370 with)
                const bool second = __float_as_int(w.zq[lane].w) >= 0;
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    const float4 a = *reinterpret_cast<const float4*>(jp + 8 * q), b = *reinterpret_cast<const float4*>(jp + 8 * q + 4);
                    const float2 s2 = __fadd2_rn(__fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                                                 __fadd2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w)));
                    long long* dst = q % 3 == 0 ? p.fx : (q % 3 == 1 ? p.fy : p.fz);
                    red_fix_if(dst + slot + 4 * (q / 3), -(s2.x + s2.y), q < 3 || second, bad);
                }
            }
        }
        // the next chunk's entries
        e4 = make_uint4(0u, 0u, 0u, 0u);
        if (any(next) && lane < (ch.z & 0xffff)) e4 = p.pl[ch.y + lane];
        item = next;
        // i forces: sum over the four lane rows, a transposing reduction that leaves
        // two i-clusters to each row; sums of exact zero (tiles never evaluated) add nothing
        {
            const bool up2 = (ty & 2) != 0, up1 = (ty & 1) != 0;
            auto rows = [&](const float* a, long long* dst) {
                float b[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    b[q] = (up2 ? a[q + 4] : a[q]) + __shfl_xor_sync(kFull, up2 ? a[q] : a[q + 4], 16);
                dst += (fc + (up2 ? 4 : 0) + (up1 ? 2 : 0)) * kClusterSize + tx;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float s = (up1 ? b[q + 2] : b[q]) + __shfl_xor_sync(kFull, up1 ? b[q] : b[q + 2], 8);
                    red_fix_if(dst + q * kClusterSize, s, s != 0.0f, bad);
                }
            };
            rows(fx, p.fx);
            rows(fy, p.fy);
            rows(fz, p.fz);
            if constexpr (ENERGY) rows(ue, p.epot);
        }
        if constexpr (ENERGY) {
#pragma unroll
            for (int o = 16; o; o >>= 1) npair += __shfl_xor_sync(kFull, npair, o);
            if (lane == 0 && npair) atomicAdd((unsigned long long*)p.pair_count, (unsigned long long)npair);
        }
    }
    if (bad) atomicOr(p.err, ERR_OVERFLOW);
}

// FP64 forces over the cluster-pair list.  A warp takes one chunk (up to kChunk
// entries of one SC) at a time from an atomic counter; each block holds its own
// copy of the LJ table.
//
// GB300 issues FP64 at 2 lanes per SM per clock (a warp instruction takes 16
// cycles of the SM), so what counts is how few pair evaluations are issued.
// Per group of kGroup64 entries the lanes first test their pairs in FP32 with a
// margin that covers the rounding of the coordinates, each keeping its pairs in
// range as bits, and then evaluate those in FP64, every lane its own next one:
// idle lanes only where a lane has fewer pairs than the fullest one (71 % of
// the issued evaluations lie within r_cut, counted in a water box and a methane
// cluster; 38 % when all lanes followed the
// entries' masks together).  The pairs left out only ever added exact zeros and
// the others keep their order, so the sums are the same bit for bit.
// Per launch, 30,000-atom water box: 2,730 -> 1,600 us; 8 warps per SM and 4 in
// each of two blocks take the same time, 4 alone 18 % more.
template <bool ENERGY, bool HYB>
__global__ void __launch_bounds__(256, 1) k_pair64(Params p)
{
    using P = Prec<true>;
    using T = double;
    using T4 = double4_32a;
    using S4 = double4_16a;
    using C2 = double2;
    using WS = Warp64<HYB>;
    constexpr unsigned kFull = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nts = p.n_ts_lj;
    C2* s_lj = reinterpret_cast<C2*>(smem);
    const unsigned char* lj_bytes = smem;
    const size_t tab = ((size_t)nts * nts * sizeof(C2) + 127) / 128 * 128;
    // s_kq[c]: the set bits of the 8-bit column mask c as 4-bit cluster indices,
    // lowest first, the unused nibbles 8 (a column's stand-in row)
    unsigned* s_kq = reinterpret_cast<unsigned*>(smem + tab);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WS& w = reinterpret_cast<WS*>(smem + tab + 256 * sizeof(unsigned))[warp];

    for (int k = threadIdx.x; k < nts * nts; k += blockDim.x) s_lj[k] = P::table(p)[k];
    for (int c = threadIdx.x; c < 256; c += blockDim.x) {
        unsigned q = 0x88888888u;
        int n = 0;
        for (int k = 0; k < 8; ++k)
            if ((c >> k) & 1) {
                q = (q & ~(0xfu << (4 * n))) | ((unsigned)k << (4 * n));
                ++n;
            }
        s_kq[c] = q;
    }
    for (int k = lane; k < 4 * kSCAtoms; k += 32) w.fi[k] = P::mk(T(0), T(0), T(0), T(0));
    for (int k = 0; k < 6 * kGroup64; ++k) w.fj[k][lane] = 0.0;
    if (lane < kClusterSize) {
        w.ixf[kSCAtoms + lane] = make_float4(-1.0e6f, -1.0e6f, -1.0e6f, 0.0f);
        w.it[kSCAtoms + lane] = make_int2(0, (int)0x80000000);
    }
    __syncthreads();
    if (*p.err & (ERR_CELL | ERR_LIST)) return;
    bonded_prologue<true, ENERGY>(p);

    const int tx = lane & 7, ty = lane >> 3;
    const int2 counts = chunk_counts(p);
    // after the j-force reduction lane (tx, ty) holds component tx & 3 of atom
    // ty (tx < 4) or ty + 4 (tx >= 4) of the entry's j-cluster
    const int comp = tx & 3;
    long long* const jdst = comp == 0 ? p.fx : (comp == 1 ? p.fy : p.fz);
    // In the step of a Verlet-buffered build the positions are the build's:
    // i-atoms with no j-atom within r_cut + skin (to the FP32 test's margin) are
    // dropped from an entry's mask for the list's lifetime (they cannot come within
    // r_cut before the next build), and so is the fragment flag of an entry with no
    // pair in range inside one fragment.
    const bool prune = p.builds != nullptr && list_half_skin2(p) > 0.0f && p.builds[1] != 0;
    const float rlb = list_rlist_f(p) + kBBoxMargin;
    const T rc2 = p.rc2;
    const T irc = T(1.0 / p.r_cut);
    const T coulf = p.coulomb_f;

    // A warp's first chunk is its own index, neighbours on different SMs, the rest
    // come from the counter.  The FP64 pipe is the SM's: with every first chunk from
    // the counter, the first SMs to ask took up to eight of a small system's chunks
    // and others none.  Per launch 3,224 atoms 317 -> 252 us, 1,500 atoms 239 -> 232,
    // 30,000 atoms 1,561 -> 1,551.
    const int n_warps = gridDim.x * (blockDim.x >> 5);
    bool first = true;
    while (true) {
        int item = warp * gridDim.x + blockIdx.x;
        if (!first) {
            if (counts.x <= n_warps) break;
            if (lane == 0) item = n_warps + atomicAdd(&p.counters[2], 1);
            item = __shfl_sync(kFull, item, 0);
        }
        first = false;
        item = chunk_at(p, item, counts);
        if (item < 0) break;
        const int4 ch = p.pl_chunk[item];   // (first cluster, first entry, entries | clusters << 16, replica)
        const int fc = ch.x, n_ent = ch.z & 0xffff, ncl = ch.z >> 16, rr = ch.w;
        __syncwarp();   // the previous chunk's reads of the staged entries are done
        if (lane < n_ent) w.ent[lane] = p.pl[ch.y + lane];
        const Grid& g = p.grid_b[rr];
        const T kap = p.rs[rr].kappa_force;
        const T kl = kap * T(-1.4426950408889634);   // -kappa log2(e)
        const T erc = ENERGY ? P::expneg(kap * T(p.r_cut)) : T(0);
        HybArg<T> ha{};
        const HybQ* hrows = nullptr;
        if constexpr (HYB) {
            hrows = p.hq + (size_t)rr * kHybQ;
            const HybRep hr = p.hrep[rr];
            ha.kap = kap;
            ha.c2 = hr.c2;
            ha.rpm2 = hr.rpm2;
            ha.hf = T(0.5) * coulf;
            ha.rows = hrows;
        }
        // FP32 tests: coordinates of up to twice the cell edge E rounded to 24 bits
        // move r^2 by less than 1e-6 E r
        const float E = fmaxf(g.edge_f[0], fmaxf(g.edge_f[1], g.edge_f[2]));
        const float rc2t = (float)rc2 + 2.0e-6f * E * (float)p.r_cut, rl2t = rlb * rlb + 2.0e-6f * E * rlb;

        // the super-cluster's atoms and the chunk's j-atoms (shifted into the
        // SC's cell frame) into shared memory: one load latency per chunk
        // instead of one per entry
        __syncwarp();
        for (int a = lane; a < kSCAtoms; a += 32) {
            if ((a >> 3) < ncl) {
                const int slot = fc * kClusterSize + a;
                const T4 v = P::pos(p, slot);
                const int2 t = p.tf[slot];
                w.ix[a] = P::mk(v.x, v.y, v.z, coulf * v.w);
                w.ixf[a] = make_float4((float)v.x, (float)v.y, (float)v.z, 0.0f);
                w.it[a] = make_int2(t.x * nts * (int)sizeof(C2), t.y);   // byte offset of the LJ row
                if constexpr (HYB) {
                    const T G = hrows[(int)v.w].G;
                    w.hy.ih[a] = P::mk(T(0.5) * coulf * G, T(0.5) * coulf * v.w, v.w, T(0));
                }
            }
        }
        for (int a0 = 0; a0 < kChunk * kClusterSize; a0 += 32) {
            const int a = a0 + lane, e = a >> 3;                 // entry e, atom a & 7
            if (e < n_ent) {
                const unsigned jc = w.ent[e].x, cd = w.ent[e].y;
                int dx, dy, dz;
                half_shell((int)(cd & 0xffu), dx, dy, dz);
                const int slot = (int)jc * kClusterSize + (a & 7);
                const T4 v = P::pos(p, slot);
                const int2 t = p.tf[slot];
                const S4 x = P::mk(v.x + T(dx * g.edge[0]), v.y + T(dy * g.edge[1]), v.z + T(dz * g.edge[2]), v.w);
                w.jx[a] = x;
                w.jxf[a] = make_float4((float)x.x, (float)x.y, (float)x.z, 0.0f);
                w.jt[a] = make_int2(t.x * (int)sizeof(C2), t.y);   // byte offset of the LJ column
                w.jqk[a] = v.w * kap;
                if constexpr (HYB) w.hy.jG[a] = hrows[(int)v.w].G;
            }
        }
        __syncwarp();
        int npair = 0;

        for (int v0 = 0; v0 < n_ent; v0 += kGroup64) {
            const int nv = min(kGroup64, n_ent - v0);
            // this lane's pairs in range: bit 16 e + 2 t + j for entry v0 + e, place t of
            // the column's queue, j-atom ty + 4 j
            unsigned long long bits = 0ull;
            for (int e = 0; e < nv; ++e) {
                const int v = v0 + e;
                const PairEntry e4 = w.ent[v];   // one broadcast read
                const unsigned mlo = e4.z, mhi = e4.w;
                if ((mlo | mhi) == 0u) continue;   // no i-atom in range (or emptied by pruning)
                const int nb = (int)(e4.y & 0xffu);
                const int kdiag = nb == 0 ? (int)e4.x - fc : -1;   // i-cluster equal to this j-cluster
                // this lane column's i-clusters (byte tx of the column-major mask: bit k
                // when atom tx of i-cluster k is in)
                const unsigned col0 = __byte_perm(mlo, mhi, (unsigned)tx) & 0xffu;   // byte tx of (mhi:mlo)
                const int n_t = (int)__reduce_max_sync(kFull, (unsigned)__popc(col0));
                unsigned kq = s_kq[col0];
                w.kq[e][lane] = kq;
                const float4 a0 = w.jxf[v * kClusterSize + ty], a1 = w.jxf[v * kClusterSize + ty + 4];
                const int f0 = w.jt[v * kClusterSize + ty].y, f1 = w.jt[v * kClusterSize + ty + 4].y;
                unsigned in = 0u, keep = 0u;
                bool share = false;
                for (int t = 0; t < n_t; ++t) {
                    const int k = (int)(kq & 0xfu);   // 8 once the column is used up: the stand-in row
                    kq >>= 4;
                    const float4 xi = w.ixf[k * kClusterSize + tx];
                    const float dx0 = xi.x - a0.x, dy0 = xi.y - a0.y, dz0 = xi.z - a0.z;
                    const float dx1 = xi.x - a1.x, dy1 = xi.y - a1.y, dz1 = xi.z - a1.z;
                    const float q0 = dx0 * dx0 + dy0 * dy0 + dz0 * dz0, q1 = dx1 * dx1 + dy1 * dy1 + dz1 * dz1;
                    const bool dg = k == kdiag;   // the self-cluster diagonal: i < j
                    const bool ok0 = !dg || tx < ty, ok1 = !dg || tx < ty + 4;
                    in |= ((ok0 && q0 < rc2t ? 1u : 0u) | (ok1 && q1 < rc2t ? 2u : 0u)) << (2 * t);
                    if (prune) {
                        const bool n0 = ok0 && q0 < rl2t, n1 = ok1 && q1 < rl2t;
                        if (n0 || n1) {   // never for the far stand-in row
                            keep |= 1u << k;
                            const int fr = w.it[k * kClusterSize + tx].y;
                            share |= (n0 && fr == f0) || (n1 && fr == f1);
                        }
                    }
                }
                bits |= (unsigned long long)in << (16 * e);
                if (prune) {
                    // columns back to the column-major mask (byte tx: the OR over the
                    // column's four lane rows), and any pair in range within a fragment
                    const unsigned klo = __reduce_or_sync(kFull, tx < 4 ? keep << ((tx & 3) * 8) : 0u);
                    const unsigned khi = __reduce_or_sync(kFull, tx >= 4 ? keep << ((tx & 3) * 8) : 0u);
                    share = __any_sync(kFull, share);
                    if (lane == 0) {
                        if (klo != mlo || khi != mhi) *reinterpret_cast<uint2*>(&p.pl[ch.y + v].z) = make_uint2(klo, khi);
                        if (share != ((e4.y & kEntryExcl) != 0u)) p.pl[ch.y + v].y = (unsigned)nb | (share ? kEntryExcl : 0u);
                    }
                }
            }
            __syncwarp();
            while (__any_sync(kFull, bits != 0ull)) {
                if (bits != 0ull) {
                    const int b = __ffsll((long long)bits) - 1;
                    bits &= bits - 1ull;
                    const int e = b >> 4, j = b & 1;
                    const int ia = (int)((w.kq[e][lane] >> (2 * (b & 14))) & 0xfu) * kClusterSize + tx;
                    const int ja = (v0 + e) * kClusterSize + ty + 4 * j;
                    const S4 xi = w.ix[ia], xj = w.jx[ja];
                    const int2 ti = w.it[ia], tj = w.jt[ja];
                    S4 acc = w.fi[ty * kSCAtoms + ia];
                    HybArg<T> h = ha;
                    if constexpr (HYB) {
                        const S4 hi = w.hy.ih[ia];
                        h.hGi = hi.x;
                        h.hqi = hi.y;
                        h.qi = hi.z;
                        h.Gj = w.hy.jG[ja];
                        h.Gjk = h.Gj * kap;
                    }
                    double* const fj = &w.fj[6 * e + 3 * j][lane];
                    T jx = fj[0], jy = fj[32], jz = fj[64];
                    pair64<ENERGY, HYB>(xi, ti.x, ti.y, xj.x, xj.y, xj.z, xj.w, w.jqk[ja], tj.x, tj.y, lj_bytes, kl, rc2, acc.x,
                                        acc.y, acc.z, jx, jy, jz, acc.w, npair, erc, irc, h);
                    fj[0] = jx;
                    fj[32] = jy;
                    fj[64] = jz;
                    w.fi[ty * kSCAtoms + ia] = acc;
                }
            }
            // j forces: sum over the 8 i-lanes of each ty group.  Lanes tx < 4 keep
            // atom ty (j0), lanes tx >= 4 atom ty + 4 (j1); then each lane holds one
            // component of one atom and issues one RED.
            for (int e = 0; e < nv; ++e) {
                const PairEntry e4 = w.ent[v0 + e];
                if ((e4.z | e4.w) == 0u) continue;
                T f[6];
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    f[q] = w.fj[6 * e + q][lane];
                    w.fj[6 * e + q][lane] = 0.0;
                }
                const bool up = tx >= 4;
                T ax = up ? f[3] : f[0], ay = up ? f[4] : f[1], az = up ? f[5] : f[2];
                ax += __shfl_xor_sync(kFull, up ? f[0] : f[3], 4);
                ay += __shfl_xor_sync(kFull, up ? f[1] : f[4], 4);
                az += __shfl_xor_sync(kFull, up ? f[2] : f[5], 4);
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    ax += __shfl_xor_sync(kFull, ax, o);
                    ay += __shfl_xor_sync(kFull, ay, o);
                    az += __shfl_xor_sync(kFull, az, o);
                }
                if (comp < 3) {
                    const T v3 = comp == 0 ? ax : (comp == 1 ? ay : az);
                    red_fix<true>(jdst + (int)e4.x * kClusterSize + ty + (up ? 4 : 0), v3, p.err);
                }
            }
        }
        __syncwarp();
        // i forces of this chunk: sum the 4 ty partials of each atom, clearing
        // them for the next chunk
        for (int a = lane; a < ncl * kClusterSize; a += 32) {
            S4 sum = w.fi[a];
            w.fi[a] = P::mk(T(0), T(0), T(0), T(0));
#pragma unroll
            for (int q = 1; q < 4; ++q) {
                const S4 v = w.fi[q * kSCAtoms + a];
                w.fi[q * kSCAtoms + a] = P::mk(T(0), T(0), T(0), T(0));
                sum.x += v.x; sum.y += v.y; sum.z += v.z;
                if (ENERGY) sum.w += v.w;
            }
            const int slot = fc * kClusterSize + a;
            red_fix<true>(p.fx + slot, sum.x, p.err);
            red_fix<true>(p.fy + slot, sum.y, p.err);
            red_fix<true>(p.fz + slot, sum.z, p.err);
            if (ENERGY) red_fix<true>(p.epot + slot, sum.w, p.err);
        }
        __syncwarp();
        if (ENERGY) {
#pragma unroll
            for (int o = 16; o; o >>= 1) npair += __shfl_xor_sync(kFull, npair, o);
            if (lane == 0 && npair) atomicAdd((unsigned long long*)p.pair_count, (unsigned long long)npair);
        }
    }
}

// Walks of the cluster-pair list for the analyses: every unordered pair of
// atoms within r_cut once, with the force kernel's traversal (chunks, staged
// atoms, column queues), so the distances are the force evaluation's.  The
// per-pair work is an operation type:
//   RdfOp   pair-distance histogram for the radial distribution functions of
//           Sec. II.C, Eq. 18: every pair within r_max <= r_cut by species
//           pair (a <= b) and bin k = floor(r / dr), counted in a block
//           histogram in shared memory (when it fits, else straight to global
//           memory) and added to the global one as 64-bit integers;
//   FragOp  fragments for the ion yields of Sec. III: every pair closer than
//           r_frag <= r_cut joins the atoms' sets in a lock-free union-find
//           whose parent indices only decrease, so each root is its set's
//           smallest atom index.
// An operation states how far apart it looks (reach): where that is well inside
// the list's radius, a chunk's i-clusters are first tested by their boxes, and
// most chunks of a fragment search are done with after that (a million droplet
// atoms at r_frag 0.16 nm: 1,111 -> 475 us).  The histogram of a block holds
// each species pair once, so that six blocks fit an SM instead of four
// (1,230 -> 1,181 us for 240 bins of five species).
template <bool FP64>
struct WalkWarp {
    typename Prec<FP64>::S4 ix[kFiRow];                  // x, y, z of the SC atoms
    typename Prec<FP64>::S4 jx[kChunk * kClusterSize];   // the chunk's j-atoms, shifted
    int ia[kFiRow];                                      // the operation's labels of the atoms (-1: none)
    int ja[kChunk * kClusterSize];
};
constexpr size_t kRowBytes = kMaxSpecies * kMaxSpecies * sizeof(int);   // RdfOp's table of species pairs

template <bool FP64>
struct RdfOp {
    using T = typename Prec<FP64>::T;
    using S4 = typename Prec<FP64>::S4;
    int n_bins, nsp, smem_hist;
    T rmax2, inv_dr;
    unsigned long long* hist;
    unsigned* s_h;
    const int* s_row;   // first bin of each species pair
    __host__ __device__ int pair_rows() const { return nsp * (nsp + 1) / 2; }   // rows of the block histogram: a <= b
    __device__ float reach(const Params&) const { return 1.0e30f; }   // every listed pair may be binned
    __device__ size_t smem_bytes() const
    {
        return kRowBytes + (smem_hist ? ((size_t)pair_rows() * n_bins * sizeof(unsigned) + 15) / 16 * 16 : 0);
    }
    __device__ void init(unsigned char* smem)
    {
        int* row = reinterpret_cast<int*>(smem);
        for (int k = threadIdx.x; k < kMaxSpecies * kMaxSpecies; k += blockDim.x) {
            const int sa = k / kMaxSpecies, sb = k % kMaxSpecies;
            const int lo = min(sa, sb), hi = max(sa, sb);
            row[k] = (smem_hist ? hi * (hi + 1) / 2 + lo : lo * nsp + hi) * n_bins;
        }
        s_row = row;
        s_h = reinterpret_cast<unsigned*>(smem + kRowBytes);
        if (smem_hist)
            for (int k = threadIdx.x; k < pair_rows() * n_bins; k += blockDim.x) s_h[k] = 0u;
    }
    // label of an atom: its species (-1: no atom)
    __device__ int label(const Params& p, int at) const { return at >= 0 ? (int)p.species[at] : -1; }
    __device__ void pair(const S4& a, int la, const S4& b, int lb, bool ok)
    {
        const T dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
        const T r2 = Prec<FP64>::fma(dz, dz, Prec<FP64>::fma(dy, dy, dx * dx));
        if (ok && r2 < rmax2 && (la | lb) >= 0) {
            const int k = min((int)(sqrt(r2) * inv_dr), n_bins - 1);
            const int idx = s_row[la * kMaxSpecies + lb] + k;
            if (smem_hist) atomicAdd(&s_h[idx], 1u);
            else atomicAdd(&hist[idx], 1ull);
        }
    }
    __device__ void finish()
    {
        if (smem_hist) {
            __syncthreads();
            for (int hi = 0; hi < nsp; ++hi)
                for (int lo = 0; lo <= hi; ++lo)
                    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
                        const unsigned n = s_h[s_row[lo * kMaxSpecies + hi] + k];
                        if (n) atomicAdd(&hist[((size_t)lo * nsp + hi) * n_bins + k], (unsigned long long)n);
                    }
        }
    }
};

// Root of x's set.  Parents only ever point to smaller indices, so the walk
// ends within x steps; each step halves the path (the grandparent written is
// an ancestor whichever thread wrote last).
__device__ __forceinline__ int uf_find(int* parent, int x)
{
    while (true) {
        const int px = __ldcg(parent + x);
        if (px == x) return x;
        const int gp = __ldcg(parent + px);
        if (gp != px) parent[x] = gp;
        x = px;
    }
}

// Joins the sets of a and b: the larger root is hooked under the smaller one
// by a compare-and-swap that succeeds only on a root.  A failed swap means
// another thread hooked that root meanwhile; each retry follows a merge, so
// there are fewer retries than atoms (bounded anyway, with an error flag).
__device__ __forceinline__ void uf_unite(int* parent, int a, int b, int n, unsigned* err)
{
    for (int it = 0; it <= n; ++it) {
        a = uf_find(parent, a);
        b = uf_find(parent, b);
        if (a == b) return;
        if (a > b) { const int t = a; a = b; b = t; }
        if (atomicCAS(parent + b, b, a) == b) return;
    }
    atomicOr(err, ERR_OVERFLOW);
}

template <bool FP64>
struct FragOp {
    using T = typename Prec<FP64>::T;
    using S4 = typename Prec<FP64>::S4;
    T rf2;
    int* parent;
    int n;
    unsigned* err;
    // farthest apart two clusters' boxes of the last build may be for a pair
    // closer than r_frag now: each atom has moved by half the skin at most
    __device__ float reach(const Params& p) const
    {
        return (float)sqrt(rf2) + (list_rlist_f(p) - p.rc_f) + 2.0f * kBBoxMargin;
    }
    __device__ int label(const Params&, int at) const { return at; }
    __device__ size_t smem_bytes() const { return 0; }
    __device__ void init(unsigned char*) {}
    __device__ void pair(const S4& a, int ia, const S4& b, int ib, bool ok)
    {
        const T dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
        const T r2 = Prec<FP64>::fma(dz, dz, Prec<FP64>::fma(dy, dy, dx * dx));
        if (ok && r2 < rf2 && ia >= 0 && ib >= 0) uf_unite(parent, ia, ib, n, err);
    }
    __device__ void finish() {}
};

template <bool FP64, bool LIGHT, class Op>
__global__ void __launch_bounds__(256) k_walk(Params p, Op op)
{
    using P = Prec<FP64>;
    using T = typename P::T;
    using T4 = typename P::T4;
    using S4 = typename P::S4;
    constexpr unsigned kFull = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const size_t hb = op.smem_bytes();
    op.init(smem);
    unsigned* s_kq = reinterpret_cast<unsigned*>(smem + hb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WalkWarp<FP64>& w = reinterpret_cast<WalkWarp<FP64>*>(smem + hb + 256 * sizeof(unsigned))[warp];
    for (int c = threadIdx.x; c < 256; c += blockDim.x) {
        unsigned q = 0x88888888u;
        int n = 0;
        for (int k = 0; k < 8; ++k)
            if ((c >> k) & 1) {
                q = (q & ~(0xfu << (4 * n))) | ((unsigned)k << (4 * n));
                ++n;
            }
        s_kq[c] = q;
    }
    if (lane < kClusterSize) {
        w.ix[kSCAtoms + lane] = P::mk(T(-1.0e6), T(-1.0e6), T(-1.0e6), T(0));
        w.ia[kSCAtoms + lane] = -1;
    }
    __syncthreads();
    const int tx = lane & 7, ty = lane >> 3;
    const int n_chunks = min(p.counters[7], p.chunk_cap), n_heavy = LIGHT ? chunk_counts(p).y : n_chunks;
    const float reach = op.reach(p);
    const bool near_only = reach < list_rlist_f(p);   // the operation needs only pairs well inside the list's radius
    while (true) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&p.counters[2], 1);
        item = __shfl_sync(kFull, item, 0);
        if (item >= n_chunks) break;
        if (LIGHT) item = chunk_at(p, item, make_int2(n_chunks, n_heavy));
        const int4 ch = p.pl_chunk[item];
        const int fc = ch.x, n_ent = ch.z & 0xffff, ncl = ch.z >> 16, rr = ch.w;
        PairEntry ent = lane < n_ent ? p.pl[ch.y + lane] : make_uint4(0u, 0u, 0u, 0u);
        const Grid& g = p.grid_b[rr];
        if (near_only) {
            // keep the i-clusters whose boxes come within reach of the entry's
            // j-cluster: lane tests entry lane >> 2 against i-clusters 2 (lane & 3)
            // and the next; a chunk with none left is not staged at all
            const int e = lane >> 2;
            const unsigned jc = __shfl_sync(kFull, ent.x, e), cd = __shfl_sync(kFull, ent.y, e);
            unsigned near = 0u;
            if (e < n_ent) {
                int dx, dy, dz;
                half_shell((int)(cd & 0xffu), dx, dy, dz);
                const float Dx = (float)dx * g.edge_f[0], Dy = (float)dy * g.edge_f[1], Dz = (float)dz * g.edge_f[2];
                const float4 jl = p.bb_lo[jc], jh = p.bb_hi[jc];
                for (int k = 2 * (lane & 3); k < min(2 * (lane & 3) + 2, ncl); ++k) {
                    const float4 il = p.bb_lo[fc + k], ih = p.bb_hi[fc + k];
                    const float gx = max3f(il.x - (jh.x + Dx), (jl.x + Dx) - ih.x, 0.0f);
                    const float gy = max3f(il.y - (jh.y + Dy), (jl.y + Dy) - ih.y, 0.0f);
                    const float gz = max3f(il.z - (jh.z + Dz), (jl.z + Dz) - ih.z, 0.0f);
                    if (gx * gx + gy * gy + gz * gz < reach * reach) near |= 1u << k;
                }
            }
            near |= __shfl_xor_sync(kFull, near, 1);
            near |= __shfl_xor_sync(kFull, near, 2);
            near = __shfl_sync(kFull, near, (4 * lane) & 31) * 0x01010101u;   // entry lane's clusters, in every column
            ent.z &= near;
            ent.w &= near;
            if (__all_sync(kFull, lane >= n_ent || (ent.z | ent.w) == 0u)) continue;
        }
        __syncwarp();
        for (int a = lane; a < kSCAtoms; a += 32) {
            if ((a >> 3) < ncl) {
                const int slot = fc * kClusterSize + a;
                const T4 v = P::pos(p, slot);
                w.ix[a] = P::mk(v.x, v.y, v.z, T(0));
                w.ia[a] = op.label(p, p.atom_of[slot]);
            }
        }
        for (int a0 = 0; a0 < kChunk * kClusterSize; a0 += 32) {
            const int a = a0 + lane, e = a >> 3;
            const unsigned jc = __shfl_sync(kFull, ent.x, e);
            const unsigned cd = __shfl_sync(kFull, ent.y, e);
            if (e < n_ent) {
                int dx, dy, dz;
                half_shell((int)(cd & 0xffu), dx, dy, dz);
                const int slot = (int)jc * kClusterSize + (a & 7);
                const T4 v = P::pos(p, slot);
                if (FP64) w.jx[a] = P::mk(v.x + T(dx * g.edge[0]), v.y + T(dy * g.edge[1]), v.z + T(dz * g.edge[2]), T(0));
                else w.jx[a] = P::mk(v.x + T((float)dx * g.edge_f[0]), v.y + T((float)dy * g.edge_f[1]),
                                     v.z + T((float)dz * g.edge_f[2]), T(0));
                w.ja[a] = op.label(p, p.atom_of[slot]);
            }
        }
        __syncwarp();
        for (int v = 0; v < n_ent; ++v) {
            const int jcl = (int)__shfl_sync(kFull, ent.x, v);
            const unsigned code = __shfl_sync(kFull, ent.y, v);
            const unsigned mlo = __shfl_sync(kFull, ent.z, v), mhi = __shfl_sync(kFull, ent.w, v);
            if ((mlo | mhi) == 0u) continue;
            const int kdiag = (code & 0xffu) == 0u ? jcl - fc : -1;
            const int j0 = v * kClusterSize + ty;
            const S4 a0 = w.jx[j0], a1 = w.jx[j0 + 4];
            const int b0 = w.ja[j0], b1 = w.ja[j0 + 4];
            const unsigned col0 = ((tx < 4 ? mlo : mhi) >> ((tx & 3) * 8)) & 0xffu;
            const int n_t = (int)__reduce_max_sync(kFull, (unsigned)__popc(col0));
            unsigned kq = s_kq[col0];
            for (int t = 0; t < n_t; ++t) {
                const int k = (int)(kq & 0xfu);
                kq >>= 4;
                const int si = k * kClusterSize + tx;
                const S4 xi = w.ix[si];
                const int ii = w.ia[si];
                const bool dg = k == kdiag;
                op.pair(xi, ii, a0, b0, !dg || tx < ty);
                op.pair(xi, ii, a1, b1, !dg || tx < ty + 4);
            }
        }
    }
    op.finish();
}

template <bool FP64, class Op>
static void launch_walk(const Params& p, cudaStream_t s, int n_sm, Op op, size_t op_smem)
{
    const size_t smem = op_smem + 256 * sizeof(unsigned) + 8 * sizeof(WalkWarp<FP64>);
    const auto f = has_light(p) ? k_walk<FP64, true, Op> : k_walk<FP64, false, Op>;
    cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    // as many blocks as an SM holds: the walks wait on dependent loads
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, 256, smem);
    f<<<n_sm * std::max(per_sm, 1), 256, smem, s>>>(p, op);
}

template <bool FP64>
static void rdf_typed(const Params& p, cudaStream_t s, int n_sm, int n_bins, double r_max, unsigned long long* hist)
{
    RdfOp<FP64> op{};
    op.n_bins = n_bins;
    op.nsp = p.n_species;
    op.rmax2 = (typename Prec<FP64>::T)(r_max * r_max);
    op.inv_dr = (typename Prec<FP64>::T)((double)n_bins / r_max);
    op.hist = hist;
    const size_t nh = (size_t)op.pair_rows() * n_bins;
    const size_t base = kRowBytes + 256 * sizeof(unsigned) + 8 * sizeof(WalkWarp<FP64>);
    const size_t hb = (nh * sizeof(unsigned) + 15) / 16 * 16;
    op.smem_hist = base + hb <= 160 * 1024 ? 1 : 0;
    launch_walk<FP64>(p, s, n_sm, op, kRowBytes + (op.smem_hist ? hb : 0));
}

void launch_rdf(const Params& p, cudaStream_t s, int n_sm, int n_bins, double r_max, unsigned long long* hist)
{
    if (p.precision != 0) rdf_typed<true>(p, s, n_sm, n_bins, r_max, hist);
    else rdf_typed<false>(p, s, n_sm, n_bins, r_max, hist);
}

void launch_frag_link(const Params& p, cudaStream_t s, int n_sm, double r_frag, int* parent)
{
    if (p.precision != 0) {
        FragOp<true> op{r_frag * r_frag, parent, p.n_atoms, p.err};
        launch_walk<true>(p, s, n_sm, op, 0);
    } else {
        FragOp<false> op{(float)(r_frag * r_frag), parent, p.n_atoms, p.err};
        launch_walk<false>(p, s, n_sm, op, 0);
    }
}

template <bool FP64, bool ENERGY, bool HYB>
static size_t pair_smem(int n_ts, int warps)
{
    const size_t tab = ((size_t)n_ts * n_ts * sizeof(typename Prec<FP64>::C2) + 127) / 128 * 128;
    if (FP64) return tab + 256 * sizeof(unsigned) + (size_t)warps * sizeof(Warp64<HYB>);
    return tab + (size_t)warps * sizeof(WarpF32<HYB ? (ENERGY ? 2 : 1) : 0>);
}

// Registers of the mixed-precision force kernel: 96 (20 warps per SM) where
// chunks are plenty; 128 (16 warps, no recomputation) for the hybrid and the
// energy instances, which spill otherwise, and for systems with too few chunks
// to fill more warps (atoms stand for chunks, which are counted on the device after
// the instance has been captured): per launch 1,500 atoms 18.4 (96) and 15.6 us (128; 10.5 since), 8,005
// atoms in unbuffered lists 25.9 and 23.9, 30,000 atoms 64.6 and 65.0.
constexpr int kFewChunksAtoms = 16384;
template <bool FP64, bool ENERGY, bool HYB, bool FEW, bool LIGHT>
static auto pair_kernel()
{
    if constexpr (FP64) return k_pair64<ENERGY, HYB>;
    else return k_pair<ENERGY, HYB, LIGHT, ENERGY || HYB || FEW ? 128 : 96>;
}

constexpr size_t kSmemMax = 227 * 1024;   // shared memory a block may ask for

// Warps of the blocks that a launch shape of `warps` per block is launched with,
// given the block's own LJ table; the shape changes no result.
//   FP64: blocks of 8 warps leave 47 KB for the table (55 type states; 41 with
//   hybrid screening), blocks of 4 take up to 93 (90), of 2 up to 107 (106) and of
//   one up to 114 (113); more blocks of fewer warps replace those that do not fit.
//   Mixed, 96 registers: 20 warps fit an SM's registers, as five blocks of 4 while
//   the five tables are small (up to 28 type states), then as two blocks of 10 (up
//   to 46) or one of 20 (up to 67).  Protein crystal, 43 type states, 199,773
//   atoms: 398.8 us with 16 warps, 363.4 with 20.  The same for blocks of 12, of
//   which an SM would hold one; of 8 it holds two, nearly as good as 20 warps.
template <bool FP64, bool ENERGY, bool HYB, bool FEW>
static int fit_warps(int warps, int n_ts)
{
    if constexpr (FP64) {
        while (warps > 1 && pair_smem<FP64, ENERGY, HYB>(n_ts, warps) > kSmemMax) warps /= 2;
    } else if constexpr (ENERGY && HYB) {   // whose warps take 1 KB more than the forces' that chose the shape
        while (warps % 2 == 0 && pair_smem<FP64, ENERGY, HYB>(n_ts, warps) > kSmemMax) warps /= 2;
    } else if constexpr (!ENERGY && !HYB && !FEW) {
        constexpr int kWarps96 = 20, kSmemSm = 228 * 1024, kSmemBlock = 1024;   // an SM's shared memory, and what a block takes besides its own
        if (warps == 8) return warps;
        for (int w : {4, 10, 20})
            if (pair_smem<FP64, ENERGY, HYB>(n_ts, w) <= kSmemMax && kWarps96 / w * (pair_smem<FP64, ENERGY, HYB>(n_ts, w) + kSmemBlock) <= kSmemSm) return w;
    }
    return warps;
}

template <bool FP64, bool ENERGY, bool HYB, bool FEW, bool LIGHT>
static void set_smem_attr()
{
    static bool done = false;   // one per instantiation
    if (!done) {
        const auto f = pair_kernel<FP64, ENERGY, HYB, FEW, LIGHT>();
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
        cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        done = true;
    }
}

template <bool FP64, bool ENERGY, bool HYB, bool FEW, bool LIGHT>
static void launch_one(const Params& p, cudaStream_t s, int blocks, int warps)
{
    set_smem_attr<FP64, ENERGY, HYB, FEW, LIGHT>();
    const int fit = fit_warps<FP64, ENERGY, HYB, FEW>(warps, p.n_ts_lj);
    if (fit < warps || blocks * warps % fit == 0) {   // (not fewer, larger blocks than the caller's warps fill)
        blocks = (blocks * warps + fit - 1) / fit;
        warps = fit;
    }
    pair_kernel<FP64, ENERGY, HYB, FEW, LIGHT>()<<<blocks, warps * 32, pair_smem<FP64, ENERGY, HYB>(p.n_ts_lj, warps), s>>>(p);
}

template <bool FP64, bool ENERGY, bool HYB, bool FEW>
static int resident_warps(int warps, int n_ts)
{
    set_smem_attr<FP64, ENERGY, HYB, FEW, true>();
    const int fit = fit_warps<FP64, ENERGY, HYB, FEW>(warps, n_ts);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pair_kernel<FP64, ENERGY, HYB, FEW, true>(), fit * 32,
                                                  pair_smem<FP64, ENERGY, HYB>(n_ts, fit));
    return n * fit;
}

// Calls f with the force kernel's instance as compile-time constants.
template <class F>
static void with_instance(bool fp64, bool energy, bool hyb, bool few, F&& f)
{
    using T = std::true_type;
    using N = std::false_type;
    auto eh = [&](auto d, auto w) {
        if (hyb) {
            if (energy) f(d, T{}, T{}, w);
            else f(d, N{}, T{}, w);
        } else {
            if (energy) f(d, T{}, N{}, w);
            else f(d, N{}, N{}, w);
        }
    };
    if (fp64) eh(T{}, N{});
    else if (few && !energy && !hyb) f(N{}, N{}, N{}, T{});
    else eh(N{}, N{});
}

int launch_pair_list(const Params& p, cudaStream_t s, int per_sm, int n_sm)
{
    const int blocks = list_grid(p.list_fused, p.sc_cap, per_sm, n_sm);
    if (p.list_fused) {
        const auto f = has_light(p) ? k_list_fused<true> : k_list_fused<false>;
        f<<<blocks, kListWarps * 32, 0, s>>>(p);
        return 1;
    }
    k_list_count<<<blocks, kListWarps * 32, 0, s>>>(p);
    const int ctas = std::min(kScanCtasMax, (p.sc_cap + 2047) / 2048);
    k_list_scan_sums<<<ctas, 1024, 0, s>>>(p);
    k_list_scan_top<<<1, 1024, 0, s>>>(p, ctas);
    k_list_scan_apply<<<ctas, 1024, 0, s>>>(p);
    k_list_write<<<blocks, kListWarps * 32, 0, s>>>(p);
    return 5;
}

void launch_pair_forces(const Params& p, cudaStream_t s, bool energy, int blocks, int warps)
{
    with_instance(p.precision != 0, energy, p.screening != 0, p.n_atoms <= kFewChunksAtoms,
                  [&](auto fp64, auto en, auto hyb, auto few) {
                      constexpr bool D = decltype(fp64)::value, E = decltype(en)::value, H = decltype(hyb)::value, F = decltype(few)::value;
                      if (D || has_light(p)) launch_one<D, E, H, F, true>(p, s, blocks, warps);
                      else launch_one<D, E, H, F, D>(p, s, blocks, warps);
                  });
}

int pair_resident_warps(bool fp64, bool energy, bool hyb, int warps, int n_ts, int n_atoms)
{
    int n = 0;
    with_instance(fp64, energy, hyb, n_atoms <= kFewChunksAtoms, [&](auto d, auto en, auto h, auto few) {
        n = resident_warps<decltype(d)::value, decltype(en)::value, decltype(h)::value, decltype(few)::value>(warps, n_ts);
    });
    return n;
}

int pair_max_blocks_per_sm(bool fp64, bool energy, bool hyb, int warps, int n_ts, int n_atoms)
{
    return (pair_resident_warps(fp64, energy, hyb, warps, n_ts, n_atoms) + warps - 1) / warps;
}

}  // namespace mdg
