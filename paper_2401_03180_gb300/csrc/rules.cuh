// Index arithmetic and launch rules without CUDA types: the same functions on
// the device, in the library's host code and in a plain C++ compiler.
#pragma once

#include <cmath>

#if defined(__CUDACC__)
#define MDG_HD __host__ __device__ __forceinline__
#else
#define MDG_HD inline
#endif

namespace mdg {

constexpr int kClusterSize = 8;       // atoms per cluster
constexpr int kSuperClusters = 8;     // K_SC: i-clusters of a super-cluster

// Which i-cluster of the super-cluster that starts at cluster fc a j-cluster jc of
// its own cell is; kNoSelf for none.  The whole difference is compared: a cell may
// hold any number of clusters.
constexpr unsigned kNoSelf = 0xffffu;
MDG_HD unsigned self_cluster(bool own_cell, unsigned jc, unsigned fc)
{
    const unsigned d = jc - fc;
    return own_cell && d < (unsigned)kSuperClusters ? d : kNoSelf;
}

// Padding slots fill a cell's last cluster.  Their records lie far from every atom,
// 1,024 nm apart along x in 64 bits; in 32 bits neighbouring ones coincide from
// slot 2^24 on (beyond 2^34 nm), and a cell's shift may bring those of two cells
// together.  The mixed force kernel evaluates whole cluster tiles, pads included, so
// it stages the pads of the i side on the other side of the origin, out of reach of
// every j-atom and pad; they carry the charge -0, which no atom has.
constexpr double kPadFar = 1.0e6, kPadStep = 1024.0;   // nm
constexpr float kPadCharge = -0.0f;
constexpr float kPadStaged = -1.0e18f;
MDG_HD double pad_x(int slot) { return kPadFar + kPadStep * (double)slot; }
MDG_HD float staged_x(float x, float q) { return std::signbit(q) ? kPadStaged : x; }

// Largest blocks per SM that a caller may pin for blocks of `warps` warps, beside an
// LJ table of n_ts type states.  The limit is a promise of the interface and stands
// apart from the kernels of the day: it is what an SM held (registers, then shared
// memory) of the force kernels with which the interface was first given, whose warps
// took the bytes below.  More blocks than an SM holds of the present ones are
// correct as well: they run one after another and take chunks until none is left.
constexpr int kPinWarpBytes[2][2] = {{8272, 9664}, {15312, 18112}};   // [FP64][hybrid electrostatics]
constexpr int kPinSmWarps[2] = {24, 16};                              // resident warps by registers, [FP64]
constexpr int kPinBlockBytes = 1024 + 1024;                           // a block's lookup table, and what the SM keeps per block
constexpr int kPinSmBytes = 228 * 1024;
inline int pair_pin_limit(bool fp64, bool hyb, int warps, int n_ts)
{
    const int table = (n_ts * n_ts * (fp64 ? 16 : 8) + 127) / 128 * 128;
    const int by_smem = kPinSmBytes / (table + kPinBlockBytes + warps * kPinWarpBytes[fp64][hyb]);
    const int by_regs = kPinSmWarps[fp64] / warps;
    const int n = by_smem < by_regs ? by_smem : by_regs;
    return n > 1 ? n : 1;
}

// Blocks of a list build at `per_sm` blocks per SM: at most a block per super-cluster
// in the one-kernel build, a warp (of eight) per super-cluster in the kernels for
// many of them.
constexpr int kListWarps = 8;
inline int list_grid(bool fused, int sc_cap, int per_sm, int n_sm)
{
    const long long most = fused ? sc_cap : ((long long)sc_cap + kListWarps - 1) / kListWarps;
    const long long n = (long long)per_sm * n_sm;
    return (int)(n < 1 || most < 1 ? 1 : (n < most ? n : most));
}

// Whether the list is built by one kernel, a block per super-cluster (SC), or by five
// that give a warp an SC or a part of one.  The first saves launches and staging, the
// second keeps eight times as many SCs in flight: of `scs` SCs, estimated from the
// cells that the sample fills and its atoms, up to 7,000 take the first where cells hold
// 16 atoms or more, and up to 3,500 where they hold fewer, whose SCs are one cluster of
// work each.  us per step, five kernels and one, lists built at every step: one atom a
// cell 66.4 and 65.2 at 3,427 SCs, 79.6 and 80.3 at 4,989, 174 and 278 at 30,256; eight
// a cell 61.7 and 57.0 at 1,944, 75.2 and 77.1 at 3,796; 27 a cell 161.7 and 143.4 at
// 4,798, 219.7 and 253.6 at 9,752; 64 a cell 253.8 and 235.8 at 6,750; water (170 a
// cell) 572.7 and 547.8 at 5,081.  Beyond a capacity of 32,768 SCs the kernels count
// SCs that a batch's empty cells reserve; 500,001 atoms take 194 us a build in one
// kernel and 186 in five, 2 M atoms 739 and 647, a batch of 300,000 96 and 93.
constexpr int kListFusedScs = 32768;
inline bool list_in_one_kernel(long long cells, long long atoms, int sc_cap)
{
    const long long scs = (cells < atoms ? cells : atoms) + atoms / (kSuperClusters * kClusterSize);
    return sc_cap <= kListFusedScs && scs <= (atoms >= 16 * cells ? 7000 : 3500);
}

// The step kernel of large systems: `wide` from kWideBlocks blocks of kStepAtoms atoms
// per SM on, and there the charge update against a table of the total rates where the
// table (two entries per replica and type state) is no larger than the sample; an
// atom's own rates cost about as much as an entry.  8,000 replicas of 10 atoms, 43
// type states: the table alone took 20 us of a step kernel of 31, 12 without it.
constexpr int kStepAtoms = 32;
constexpr int kWideBlocks = 16;
inline bool step_is_wide(long long atoms, int n_sm) { return (atoms + kStepAtoms - 1) / kStepAtoms >= (long long)kWideBlocks * n_sm; }
inline bool rates_by_table(long long atoms, long long replicas, int n_ts, int n_sm)
{
    return step_is_wide(atoms, n_sm) && 2 * replicas * n_ts <= atoms;
}

}  // namespace mdg
