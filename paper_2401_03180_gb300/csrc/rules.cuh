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

}  // namespace mdg
