// Index arithmetic and launch rules without CUDA types: the same functions on
// the device, in the library's host code and in a plain C++ compiler.
#pragma once

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

}  // namespace mdg
