// nd_cluster_f64.cu -- instantiations of the cluster kernel in FP64.
#include "nd_cluster.cuh"

namespace nd {

// Cluster plans: NC = 8 CTAs for every on-chip size, NC = 16 for P >= 32
// (where the P/2 column slots split over 16 CTAs).
#define ND_CLUSTER_CASES(X)      \
    X(16, 8) X(32, 8) X(64, 8) X(128, 8) X(32, 16) X(64, 16) X(128, 16)

size_t cluster_smem_f64(int P, int D, int Dpad, bool wbuf, int nc)
{
#define X(p, n) if (P == p && nc == n) return cluster_smem_bytes<p, double, n>(D, Dpad, wbuf);
    ND_CLUSTER_CASES(X)
#undef X
    return (size_t)-1;
}

int cluster_max_active_f64(int P, int D, int Dpad, bool wbuf, int nc)
{
#define X(p, n) if (P == p && nc == n) return cluster_max_active_t<p, double, n>(D, Dpad, wbuf);
    ND_CLUSTER_CASES(X)
#undef X
    return 0;
}

cudaError_t launch_cluster_f64(int P, const LaunchArgs &a, int maxD, int maxDpad, int nc)
{
#define X(p, n) if (P == p && nc == n) return launch_cluster_p<p, double, n>(a, maxD, maxDpad);
    ND_CLUSTER_CASES(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace nd
