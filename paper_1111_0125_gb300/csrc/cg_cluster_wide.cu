// Instantiations of the cluster solver with FP64 and FP32 inner iterations.
#include "cg_cluster.cuh"

namespace stg {

int cl_active_clusters(int ctas) { return cl_active<P32, 12>(ctas); }

bool cl_granted_wide(int pd, int recon, int per)
{
    if (pd == P64) return recon == 12 ? cl_granted<P64, 12>(per) : cl_granted<P64, 18>(per);
    return recon == 12 ? cl_granted<P32, 12>(per) : cl_granted<P32, 18>(per);
}

cudaError_t cl_dispatch_wide(int pd, int recon, const ClArgs &a, int nsys, int ctas, cudaStream_t s)
{
    if (pd == P64)
        return recon == 12 ? cl_launch_pr<P64, 12>(a, nsys, ctas, s) : cl_launch_pr<P64, 18>(a, nsys, ctas, s);
    return recon == 12 ? cl_launch_pr<P32, 12>(a, nsys, ctas, s) : cl_launch_pr<P32, 18>(a, nsys, ctas, s);
}

}  // namespace stg
