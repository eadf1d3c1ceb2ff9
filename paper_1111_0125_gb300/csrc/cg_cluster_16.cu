// Instantiations of the cluster solver with 16-bit inner iterations.
#include "cg_cluster.cuh"

namespace stg {

bool cl_granted_16(int pd, int recon, int per)
{
    const bool r12 = recon == 12;
    if (pd == P16) return r12 ? cl_granted<P16, 12>(per) : cl_granted<P16, 18>(per);
    if (pd == PB16) return r12 ? cl_granted<PB16, 12>(per) : cl_granted<PB16, 18>(per);
    return r12 ? cl_granted<PX16, 12>(per) : cl_granted<PX16, 18>(per);
}

cudaError_t cl_dispatch_16(int pd, int recon, const ClArgs &a, int nsys, int ctas, cudaStream_t s)
{
    const bool r12 = recon == 12;
    if (pd == P16) return r12 ? cl_launch_pr<P16, 12>(a, nsys, ctas, s) : cl_launch_pr<P16, 18>(a, nsys, ctas, s);
    if (pd == PB16) return r12 ? cl_launch_pr<PB16, 12>(a, nsys, ctas, s) : cl_launch_pr<PB16, 18>(a, nsys, ctas, s);
    return r12 ? cl_launch_pr<PX16, 12>(a, nsys, ctas, s) : cl_launch_pr<PX16, 18>(a, nsys, ctas, s);
}

}  // namespace stg
