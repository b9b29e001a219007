// The stencil's free-surface variants, a translation unit of their own (they compile beside the others).
#include "fwime_prop.cuh"

namespace fwk {

cudaError_t launch_prop_surface(const PropArgs &a, int nshot, cudaStream_t st)
{
    return dispatch_prop<true>(a, nshot, st);
}

}  // namespace fwk
