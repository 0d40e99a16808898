// sw_static.cu -- the fixed device scratch of sw_gcr_solve_noalloc.  The arrays
// are part of this translation unit's device code, so they come into being when
// the module is loaded, not through a runtime allocation.  They sit in a file
// of its own so that, with lazy module loading, only programs that use the
// no-allocation solve load it.
#include "../../include/sw_elliptic.h"
#include "sw_common.cuh"
#include "sw_internal.h"

namespace sw {

static __device__ __align__(256) unsigned char g_noalloc_scratch[SW_NOALLOC_SCRATCH_BYTES];

// the nine-point weights of an FP64 solve on a grid without weights of its
// own, for as many points as the work vectors (at least nine doubles a point)
// fit in the scratch for
constexpr size_t NOALLOC_POINTS = SW_NOALLOC_SCRATCH_BYTES / (9 * sizeof(double));
static __device__ __align__(256) unsigned char g_noalloc_weights[NWGT * NOALLOC_POINTS * sizeof(double)];

// The device addresses of the scratch in the current context.  Host code only
// holds stand-ins for the arrays, so the addresses are asked of the runtime on
// every call: a context that was torn down and created again (a device reset,
// a released and re-retained primary context) reloads the module, and the
// arrays may then sit elsewhere.  The lookup allocates nothing.
cudaError_t noalloc_scratch(void **ptr, double **weights)
{
    *ptr = nullptr;
    void *p = nullptr, *w = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e == cudaSuccess && weights) e = cudaGetSymbolAddress(&w, g_noalloc_weights);
    if (e != cudaSuccess) return e;
    *ptr = p;
    if (weights) *weights = (double *)w;
    return cudaSuccess;
}

} // namespace sw
