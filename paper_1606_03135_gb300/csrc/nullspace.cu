// nullspace.cu -- the traversal and own-stencil kernels that solve in the null space of the
// polynomial constraints (nullspace.cuh), by dimension and team size.
#include <cuda_runtime.h>

#include "rbffd_internal.cuh"
#include "traversal.cuh"

namespace rbffd {

template <int D, bool CH>
static const void* traversal_kernel(int nt) {
    switch (nt) {
        case 32: return (const void*)k_traversal<D, kNull, 32, CH>;
        case 64: return (const void*)k_traversal<D, kNull, 64, CH>;
        case 96: return (const void*)k_traversal<D, kNull, 96, CH>;
        case 128: return (const void*)k_traversal<D, kNull, 128, CH>;
        case 256: return (const void*)k_traversal<D, kNull, 256, CH>;
        case 512: return (const void*)k_traversal<D, kNull, 512, CH>;
        default: return nullptr;
    }
}

const void* null_traversal_kernel(int D, int nt, bool chunked) {
    if (D == 2) return chunked ? traversal_kernel<2, true>(nt) : traversal_kernel<2, false>(nt);
    return chunked ? traversal_kernel<3, true>(nt) : traversal_kernel<3, false>(nt);
}

template <int D>
static const void* fallback_kernel(int nt) {
    switch (nt) {
        case 32: return (const void*)k_fallback_solve<D, kNull, 32>;
        case 128: return (const void*)k_fallback_solve<D, kNull, 128>;
        case 256: return (const void*)k_fallback_solve<D, kNull, 256>;
        case 512: return (const void*)k_fallback_solve<D, kNull, 512>;
        default: return nullptr;
    }
}

const void* null_fallback_kernel(int D, int nt) {
    return D == 2 ? fallback_kernel<2>(nt) : fallback_kernel<3>(nt);
}

}  // namespace rbffd
