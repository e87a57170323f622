// Shading with the comparison draws of Sec. 5 and Sec. 7 (single-gated
// Gaussians, Eq. gated; the older form, Eq. oldgated; Wang 2020's
// environment-independent glints) and with the anisotropic grid (footprint
// level, anisotropy and orientation, Sec. 3.3), all with the E1 probabilities
// and the per-pixel intermediates available.  A translation unit of its own so
// that the build compiles it in parallel with the main shading kernels.
#include "glint_shade_pixel.cuh"

namespace {

template <int K, bool INTEGER, int DRAW, int GRID>
__global__ void __launch_bounds__(kShadeNT, shade_min_blocks(K)) k_shade_var(ShadeArgs a) {
    pdl_wait_then_release();
    const long q = (long)blockIdx.x * kShadeNT + threadIdx.x;
    if (q >= a.npix) return;
    shade_pixel<K, INTEGER, true, EV_E1, DRAW, GRID>(a, q);
}

template <int K, int DRAW, int GRID>
cudaError_t launch_kd(const ShadeArgs &a, bool integer, cudaStream_t s) {
    const unsigned grid = (unsigned)((a.npix + kShadeNT - 1) / kShadeNT);
    return launch_pdl(true, integer ? k_shade_var<K, true, DRAW, GRID> : k_shade_var<K, false, DRAW, GRID>, grid,
                      kShadeNT, 0, s, a);
}

template <int K>
cudaError_t launch_k(const ShadeArgs &a, bool integer, int draw, int grid, cudaStream_t s) {
    if (grid) return launch_kd<K, kDrawDual, 1>(a, integer, s);
    if (draw == kDrawSingle) return launch_kd<K, kDrawSingle, 0>(a, integer, s);
    if (draw == kDrawSingleOld) return launch_kd<K, kDrawSingleOld, 0>(a, integer, s);
    return launch_kd<K, kDrawWang, 0>(a, integer, s);
}

}  // namespace

cudaError_t glint_launch_shade_variant(const ShadeArgs &a, int K, bool integer, int draw, int grid, cudaStream_t s) {
    if (a.npix == 0) return cudaSuccess;
    switch (K) {
    case 2: return launch_k<2>(a, integer, draw, grid, s);
    case 4: return launch_k<4>(a, integer, draw, grid, s);
    case 8: return launch_k<8>(a, integer, draw, grid, s);
    case 16: return launch_k<16>(a, integer, draw, grid, s);
    default: return cudaErrorInvalidValue;
    }
}
