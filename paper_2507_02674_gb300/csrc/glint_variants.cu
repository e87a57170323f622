// Shading with the comparison draws of Sec. 5 and Sec. 7 (single-gated
// Gaussians, Eq. gated; the older form, Eq. oldgated; Wang 2020's
// environment-independent glints) and with the anisotropic grid (footprint
// level, anisotropy and orientation, Sec. 3.3), all with the E1 probabilities.
// As the main kernels they are compiled with and without the per-pixel
// intermediates: without, the draws keep no running addresses and masks (1280 x
// 720, anisotropic grid: K = 8 185.3 to 180.0 us, K = 2 64.8 to 61.1 us, K = 4
// with real counts 117.3 to 107.2 us; single-gated draws, K = 8, 135.9 to 132.0).
// A translation unit of its own so that the build compiles it in parallel with
// the main shading kernels.
#include "glint_shade_pixel.cuh"

namespace {

template <int K, bool INTEGER, bool DEBUG, int DRAW, int GRID>
__global__ void __launch_bounds__(kShadeNT, shade_min_blocks(K)) k_shade_var(ShadeArgs a) {
    pdl_wait_then_release_few();
    const long q = (long)blockIdx.x * kShadeNT + threadIdx.x;
    if (q >= a.npix) return;
    shade_pixel<K, INTEGER, DEBUG, EV_E1, DRAW, GRID>(a, q);
}

template <int K, int DRAW, int GRID>
cudaError_t launch_kd(const ShadeArgs &a, bool integer, bool debug, cudaStream_t s) {
    const unsigned grid = (unsigned)((a.npix + kShadeNT - 1) / kShadeNT);
    auto kernel = integer ? (debug ? k_shade_var<K, true, true, DRAW, GRID> : k_shade_var<K, true, false, DRAW, GRID>)
                          : (debug ? k_shade_var<K, false, true, DRAW, GRID> : k_shade_var<K, false, false, DRAW, GRID>);
    return launch_pdl(true, kernel, grid, kShadeNT, 0, s, a);
}

template <int K>
cudaError_t launch_k(const ShadeArgs &a, bool integer, bool debug, int draw, int grid, cudaStream_t s) {
    if (grid) return launch_kd<K, kDrawDual, 1>(a, integer, debug, s);
    if (draw == kDrawSingle) return launch_kd<K, kDrawSingle, 0>(a, integer, debug, s);
    if (draw == kDrawSingleOld) return launch_kd<K, kDrawSingleOld, 0>(a, integer, debug, s);
    return launch_kd<K, kDrawWang, 0>(a, integer, debug, s);
}

}  // namespace

cudaError_t glint_launch_shade_variant(const ShadeArgs &a, int K, bool integer, bool debug, int draw, int grid,
                                       cudaStream_t s) {
    if (a.npix == 0) return cudaSuccess;
    switch (K) {
    case 2: return launch_k<2>(a, integer, debug, draw, grid, s);
    case 4: return launch_k<4>(a, integer, debug, draw, grid, s);
    case 8: return launch_k<8>(a, integer, debug, draw, grid, s);
    case 16: return launch_k<16>(a, integer, debug, draw, grid, s);
    default: return cudaErrorInvalidValue;
    }
}
