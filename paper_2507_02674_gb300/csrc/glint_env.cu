// Per-environment preprocessing: radiance levels, fuzzy weights, pyramid and
// filtered maps (Sec. 4 "Discrete Radiance Levels", "Fuzzy Indicator
// Functions", Eq. wkdefpractice, "Integrated NDF" Eq. rtiblndf; Sec. 3.4
// Eq. rtibl).
//
// Data layout in HBM.  Pyramid: per level, the texels' colour (R, G, B, 0),
// one float4 each, then their weights w_1..w_K, Cpad/4 - 1 float4 each
// (Cpad = 4 ceil((3+K)/4); 32 bytes at K = 8, read with one 256-bit load);
// levels concatenated.  Filtered maps: R levels of W_r/2 x W_r texels, each
// texel the record (R, G, B, w_1..w_K, 0 padding) of Cpad floats (or an fp32
// colour and K codes for a compressed format), levels concatenated; beside
// them a weights-only copy (Cpad/4 - 1 float4 a texel, the weights as stored).
// Brightness min/max go through a small per-block scratch array and a
// finished-block counter.
#include <stdio.h>

#include <algorithm>

#include "glint_internal.cuh"

using namespace glint;

namespace {

constexpr int kNT = 256;

__device__ __forceinline__ float4 load_texel(const void *texels, int fmt, long i) {
    if (fmt == GLINT_FMT_RGBA16F) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(texels) + i);
        const __half2 rg = *reinterpret_cast<const __half2 *>(&raw.x);
        const __half2 ba = *reinterpret_cast<const __half2 *>(&raw.y);
        const float2 f0 = __half22float2(rg), f1 = __half22float2(ba);
        return make_float4(f0.x, f0.y, f1.x, f1.y);
    }
    return __ldg(reinterpret_cast<const float4 *>(texels) + i);
}

// Rec. 709 luminance of scaled radiance, clamped at 0.
__device__ __forceinline__ float brightness(float4 t, float scale) {
    float y = 0.2126f * (t.x * scale) + 0.7152f * (t.y * scale) + 0.0722f * (t.z * scale);
    return fmaxf(y, 0.f);
}

// Step 2 from the per-block (min, max) pairs: lo = max(min Y, ell),
// hi = max(max Y, lo); L_1 = 0, L_k = lo (hi/lo)^((k-1)/(K-1)) =
// exp(lerp(ln lo, ln hi, (k-1)/(K-1))).  Run by one block.
__device__ void levels_from_partials(const float2 *partial, int nblk, int K, float ell, float *levels) {
    float lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x; i < nblk; i += kNT) {
        const float2 v = __ldcg(partial + i);  // written by other blocks: read from L2
        lo = fminf(lo, v.x);
        hi = fmaxf(hi, v.y);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __shared__ float2 red[kNT / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(lo, hi);
    __syncthreads();
    if ((int)threadIdx.x < K) {
        float mn = red[0].x, mx = red[0].y;
        for (int w = 1; w < kNT / 32; ++w) {
            mn = fminf(mn, red[w].x);
            mx = fmaxf(mx, red[w].y);
        }
        lo = fmaxf(mn, ell);
        hi = fmaxf(mx, lo);
        const float l2 = log2f(hi / lo);
        const int k = (int)threadIdx.x + 1;
        const float a = (float)(k - 1) / (float)(K - 1);
        levels[k - 1] = k == 1 ? 0.f : lo * exp2f(a * l2);
        if (k == 1) {
            levels[K] = lo;
            levels[K + 1] = hi;
        }
    }
}

// Two adjacent texels 2 i, 2 i + 1 in 16-byte loads (16-byte aligned texels).
__device__ __forceinline__ void load_texel_pair(const void *texels, int fmt, long i, float4 &a, float4 &b) {
    if (fmt == GLINT_FMT_RGBA16F) {
        const uint4 raw = __ldg(reinterpret_cast<const uint4 *>(texels) + i);
        const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
        const float2 f0 = __half22float2(h[0]), f1 = __half22float2(h[1]), f2 = __half22float2(h[2]),
                     f3 = __half22float2(h[3]);
        a = make_float4(f0.x, f0.y, f1.x, f1.y);
        b = make_float4(f2.x, f2.y, f3.x, f3.y);
    } else {
        a = __ldg(reinterpret_cast<const float4 *>(texels) + 2 * i);
        b = __ldg(reinterpret_cast<const float4 *>(texels) + 2 * i + 1);
    }
}

// Steps 1 and 2: per-block min / max of the brightness into the scratch
// array; the last block to finish (counted in *done, which it resets) turns
// the pairs into the levels, a thread a level.  Latency-bound (the map is a few
// microseconds of HBM traffic): kMinMaxPairs independent loads of two texels a
// thread.  wide: the texels are 16-byte aligned (n is even, a map being twice as
// wide as high).
constexpr int kMinMaxPairs = 4;
__global__ void __launch_bounds__(kNT) k_minmax(const void *__restrict__ texels, int fmt, long n, float scale,
                                                  float2 *__restrict__ partial, unsigned *__restrict__ done, int K,
                                                  float ell, float *__restrict__ levels, bool wide) {
    pdl_release();
    float lo = INFINITY, hi = -INFINITY;
    if (wide) {
        for (long i0 = (long)blockIdx.x * (kNT * kMinMaxPairs) + threadIdx.x; i0 < n / 2;
             i0 += (long)gridDim.x * (kNT * kMinMaxPairs)) {
            float4 t[2 * kMinMaxPairs];
#pragma unroll
            for (int j = 0; j < kMinMaxPairs; ++j) {  // past the end: the first pair once more
                const long i = i0 + j * kNT;
                load_texel_pair(texels, fmt, i < n / 2 ? i : i0, t[2 * j], t[2 * j + 1]);
            }
#pragma unroll
            for (int j = 0; j < 2 * kMinMaxPairs; ++j) {
                const float y = brightness(t[j], scale);
                lo = fminf(lo, y);
                hi = fmaxf(hi, y);
            }
        }
    } else {
        for (long i = (long)blockIdx.x * kNT + threadIdx.x; i < n; i += (long)gridDim.x * kNT) {
            const float y = brightness(load_texel(texels, fmt, i), scale);
            lo = fminf(lo, y);
            hi = fmaxf(hi, y);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __shared__ float2 red[kNT / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(lo, hi);
    __syncthreads();
    if (threadIdx.x < 32) {
        float2 v = threadIdx.x < kNT / 32 ? red[threadIdx.x] : make_float2(INFINITY, -INFINITY);
        for (int o = 16; o > 0; o >>= 1) {
            v.x = fminf(v.x, __shfl_xor_sync(0xffffffffu, v.x, o));
            v.y = fmaxf(v.y, __shfl_xor_sync(0xffffffffu, v.y, o));
        }
        if (threadIdx.x == 0) partial[blockIdx.x] = v;
    }
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();  // this block's pair is visible before it is counted
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    levels_from_partials(partial, gridDim.x, K, ell, levels);
    if (threadIdx.x == 0) *done = 0u;
}

// One texel's channels in the pyramid's slot order (R, G, B, 0, w_1 .. w_K, 0
// padding): its colour and the fuzzy weights of the two levels bracketing its
// brightness (Eq. wkdefpractice).
struct TexelChannels {
    float R, G, B;
    int j;         // w_{j+1} = wa, w_{j+2} = wb, the others 0
    float wa, wb;
    __device__ __forceinline__ float weight(int k) const { return k == j ? wa : k == j + 1 ? wb : 0.f; }
    __device__ __forceinline__ float4 slot(int c) const {
        return c == 0 ? make_float4(R, G, B, 0.f)
                      : make_float4(weight(4 * c - 4), weight(4 * c - 3), weight(4 * c - 2), weight(4 * c - 1));
    }
};
__device__ __forceinline__ TexelChannels texel_channels(float4 t, float scale, int K, const float *L, bool log_w) {
    TexelChannels o;
    o.R = t.x * scale; o.G = t.y * scale; o.B = t.z * scale;
    const float Y = fmaxf(0.2126f * o.R + 0.7152f * o.G + 0.0722f * o.B, 0.f);
    // bracket: largest j in [0, K-2] with L[j] <= Y; Y >= L[K-1] -> w_K = 1
    int j = 0;
    for (int k = 1; k < K - 1; ++k)
        if (L[k] <= Y) j = k;
    const bool top = Y >= L[K - 1];
    // log space (optional, Sec. 7): between L_j > 0 and L_{j+1}; linear below L_2 (L_1 = 0)
    const float tt = (log_w && j > 0) ? (logf(Y) - logf(L[j])) / (logf(L[j + 1]) - logf(L[j]))
                                      : (Y - L[j]) / (L[j + 1] - L[j]);
    o.j = top ? K - 2 : j;
    o.wa = top ? 0.f : 1.f - tt;
    o.wb = top ? 1.f : tt;
    return o;
}

// Slot c of texel (x, y) of a pyramid level of width W (float4 units of the
// split storage): slot 0 is the colour (R, G, B, 0) at rgb4 + y W + x, slots 1
// .. C4-1 the weights at w4 + (y W + pyr_column(x, y, C4 - 1)) (C4 - 1) + c - 1.
template <int C4>
__device__ __forceinline__ size_t pyr_slot(size_t rgb4, size_t w4, int x, int y, int W, int c) {
    const size_t row = (size_t)y * W;
    return c == 0 ? rgb4 + row + x : w4 + (row + pyr_column(x, y, C4 - 1)) * (C4 - 1) + (c - 1);
}

// Row weights of a level built from a parent of height Hp: of the two parent
// rows under row Y and the reciprocal of their sum over the 2 x 2 children.  A
// row spanning [theta0, theta1] weighs cos theta0 - cos theta1 = 2 sin(mid)
// sin(half), written as a product to stay accurate near the poles.
__device__ __forceinline__ float3 row_weights(int Y, int Hp) {
    const float half = 0.5f * kPi / (float)Hp;
    const float w0 = sinf((2.f * Y + 0.5f) * (kPi / (float)Hp)) * sinf(half);
    const float w1 = sinf((2.f * Y + 1.5f) * (kPi / (float)Hp)) * sinf(half);
    return make_float3(w0, w1, 1.f / (2.f * (w0 + w1)));
}

// Solid-angle weighted mean of the 2 x 2 children a0 a1 / b0 b1.
__device__ __forceinline__ float mean4(float a0, float a1, float b0, float b1, float w0, float w1, float inv) {
    return (w0 * (a0 + a1) + w1 * (b0 + b1)) * inv;
}
__device__ __forceinline__ float4 mean4(const float4 &a0, const float4 &a1, const float4 &b0, const float4 &b1,
                                        const float3 &w) {
    return make_float4(mean4(a0.x, a1.x, b0.x, b1.x, w.x, w.y, w.z), mean4(a0.y, a1.y, b0.y, b1.y, w.x, w.y, w.z),
                       mean4(a0.z, a1.z, b0.z, b1.z, w.x, w.y, w.z), mean4(a0.w, a1.w, b0.w, b1.w, w.x, w.y, w.z));
}

// Steps 3 and 4: pyramid.  A block takes a 32 x 32 tile (T, a power of two; less
// on maps below 32 rows) of pyramid level m and builds log2 T further levels.
// Each thread holds a 2 x 2 quad of the tile in registers, writes it if the
// texels' channels are computed here (m = 0), and writes the quad's mean, level
// m + 1, to memory and to shared memory, where the upper levels are reduced.
// (With the whole tile staged in shared memory, 60 KB a block at K = 8, only
// three blocks fit an SM, 456 of the 512 of a 1024 x 512 map: two waves.)
// Latency bounds it at small maps, so the row weights of all levels are computed
// at the start and the texels fetched before the wait for the levels; at large
// ones the stores, so they are whole 32-byte sectors a thread (16-byte pieces of
// two texels a thread left half-written sectors).  1024 x 512, K = 8: 25.8 ->
// 17.4 us; 2048 x 1024, K = 16 (223 MB written): 111 -> 75 us.  With tail_to > m + nlev the last block to finish
// (counted in *done, which it resets) builds levels m + nlev + 1 .. tail_to from
// level m + nlev, which every block has written by then: the first from memory,
// the others from shared memory (at most kPyrTailTexels / 4 texels).
constexpr long kPyrTailTexels = 2048;

template <int C4>
constexpr size_t pyramid_smem() {  // level m + 1 of a tile (256 texels) and m + 2, or the first two tail levels
    return sizeof(float4) * C4 * (kPyrTailTexels / 4 + kPyrTailTexels / 16);
}

template <bool FROM_TEXELS, int C4>
__global__ void __launch_bounds__(kNT, 4) k_pyramid(
    const void *__restrict__ texels, int fmt, float scale, int K, const float *__restrict__ levels,
    float4 *__restrict__ pyr, const size_t *__restrict__ rgb4, const size_t *__restrict__ w4, int m, int Ws, int Hs,
    int T, int nlev, int log_w, int tail_to, unsigned *__restrict__ done, bool wide) {
    extern __shared__ float4 smem4[];
    __shared__ float L[GLINT_MAX_K];
    __shared__ float3 rw[32];  // rows of levels m + 1, m + 2, ..: T/2, T/4, .., 1 of them
    // T is a power of two (2^nlev): tile coordinates by shifts and masks
    const int tiles_x = Ws >> nlev;
    const int tx0 = ((int)blockIdx.x & (tiles_x - 1)) << nlev, ty0 = ((int)blockIdx.x / tiles_x) << nlev;
    {
        const int i = (int)threadIdx.x - (kNT - 32);  // the last warp
        if (i >= 0 && i < T - 1) {
            int l = 1, first = 0;
            while (i >= first + (T >> l)) first += T >> l++;
            rw[i] = row_weights((ty0 >> l) + i - first, Hs >> (l - 1));
        }
    }
    // The first quad's texels are fetched before the wait on the kernel that finds
    // the levels (which waited for whatever wrote them).
    float4 tex[4] = {};
    const int cur0 = T / 2;
    if (FROM_TEXELS && (int)threadIdx.x < cur0 * cur0) {
        const int x = threadIdx.x & (cur0 - 1), y = threadIdx.x >> (nlev - 1);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const long g = (long)(ty0 + 2 * y + r) * Ws + tx0 + 2 * x;
            if (wide) {
                load_texel_pair(texels, fmt, g / 2, tex[2 * r], tex[2 * r + 1]);
            } else {
                tex[2 * r] = load_texel(texels, fmt, g);
                tex[2 * r + 1] = load_texel(texels, fmt, g + 1);
            }
        }
    }
    pdl_wait_then_release();
    if (FROM_TEXELS && threadIdx.x < K) L[threadIdx.x] = __ldcg(levels + threadIdx.x);
    __syncthreads();
    // level m + 1 from quads (one a thread: a tile has at most 16 x 16)
    int cur = cur0, row0 = 0;
    float4 *bufA = smem4, *bufB = smem4 + (size_t)cur * cur * C4;
    static_assert(kNT >= 16 * 16, "a thread a quad");
    if (const int i = threadIdx.x; i < cur * cur) {
        const int x = i & (cur - 1), y = i >> (nlev - 1);
        const int gx = tx0 + 2 * x, gy = ty0 + 2 * y;
        TexelChannels t[4];  // texels (0,0) (1,0) (0,1) (1,1)
        if (FROM_TEXELS) {
#pragma unroll
            for (int h = 0; h < 4; ++h) t[h] = texel_channels(tex[h], scale, K, L, log_w != 0);
        }
        // Whole 32-byte sectors at a time: the colours of two texels, the weights
        // of one (two at K <= 4); every texel with an even column is 32-byte aligned.
        const float3 w = rw[y];
        float4 v[4], u[4];  // a slot of the four texels, and the next
        auto slot = [&](int c, float4 (&o)[4]) {
#pragma unroll
            for (int h = 0; h < 4; ++h)
                o[h] = FROM_TEXELS
                           ? t[h].slot(c)
                           : __ldcg(pyr + pyr_slot<C4>(rgb4[m], w4[m], gx + (h & 1), gy + (h >> 1), Ws, c));
        };
        auto put = [&](int r, int h, int c, const float4 &a, const float4 &b) {
            if (FROM_TEXELS) st8(pyr + pyr_slot<C4>(rgb4[0], w4[0], gx + h, gy + r, Ws, c), a, b);
        };
        auto up = [&](int c) { return pyr + pyr_slot<C4>(rgb4[m + 1], w4[m + 1], gx >> 1, gy >> 1, Ws >> 1, c); };
        slot(0, v);
        put(0, 0, 0, v[0], v[1]);
        put(1, 0, 0, v[2], v[3]);
        *up(0) = bufA[i * C4] = mean4(v[0], v[1], v[2], v[3], w);
        if constexpr (C4 == 2) {
            slot(1, v);
            put(0, 0, 1, v[0], v[1]);
            put(1, 0, 1, v[2], v[3]);
            *up(1) = bufA[i * C4 + 1] = mean4(v[0], v[1], v[2], v[3], w);
        } else {
#pragma unroll
            for (int c = 1; c < C4; c += 2) {
                slot(c, v);
                slot(c + 1, u);
#pragma unroll
                for (int h = 0; h < 4; ++h) put(h >> 1, h & 1, c, v[h], u[h]);
                const float4 r0 = mean4(v[0], v[1], v[2], v[3], w), r1 = mean4(u[0], u[1], u[2], u[3], w);
                bufA[i * C4 + c] = r0;
                bufA[i * C4 + c + 1] = r1;
                st8(up(c), r0, r1);
            }
        }
    }
    __syncthreads();
    for (int l = 2; l <= nlev; ++l) {
        const int nxt = cur / 2, lg = nlev - l;  // nxt = 2^lg
        row0 += cur;
        const int X0 = tx0 >> l, Y0 = ty0 >> l;
        for (int i = threadIdx.x; i < nxt * nxt * C4; i += kNT) {
            const int c = i % C4, t = i / C4;  // C4 is a constant: no division
            const int x = t & (nxt - 1), y = t >> lg;
            const float4 *p = bufA + ((2 * y) * cur + 2 * x) * C4 + c;
            const float4 r = mean4(p[0], p[C4], p[cur * C4], p[(cur + 1) * C4], rw[row0 + y]);
            bufB[t * C4 + c] = r;
            pyr[pyr_slot<C4>(rgb4[m + l], w4[m + l], X0 + x, Y0 + y, Ws >> l, c)] = r;
        }
        __syncthreads();  // (also: every store of the level issued before the block is counted as done)
        float4 *tmp = bufA;
        bufA = bufB;
        bufB = tmp;
        cur = nxt;
    }
    if (tail_to <= m + nlev) return;
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();  // this block's levels are visible before it is counted
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    int Wc = Ws >> nlev, Hc = Hs >> nlev;  // level m + nlev, the parent of the first tail level
    bufA = smem4;
    bufB = smem4 + (size_t)C4 * (kPyrTailTexels / 4);
    for (int l = m + nlev + 1; l <= tail_to; ++l) {
        const int Wd = Wc / 2, Hd = Hc / 2;
        const bool first = l == m + nlev + 1;
        float4 *dst = ((l - m - nlev) & 1) ? bufA : bufB;
        const float4 *src = ((l - m - nlev) & 1) ? bufB : bufA;
        for (int i = threadIdx.x; i < Wd * Hd * C4; i += kNT) {
            const int c = i % C4, t = i / C4;
            const int x = t & (Wd - 1), Y = t / Wd;
            const float3 w = row_weights(Y, Hc);
            float4 ch[4];
            if (first) {
                const size_t r4 = rgb4[l - 1], ww4 = w4[l - 1];
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    ch[h] = __ldcg(pyr + pyr_slot<C4>(r4, ww4, 2 * x + (h & 1), 2 * Y + (h >> 1), Wc, c));
            } else {
                const float4 *p = src + ((2 * Y) * Wc + 2 * x) * C4 + c;
                ch[0] = p[0]; ch[1] = p[C4]; ch[2] = p[Wc * C4]; ch[3] = p[(Wc + 1) * C4];
            }
            const float4 r = mean4(ch[0], ch[1], ch[2], ch[3], w);
            dst[t * C4 + c] = r;
            pyr[pyr_slot<C4>(rgb4[l], w4[l], x, Y, Wd, c)] = r;
        }
        __syncthreads();  // level l complete before it is read
        Wc = Wd;
        Hc = Hd;
    }
    if (threadIdx.x == 0) *done = 0u;
}

// Step 5a: filter sample table (Hammersley points mapped through the GGX
// distribution of microfacet normals weighted by cos theta_h):
// u1 = (j+1/2)/S, u2 = radical inverse of j, cos^2 th = (1-u1)/(1+(a^2-1)u1),
// reflected direction weights (sin 2th cos ph, sin 2th sin ph, cos 2th) in the
// frame (e1, e2, r), valid iff cos 2th > 0 (a prefix of j), and the pyramid
// level lod = 0.5 log2(Omega_s / Omega_0) - 1/2 with Omega_s = 4/(S D(h))
// (the bias of filtered importance sampling that keeps the filtered maps
// closest to the exact convolution on maps with bright suns).
__global__ void k_filter_table(int R, int S, float s_min, float s_max, int W, int H, int M, float4 *table,
                               int *nvalid) {
    const int r = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const float sr = (R > 1) ? s_min + (s_max - s_min) * (float)r / (float)(R - 1) : s_min;
    const float alpha = sr * sr, a2 = alpha * alpha;
    // cos^2 = (1-u)/(1-u+a^2 u), sin^2 = a^2 u/(1-u+a^2 u), cos 2th = (1-u-a^2 u)/(1-u+a^2 u):
    // each a ratio of sums of non-negative terms (no cancellation in FP32).
    if (j == 0) {
        int nv = 0;
        for (int k = 0; k < S; ++k) {
            const float u1 = ((float)k + 0.5f) / (float)S;
            if ((1.f - u1) - a2 * u1 > 0.f) ++nv;
        }
        nvalid[r] = nv;
    }
    if (j >= S) return;
    const float u1 = ((float)j + 0.5f) / (float)S;
    const float u2 = (float)__brev((unsigned)j) * 0x1p-32f;
    const float den = (1.f - u1) + a2 * u1;
    const float c2 = (1.f - u1) / den;
    const float s2 = a2 * u1 / den;
    const float cos2t = ((1.f - u1) - a2 * u1) / den;
    float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
    if (cos2t > 0.f) {
        const float sin2t = 2.f * sqrtf(c2 * s2);
        float sp, cp;
        sincosf(kTwoPi * u2, &sp, &cp);
        const float d = s2 + a2 * c2;  // = c2 (a^2 - 1) + 1
        const float D = a2 / (kPi * d * d);
        const float omega_s = 4.f / ((float)S * D);
        const float omega0 = 4.f * kPi / ((float)W * (float)H);
        float lod = 0.5f * log2f(omega_s / omega0) - 0.5f;
        lod = fminf(fmaxf(lod, 0.f), (float)(M - 1));
        e = make_float4(sin2t * cp, sin2t * sp, cos2t, lod);
    }
    table[(size_t)r * S + j] = e;
}

// Step 5b: filtered maps.  Level r is a W_r x W_r/2 equirect grid; the
// levels are concatenated and the grid of blocks runs over all of them (block
// ranges per level in FilterLevels).  kFilterSplit adjacent threads per output
// texel share its samples; their sums are combined with shuffles.  Result: the
// mean over the level's valid samples of the trilinear pyramid look-up at
// w_i = a e1 + b e2 + c r, where r is the texel direction, e1 = d r / d theta,
// e2 = d r / d phi / sin theta.
struct FilterLevels {
    int nlev;
    int width[33];
    int blk[33];          // first block of level r; blk[nlev] = total blocks
    long long off[33];    // first texel of level r
};

constexpr int kFilterSplit = 2;  // threads per output texel (samples strided over them)

// Filtered texel `at` from the sums over its nv samples: the record in the
// stored format and the weights-only copy.
template <int C4>
__device__ __forceinline__ void store_filtered(const float4 &accr, const float4 *accw, int nv, size_t at,
                                               float4 *__restrict__ out, float4 *__restrict__ outw, int wfmt, int rec4,
                                               int K) {
    constexpr int KW4 = C4 - 1;
    // back to the record layout (R, G, B, W_1 .. W_K, zero padding)
    float4 acc[C4];
    {
        float ch[4 * C4];
        ch[0] = accr.x; ch[1] = accr.y; ch[2] = accr.z;
#pragma unroll
        for (int c = 0; c < KW4; ++c) {
            ch[3 + 4 * c] = accw[c].x; ch[4 + 4 * c] = accw[c].y; ch[5 + 4 * c] = accw[c].z; ch[6 + 4 * c] = accw[c].w;
        }
        ch[4 * C4 - 1] = 0.f;
#pragma unroll
        for (int c = 0; c < C4; ++c) acc[c] = make_float4(ch[4 * c], ch[4 * c + 1], ch[4 * c + 2], ch[4 * c + 3]);
    }
    const float inv = nv > 0 ? 1.f / (float)nv : 0.f;
    const int kw4 = (K + 3) / 4;
    float4 *ow = outw + at * kw4;
    if (wfmt == GLINT_WFMT_F32) {
        float4 *o = out + at * C4;
        float ch[C4 * 4 + 4];
#pragma unroll
        for (int c = 0; c < C4; ++c) {
            o[c] = make_float4(acc[c].x * inv, acc[c].y * inv, acc[c].z * inv, acc[c].w * inv);
            ch[4 * c] = acc[c].x * inv; ch[4 * c + 1] = acc[c].y * inv;
            ch[4 * c + 2] = acc[c].z * inv; ch[4 * c + 3] = acc[c].w * inv;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) ch[C4 * 4 + i] = 0.f;
#pragma unroll
        for (int c = 0; c < C4; ++c)  // weights w_k are channels 3 + k; zero past K
            if (c < kw4)
                ow[c] = make_float4(4 * c < K ? ch[3 + 4 * c] : 0.f, 4 * c + 1 < K ? ch[4 + 4 * c] : 0.f,
                                    4 * c + 2 < K ? ch[5 + 4 * c] : 0.f, 4 * c + 3 < K ? ch[6 + 4 * c] : 0.f);
        return;
    }
    // compressed record: (R, G, B, 0) float32, then K weight codes
    float ch[C4 * 4];
#pragma unroll
    for (int c = 0; c < C4; ++c) {
        ch[4 * c] = acc[c].x * inv; ch[4 * c + 1] = acc[c].y * inv;
        ch[4 * c + 2] = acc[c].z * inv; ch[4 * c + 3] = acc[c].w * inv;
    }
    float4 *o = out + at * rec4;
    o[0] = make_float4(ch[0], ch[1], ch[2], 0.f);
    uint32_t words[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    float dec[C4 * 4];  // the weights as the stored codes decode
#pragma unroll
    for (int k = 0; k < C4 * 4; ++k) dec[k] = 0.f;
#pragma unroll
    for (int k = 0; k < C4 * 4 - 3; ++k) {
        if (k >= K) break;
        const float wv = fminf(fmaxf(ch[3 + k], 0.f), 1.f);
        if (wfmt == GLINT_WFMT_UNORM8) {
            const uint32_t c8 = __float2uint_rn(wv * 255.f) & 0xffu;
            words[k / 4] |= c8 << (8 * (k % 4));
            dec[k] = (float)c8 * (1.f / 255.f);
        } else {
            const uint32_t c16 = (wfmt == GLINT_WFMT_F16) ? (uint32_t)__half_as_ushort(__float2half_rn(ch[3 + k]))
                                                         : (__float2uint_rn(wv * 65535.f) & 0xffffu);
            words[k / 2] |= c16 << (16 * (k % 2));
            dec[k] = (wfmt == GLINT_WFMT_F16) ? __half2float(__ushort_as_half((unsigned short)c16))
                                              : (float)c16 * (1.f / 65535.f);
        }
    }
#pragma unroll
    for (int c = 0; c < C4; ++c)
        if (c < kw4) ow[c] = make_float4(dec[4 * c], dec[4 * c + 1], dec[4 * c + 2], dec[4 * c + 3]);
    uint4 *q = reinterpret_cast<uint4 *>(o + 1);
    for (int i = 0; i < rec4 - 1; ++i) q[i] = make_uint4(words[4 * i], words[4 * i + 1], words[4 * i + 2], words[4 * i + 3]);
}

// One sample's trilinear look-up at direction (dx, dy, dz): the bilinear values
// of the two levels bracketing lod, colour and weights apart (the pyramid's
// split storage); sink(wl, v, u) takes them in order.  A level that weighs
// nothing (lod at either end of the pyramid) is not read.
template <int C4, class Sink>
__device__ __forceinline__ void filter_sample(const float4 *__restrict__ pyr, const size_t *__restrict__ rgb4,
                                              const size_t *__restrict__ w4, int W, int H, int M, float dx, float dy,
                                              float dz, float lod, Sink &&sink) {
    constexpr int KW4 = C4 - 1;
    const int m0 = (int)floorf(lod);
    const float f = lod - (float)m0;
    const int m1 = min(m0 + 1, M - 1);
    const float th_i = acosf(fminf(fmaxf(dy, -1.f), 1.f));
    float ph_i = atan2f(dz, dx);
    if (ph_i < 0.f) ph_i += kTwoPi;
#pragma unroll
    for (int lv = 0; lv < 2; ++lv) {
        if (lv == 1 && f == 0.f) break;
        const int m = lv ? m1 : m0;
        const float wl = lv ? f : 1.f - f;
        const int Wm = W >> m, Hm = H >> m;
        const float xx = ph_i * (kInvTwoPi * (float)Wm) - 0.5f;
        const float yy = th_i * (kInvPi * (float)Hm) - 0.5f;
        const Taps tp = equirect_taps(xx, yy, Wm, Hm);
        const float4 *prgb = pyr + rgb4[m], *pw = pyr + w4[m];
        const int idx[4] = {tp.i00, tp.i01, tp.i10, tp.i11};
        // pyr_column of the weights
        const int s0 = KW4 >= 2 && (tp.i00 & Wm) ? 2 : 0, s1 = KW4 >= 2 && (tp.i10 & Wm) ? 2 : 0;
        const int widx[4] = {tp.i00 ^ s0, tp.i01 ^ s0, tp.i10 ^ s1, tp.i11 ^ s1};
        float4 tr[4], tw[4][KW4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            tr[j] = __ldg(prgb + idx[j]);
            ldg_texel<KW4>(pw + (size_t)widx[j] * KW4, tw[j]);
        }
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u[KW4];
        v = fma4(tp.w00, tr[0], v);
        v = fma4(tp.w01, tr[1], v);
        v = fma4(tp.w10, tr[2], v);
        v = fma4(tp.w11, tr[3], v);
#pragma unroll
        for (int c = 0; c < KW4; ++c) {
            u[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            u[c] = fma4(tp.w00, tw[0][c], u[c]);
            u[c] = fma4(tp.w01, tw[1][c], u[c]);
            u[c] = fma4(tp.w10, tw[2][c], u[c]);
            u[c] = fma4(tp.w11, tw[3][c], u[c]);
        }
        sink(lv, wl, v, u);
    }
}

// Frame of an output texel: its direction r and e1 = d r / d theta, e2 =
// d r / d phi / sin theta (e2.y = 0).
struct FilterFrame {
    float rx, ry, rz, e1x, e1y, e1z, e2x, e2z;
    __device__ __forceinline__ FilterFrame(int x, int y, int Wo, int Ho) {
        const float th = kPi * ((float)y + 0.5f) / (float)Ho;
        const float ph = kTwoPi * ((float)x + 0.5f) / (float)Wo;
        float st, ct, sp, cp;
        sincosf(th, &st, &ct);
        sincosf(ph, &sp, &cp);
        rx = st * cp; ry = ct; rz = st * sp;
        e1x = ct * cp; e1y = -st; e1z = ct * sp;
        e2x = -sp; e2z = cp;
    }
};

template <int C4>
__global__ void __launch_bounds__(128) k_filter(const float4 *__restrict__ pyr, const size_t *__restrict__ rgb4,
                                                  const size_t *__restrict__ w4,
                                                  int W, int H, int M, const float4 *__restrict__ table,
                                                  const int *__restrict__ nvalid, int S, const FilterLevels fl,
                                                  float4 *__restrict__ out, float4 *__restrict__ outw, int wfmt,
                                                  int rec4, int K) {
    extern __shared__ float4 tab[];
    int r = 0;
    while (r + 1 < fl.nlev && (int)blockIdx.x >= fl.blk[r + 1]) ++r;
    const int Wo = fl.width[r], Ho = Wo / 2;
    const int nv = nvalid[r];  // (the table is the environment's own since its creation)
    for (int k = threadIdx.x; k < nv; k += blockDim.x) tab[k] = table[(size_t)r * S + k];
    __syncthreads();
    const int g = threadIdx.x % kFilterSplit;
    const int t = ((int)blockIdx.x - fl.blk[r]) * (blockDim.x / kFilterSplit) + threadIdx.x / kFilterSplit;
    const bool active = t < Wo * Ho;
    const int tt = active ? t : 0;
    const int x = tt % Wo, y = tt / Wo;
    const FilterFrame fr(x, y, Wo, Ho);
    pdl_wait_then_release();
    // colour and weights accumulated apart (the pyramid's split storage);
    // every channel goes through the same multiply-adds as in the record layout
    constexpr int KW4 = C4 - 1;
    float4 accr = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 accw[KW4];
#pragma unroll
    for (int c = 0; c < KW4; ++c) accw[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = g; k < nv; k += kFilterSplit) {
        const float4 smp = tab[k];
        const float dx = smp.x * fr.e1x + smp.y * fr.e2x + smp.z * fr.rx;
        const float dy = smp.x * fr.e1y + smp.z * fr.ry;
        const float dz = smp.x * fr.e1z + smp.y * fr.e2z + smp.z * fr.rz;
        filter_sample<C4>(pyr, rgb4, w4, W, H, M, dx, dy, dz, smp.w,
                          [&](int, float wl, const float4 &v, const float4(&u)[KW4]) {
                              accr = fma4(wl, v, accr);
#pragma unroll
                              for (int c = 0; c < KW4; ++c) accw[c] = fma4(wl, u[c], accw[c]);
                          });
    }
    // sum the partial means of the kFilterSplit adjacent lanes of a texel
#pragma unroll
    for (int o = 1; o < kFilterSplit; o <<= 1) {
        accr.x += __shfl_xor_sync(0xffffffffu, accr.x, o);
        accr.y += __shfl_xor_sync(0xffffffffu, accr.y, o);
        accr.z += __shfl_xor_sync(0xffffffffu, accr.z, o);
#pragma unroll
        for (int c = 0; c < KW4; ++c) {
            accw[c].x += __shfl_xor_sync(0xffffffffu, accw[c].x, o);
            accw[c].y += __shfl_xor_sync(0xffffffffu, accw[c].y, o);
            accw[c].z += __shfl_xor_sync(0xffffffffu, accw[c].z, o);
            accw[c].w += __shfl_xor_sync(0xffffffffu, accw[c].w, o);
        }
    }
    if (!active || g != 0) return;
    store_filtered<C4>(accr, accw, nv, (size_t)fl.off[r] + t, out, outw, wfmt, rec4, K);
}

// The same filtered maps where they are too few for k_filter to fill the chip
// (latency-bound: a thread there takes 32 of 64 samples one after the other).  A
// thread takes one sample of one texel, kFilterSamples samples of a texel at a
// time; their values go to shared memory, and a thread for each channel and
// parity of the sample adds them up in the order k_filter does, so the sums are
// the same.  Twice the instructions a sample, so up to 64 texels an SM only (map
// update and a 16 x 16 frame, us, k_filter / this; 400 texels, K = 4, 8, 16: 39 /
// 27, 52 / 32, 90 / 43; 7456, K = 4, 8: 65 / 55, 91 / 71; 19808: 59 / 77, 79 / 95).
constexpr int kFilterSmall = 64;
constexpr int kFilterTexels = 4, kFilterSamples = 64;  // per block: 256 threads

template <int C4>
__global__ void __launch_bounds__(kFilterTexels * kFilterSamples) k_filter_small(
    const float4 *__restrict__ pyr, const size_t *__restrict__ rgb4, const size_t *__restrict__ w4, int W, int H, int M,
    const float4 *__restrict__ table, const int *__restrict__ nvalid, int S, const FilterLevels fl,
    float4 *__restrict__ out, float4 *__restrict__ outw, int wfmt, int rec4, int K) {
    constexpr int KW4 = C4 - 1, Cpad = 4 * C4;
    constexpr int kStride = 2 * C4 + 1;  // float4 per sample: both levels, odd (no bank conflicts)
    extern __shared__ float4 vals[];     // [texel][sample][kStride]
    __shared__ float wts[kFilterSamples][2];
    __shared__ float sums[kFilterTexels][2][Cpad];
    int r = 0;
    while (r + 1 < fl.nlev && (int)blockIdx.x >= fl.blk[r + 1]) ++r;
    const int Wo = fl.width[r], Ho = Wo / 2;
    const int nv = nvalid[r];
    const int t0 = ((int)blockIdx.x - fl.blk[r]) * kFilterTexels;
    const int tx = threadIdx.x / kFilterSamples, kk = threadIdx.x % kFilterSamples;
    const int t = min(t0 + tx, Wo * Ho - 1);
    const FilterFrame fr(t % Wo, t / Wo, Wo, Ho);
    // the adder of channel ch, parity g, texel at
    const int ch = threadIdx.x % Cpad, g = threadIdx.x / Cpad % 2, at = threadIdx.x / (2 * Cpad);
    pdl_wait_then_release();
    float acc = 0.f;
    for (int k0 = 0; k0 < nv; k0 += kFilterSamples) {
        const int k = k0 + kk;
        if (k < nv) {
            const float4 smp = __ldg(table + (size_t)r * S + k);
            const float dx = smp.x * fr.e1x + smp.y * fr.e2x + smp.z * fr.rx;
            const float dy = smp.x * fr.e1y + smp.z * fr.ry;
            const float dz = smp.x * fr.e1z + smp.y * fr.e2z + smp.z * fr.rz;
            float4 *o = vals + threadIdx.x * kStride;
            if (tx == 0) wts[kk][1] = 0.f;
            filter_sample<C4>(pyr, rgb4, w4, W, H, M, dx, dy, dz, smp.w,
                              [&](int lv, float wl, const float4 &v, const float4(&u)[KW4]) {
                                  if (tx == 0) wts[kk][lv] = wl;
                                  o[lv * C4] = v;
#pragma unroll
                                  for (int c = 0; c < KW4; ++c) o[lv * C4 + 1 + c] = u[c];
                              });
        }
        __syncthreads();
        if (at < kFilterTexels) {
            const float *v = reinterpret_cast<const float *>(vals + at * kFilterSamples * kStride) + ch;
            const int n = min(kFilterSamples, nv - k0);
#pragma unroll 4
            for (int i = g; i < n; i += kFilterSplit) {  // (k0 is even)
                acc = fmaf(wts[i][0], v[i * 4 * kStride], acc);
                if (wts[i][1] != 0.f) acc = fmaf(wts[i][1], v[i * 4 * kStride + Cpad], acc);
            }
        }
        __syncthreads();
    }
    if (at < kFilterTexels) sums[at][g][ch] = acc;
    __syncthreads();
    if (threadIdx.x < kFilterTexels && t0 + (int)threadIdx.x < Wo * Ho) {
        const float *s0 = sums[threadIdx.x][0], *s1 = sums[threadIdx.x][1];
        float4 a[C4];
#pragma unroll
        for (int c = 0; c < C4; ++c)
            a[c] = make_float4(s0[4 * c] + s1[4 * c], s0[4 * c + 1] + s1[4 * c + 1], s0[4 * c + 2] + s1[4 * c + 2],
                               s0[4 * c + 3] + s1[4 * c + 3]);
        store_filtered<C4>(a[0], a + 1, nv, (size_t)fl.off[r] + t0 + threadIdx.x, out, outw, wfmt, rec4, K);
    }
}
static_assert(kFilterSplit == 2 && kFilterTexels * 2 * 20 <= kFilterTexels * kFilterSamples, "an adder a channel and parity");

}  // namespace

template <int C4>
cudaError_t launch_pyramid(bool first, unsigned blocks, cudaStream_t s, const void *texels, const glint_env_desc &d,
                           float scale, glint_env *env, int m, int Ws, int Hs, int T, int nlev, int tail_to, bool wide) {
    const size_t smem = pyramid_smem<C4>();
    auto *pyr = reinterpret_cast<float4 *>(env->pyr);
    const float *levels = env->levels;
    const size_t *rgb4 = env->pyr_rgb4_dev, *w4 = env->pyr_w4_dev;
    auto kernel = first ? k_pyramid<true, C4> : k_pyramid<false, C4>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_pdl(true, kernel, blocks, kNT, smem, s, first ? texels : nullptr, d.format, scale, d.K, levels, pyr,
                      rgb4, w4, m, Ws, Hs, T, nlev, d.weight_space, tail_to, env->done + 1, wide);
}

template <int C4>
cudaError_t launch_filter(glint_env *env, const FilterLevels &fl, int blk, bool small, cudaStream_t s) {
    const glint_env_desc &d = env->d;
    const float4 *pyr4 = reinterpret_cast<const float4 *>(env->pyr), *table = env->table;
    float4 *out4 = reinterpret_cast<float4 *>(env->filt);
    const size_t *rgb4 = env->pyr_rgb4_dev, *w4 = env->pyr_w4_dev;
    const int *nvalid = env->nvalid;
    auto kernel = small ? k_filter_small<C4> : k_filter<C4>;
    const unsigned threads = small ? kFilterTexels * kFilterSamples : 128;
    const size_t smem = sizeof(float4) * (small ? (size_t)kFilterTexels * kFilterSamples * (2 * C4 + 1) : (size_t)d.samples);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    // Not early for k_filter: it is one wave of blocks bound by the L1s, and blocks
    // placed while the pyramid still runs crowd the SMs that are free first (1024 x
    // 512 map: K = 8 the update 30 us longer, K = 16 240 us).
    return launch_pdl(small, kernel, blk, threads, smem, s, pyr4, rgb4, w4, d.width, d.height, env->M, table, nvalid,
                      d.samples, fl, out4, env->filtw, d.weight_format, env->frec4, d.K);
}

// Pyramid level offsets (float4 units) are in a small device array that
// glint_env_create fills.
cudaError_t glint_launch_env(glint_env *env, const void *texels, cudaStream_t s, int *launches) {
    const glint_env_desc &d = env->d;
    const long n = (long)d.width * d.height;
    const float scale = ldexpf(1.f, d.scale_log2);
    const int C4 = env->Cpad / 4;
    int nl = 0;
    const bool wide = ((uintptr_t)texels & 15u) == 0;
    const long per_block = 2L * kNT * kMinMaxPairs;
    const int nblk = wide ? (int)std::min<long>(env->nblk_minmax, (n + per_block - 1) / per_block) : env->nblk_minmax;
    k_minmax<<<nblk, kNT, 0, s>>>(texels, d.format, n, scale, env->partial, env->done, d.K, d.ell, env->levels, wide);
    ++nl;
    {
        // level 0 and the next log2 T levels from the texels (T = 32), then
        // tiles of 32 while the base is large, and the last levels by the last
        // block of the launch that writes their base (1024 x 512 map: one
        // launch, levels 0-5 by tiles and 6-9 by the last block; 16 x 16
        // tiles left a 64 x 32 base whose five serial levels cost more)
        int m = 0, Ws = d.width, Hs = d.height;
        bool first = true;
        while (first || m < env->M - 1) {
            const int T = Hs < 32 ? Hs : 32;
            int nlev = 0;
            while ((1 << nlev) < T) ++nlev;
            const bool tail = m + nlev < env->M - 1 && (long)(Ws >> nlev) * (Hs >> nlev) <= kPyrTailTexels;
            const int tail_to = tail ? env->M - 1 : -1;
            const unsigned blocks = (unsigned)((Ws / T) * (Hs / T));
            cudaError_t e = cudaSuccess;
            switch (C4) {
            case 2: e = launch_pyramid<2>(first, blocks, s, texels, d, scale, env, m, Ws, Hs, T, nlev, tail_to, wide); break;
            case 3: e = launch_pyramid<3>(first, blocks, s, texels, d, scale, env, m, Ws, Hs, T, nlev, tail_to, wide); break;
            case 5: e = launch_pyramid<5>(first, blocks, s, texels, d, scale, env, m, Ws, Hs, T, nlev, tail_to, wide); break;
            default: return cudaErrorInvalidValue;
            }
            if (e != cudaSuccess) return e;
            ++nl;
            first = false;
            m += nlev;
            Ws >>= nlev;
            Hs >>= nlev;
            if (tail || nlev == 0) break;
        }
    }
    {
        FilterLevels fl{};
        fl.nlev = d.levels;
        // below kFilterSmall texels an SM the samples of a texel run side by side
        const bool small = env->foff[d.levels] < (long long)kFilterSmall * env->ctx->num_sms;
        const int per_block = small ? kFilterTexels : 128 / kFilterSplit;
        int blk = 0;
        for (int r = 0; r < d.levels; ++r) {
            fl.width[r] = env->fw[r];
            fl.off[r] = env->foff[r];
            fl.blk[r] = blk;
            blk += (int)((env->fw[r] * (env->fw[r] / 2) + per_block - 1) / per_block);
        }
        fl.blk[d.levels] = blk;
        cudaError_t e = cudaSuccess;
        switch (C4) {
        case 2: e = launch_filter<2>(env, fl, blk, small, s); break;
        case 3: e = launch_filter<3>(env, fl, blk, small, s); break;
        case 5: e = launch_filter<5>(env, fl, blk, small, s); break;
        default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
        ++nl;
    }
    if (launches) *launches = nl;
    return cudaGetLastError();
}

// The filter sample table depends only on the description (levels, samples,
// roughness range, map size); glint_env_create builds it once.
cudaError_t glint_launch_filter_table(glint_env *env, cudaStream_t s) {
    const glint_env_desc &d = env->d;
    dim3 grid((d.samples + 127) / 128, d.levels);
    k_filter_table<<<grid, 128, 0, s>>>(d.levels, d.samples, d.s_min, d.s_max, d.width, d.height, env->M, env->table,
                                        env->nvalid);
    return cudaGetLastError();
}
