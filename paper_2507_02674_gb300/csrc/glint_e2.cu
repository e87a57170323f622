// E2 reflection probabilities p_k alone (Eq. probhk by quadrature; the points,
// weights and pyramid level of e2_probabilities in glint_probs.cuh), 32 or 8 lanes
// a pixel.  The surrogate's labels, and the reference its error is judged by.
//
// What bounds it: the L1's look-ups of lines and banks.  A point reads 2 x 2
// texels of 32 bytes (K = 8) at a direction of its own; one thread a pixel makes
// 32 unrelated look-ups a request where neighbouring pixels differ (their
// roughness, their normal).  Here the lanes take points of one pixel, in a row
// along the lobe's radius (the closest on the map) in each request, and four
// adjacent lanes share their four points: in each of four requests a quad reads
// the 2 x 2 texels of one point, which the swapped columns of the pyramid's odd
// rows (pyr_column) put in four different banks.  The lanes exchange two words a
// point for it (texel and weight) and each accumulates what it reads; the sums
// meet at the end of the pixel.
//
// 32 lanes a pixel serve many points (a request takes eight in a row), and frames
// too small to fill the chip otherwise.  8 lanes a pixel, four neighbouring
// pixels at a time, waste fewer lanes at the end of few points, share the set-up
// and the final sums, and read the same lines where neighbouring pixels look the
// same way, as a thread a pixel does.  1280 x 720, us, thread / 8 lanes / 32 lanes;
// "rough": random roughness a pixel, "smooth": one sphere, one roughness:
//   K = 4,  S = 16 rough 1599 / 1383 / 1466, smooth 1124 / 1071 / 1151
//   K = 8,  S = 13 rough 1476 / 1145 / 1397, smooth 828 / 862 / 1021
//           S = 16 rough 2263 / 1597 / 1710, smooth 1267 / 1212 / 1446
//           S = 32 rough 9080 / 6050 / 5802, smooth 5106 / 4617 / 4706
//   K = 16, S = 8  rough 1303 / 820 / 1090, smooth 467 / 568 / 743
//           S = 16 rough 5305 / 2967 / 3225, smooth 1858 / 1950 / 2622
// (K = 8, S = 32, 32 lanes: two lanes a point took 7.3 ms; a request over every
// fourth ring instead of eight in a row 6.6; words exchanged through shared
// memory 7.4; blocks of 12 or 24 warps in step 6.3 and 6.5; without the branch over
// invalid points 6.9.  The sums of 8 lanes in the order of 32, so that both give the
// same bits: K = 8, S = 13, smooth 985 us.)
#include "glint_internal.cuh"
#include "glint_probs.cuh"

using namespace glint;

namespace {

constexpr int kWarps = 4;       // warps a block
constexpr int kMaxSteps = 8;    // pixels a group of lanes takes one after the other at most
constexpr int kMaxS = 256;

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// atan2(z, x) / 2 pi in [-1/2, 1/2]: atan(q) / 2 pi = q A(q^2) on q = min / max
// in [0, 1], A of degree 7 by iteratively reweighted least squares towards the
// minimax of the error (6e-9; 2.6e-8 as evaluated in FP32), then the octants.
__device__ __forceinline__ float turns(float z, float x) {
    const float az = fabsf(z), ax = fabsf(x);
    const float q = fminf(az, ax) * rcp_approx(fmaxf(fmaxf(az, ax), 1e-30f));
    const float u = q * q;
    float t = -0x1.527ee2p-11f;
    t = fmaf(t, u, 0x1.c83e62p-9f);
    t = fmaf(t, u, -0x1.23a898p-7f);
    t = fmaf(t, u, 0x1.f6e968p-7f);
    t = fmaf(t, u, -0x1.6ab140p-6f);
    t = fmaf(t, u, 0x1.04106cp-5f);
    t = fmaf(t, u, -0x1.b28dd2p-5f);
    t = fmaf(t, u, 0x1.45f2f8p-3f);
    t *= q;
    t = (az > ax) ? 0.25f - t : t;
    t = (x < 0.f) ? 0.5f - t : t;
    return copysignf(t, z);
}

// acos(y) / pi: sqrt(1 - |y|) B(|y|) (the form of Abramowitz & Stegun 4.4.46),
// B of degree 7 fitted likewise (4e-9; 5.8e-8 as evaluated in FP32).
__device__ __forceinline__ float half_turns(float y) {
    const float v = fminf(fabsf(y), 1.f);
    float t = -0x1.e11edep-12f;
    t = fmaf(t, v, 0x1.2e49fap-9f);
    t = fmaf(t, v, -0x1.7381f0p-8f);
    t = fmaf(t, v, 0x1.46d724p-7f);
    t = fmaf(t, v, -0x1.066400p-6f);
    t = fmaf(t, v, 0x1.d025e2p-6f);
    t = fmaf(t, v, -0x1.17cb76p-4f);
    t = fmaf(t, v, 0.5f);
    t *= sqrt_approx(1.f - v);
    return (y < 0.f) ? 1.f - t : t;
}

// A pixel's geometry, staged by one lane and read by the whole warp.
struct __align__(16) E2Pixel {
    float ax, ay, mu, ot;
    float nx, ny, nz, ob;
    float tx, ty, tz, wx;
    float bx, by, bz, wy;
    float wz;
    int level;   // pyramid level, -1: background
    int pad[2];
};

// Sums of v[0 .. K) over groups of G lanes: with K <= G, lane L of a group ends with
// the sum of v[L >> (log2 G - log2 K)] in v[0], else with those of v[L K / G ..] in
// v[0 .. K / G).
template <int K, int G>
__device__ __forceinline__ void group_sums(float (&v)[K]) {
    const int lane = threadIdx.x & 31;
    int n = K;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        if (n > 1) {
            n /= 2;
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < K / 2; ++i)
                if (i < n) {
                    const float give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
}

// acc += w (texel idx), the weights of the texel's components.  With 64-byte
// texels (K = 16) the lanes of the lower row read the second half first, again
// four banks a quad: acc[k] then holds component k ^ 8 (low: the lane's row bit).
template <int K, int KW4>
__device__ __forceinline__ void add_texel(const float4 *__restrict__ lev, unsigned idx, float w, int low,
                                          float (&acc)[K]) {
    if (w > 0.f) {  // an invalid point weighs nothing: 12% of the points, and their lines, are not read
        float4 t[KW4];
        if constexpr (KW4 == 1) {
            t[0] = __ldg(lev + idx);
        } else {
            const float4 *p = lev + (size_t)idx * KW4;
#pragma unroll
            for (int c = 0; c < KW4; c += 2)  // 32-byte aligned (even level offsets)
                ldg8(KW4 == 4 ? p + (c ^ (low << 1)) : p + c, t[c], t[c + 1]);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float4 v = t[k / 4];
            acc[k] = fmaf(w, (k % 4 == 0) ? v.x : (k % 4 == 1) ? v.y : (k % 4 == 2) ? v.z : v.w, acc[k]);
        }
    }
}

// G lanes (32 or 8) a pixel, so 32 / G pixels a warp at a time.  FIXED: S is a power
// of two from 8, so that a lane keeps its ring(s) of points.  Five blocks an SM;
// six (80 registers) where it is faster (8 lanes, rough, K = 8: S = 16 1705 -> 1597 us,
// but S = 24 3515 -> 3596; K = 16: S = 16 3116 -> 2967, S = 24 7020 -> 6687).
template <int K, bool FIXED, int G>
__global__ void __launch_bounds__(kWarps * 32, G == 8 && (FIXED || K == 16) ? 6 : 5) k_e2_probs(ShadeArgs a,
                                                                                                int steps) {
    constexpr int KW4 = (3 + K + 3) / 4 - 1, kGroups = 32 / G, kMaxPpw = kGroups * kMaxSteps;
    static_assert(kMaxPpw <= 32, "a warp's pixels are staged by a lane each");
    __shared__ float2 ring[kMaxS];   // r, 2 s
    __shared__ float2 angle[kMaxS];  // cos, sin
    __shared__ E2Pixel px[kWarps][kMaxPpw];
    const int S = a.e2S, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ppw = kGroups * steps, group = lane / G;
    // the lane's place in a step's G points: a request takes G / 4 in a row (one of each quad)
    const int lp = ((lane % G) >> 2) + (G / 4) * (lane & 3);
    const bool right = lane & 1, lower = lane & 2;  // the texel of a look-up that this lane reads
    for (int i = threadIdx.x; i < S; i += kWarps * 32) {
        const float sv = ((float)i + 0.5f) / (float)S;
        ring[i] = make_float2(sqrtf(__fsub_rn(1.f, __fmul_rn(sv, sv))) / sv, 2.f * sv);  // (not contracted, as there)
        float sp, cp;
        sincospif(2.f * ((float)i + 0.5f) / (float)S, &sp, &cp);
        angle[i] = make_float2(cp, sp);
    }
    pdl_wait();
    if (a.npix <= 128L * kFewBlocks) pdl_release();  // as the kernels of a thread a pixel do
    const long q0 = ((long)blockIdx.x * kWarps + warp) * ppw;
    if (lane < ppw) {
        E2Pixel e;
        e.level = -1;
        const long q = q0 + lane;
        if (q < a.npix) {
            const float4 g0 = ldg4(a.view_n0 + q);
            if (g0.w > 0.f) {
                const float4 g1 = ldg4(a.normal_f0 + q), g2 = ldg4(a.uv_alpha + q), tg = ldg4(a.tangent + q);
                const float tn = tg.x * g1.x + tg.y * g1.y + tg.z * g1.z;
                float tx = tg.x - tn * g1.x, ty = tg.y - tn * g1.y, tz = tg.z - tn * g1.z;
                const float tinv = 1.f / sqrtf(tx * tx + ty * ty + tz * tz);
                tx *= tinv; ty *= tinv; tz *= tinv;
                const float bx = g1.y * tz - g1.z * ty, by = g1.z * tx - g1.x * tz, bz = g1.x * ty - g1.y * tx;
                e.ax = g2.z; e.ay = g2.w;
                e.mu = g1.x * g0.x + g1.y * g0.y + g1.z * g0.z;
                e.ot = g0.x * tx + g0.y * ty + g0.z * tz;
                e.ob = g0.x * bx + g0.y * by + g0.z * bz;
                e.nx = g1.x; e.ny = g1.y; e.nz = g1.z;
                e.tx = tx; e.ty = ty; e.tz = tz;
                e.bx = bx; e.by = by; e.bz = bz;
                e.wx = g0.x; e.wy = g0.y; e.wz = g0.z;
                const float lx = fminf(g2.z, g2.w) * (4.0f / (float)S);
                e.level = 0;
                for (int k = 0; k < a.envM; ++k)
                    if ((float)(a.envH >> k) * lx >= kPi) e.level = k;
            }
        }
        px[warp][lane] = e;
    }
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < ppw; j += kGroups) {
        const long q = q0 + j + group;
        if (q0 + j >= a.npix) return;
        const E2Pixel e = px[warp][j + group];
        const bool live = e.level >= 0;  // (past the end of the frame: no)
        if (G == 32 ? !live : !__any_sync(0xffffffffu, live)) {
            if (q < a.npix)
                for (int k = lane % G; k < K; k += G) a.p_out[q * K + k] = 0.f;
            continue;
        }
        const int level = max(e.level, 0);
        const int W = a.envW >> level, H = a.envH >> level;
        const float Wf = (float)W, Hf = (float)H;
        const float4 *lev = a.pyr + a.pyr_w4[level];
        float acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = 0.f;
        float sum_all = 0.f, sum_inv = 0.f;
        auto point = [&](float axr, float ayr, float s2, float2 cs) {
            const float cp = cs.x, sp = cs.y;
            // the slope and the validity of its reflection, operation for
            // operation as e2_probabilities has them
            const float sx = axr * cp, sy = ayr * sp;
            const float hl2 = fmaf(sy, sy, fmaf(sx, sx, 1.f));
            const float oh = __fadd_rn(fmaf(-sx, e.ot, -__fmul_rn(sy, e.ob)), e.mu);
            const bool valid = fmaf(2.f, oh, -__fmul_rn(e.mu, hl2)) > 0.f;
            // 2 sqrt(s^2 + rho^2 (1 - s^2)) = 2 s |h'|
            const float wgt = s2 * sqrt_approx(hl2);
            sum_all += wgt;
            sum_inv += valid ? 0.f : wgt;
            const float w = valid && (G == 32 || live) ? wgt : 0.f;  // background beside a live pixel reads nothing
            const float c = 2.f * oh * rcp_approx(hl2);
            const float hx = e.nx - sx * e.tx - sy * e.bx;
            const float hy = e.ny - sx * e.ty - sy * e.by;
            const float hz = e.nz - sx * e.tz - sy * e.bz;
            const float dx = c * hx - e.wx, dy = c * hy - e.wy, dz = c * hz - e.wz;
            const float xx = fmaf(turns(dz, dx), Wf, -0.5f), yy = fmaf(half_turns(dy), Hf, -0.5f);
            // floors by adding 1.5 2^23 rounded down: the sum's low bits are the integer
            constexpr float kBig = 12582912.f;
            const float xb = __fadd_rd(xx, kBig), yb = __fadd_rd(yy, kBig);
            const float fx = xx - (xb - kBig), fy = yy - (yb - kBig);
            const int xi = __float_as_int(xb) & (W - 1), xn = (xi + 1) & (W - 1);
            const int y0 = __float_as_int(yb) - __float_as_int(kBig);  // in [-1, H - 1] whatever d is
            const unsigned ra = (unsigned)(max(y0, 0) * W), rn = (unsigned)(min(y0 + 1, H - 1) * W);
            const float wl = 1.f - fx, w0 = w * (1.f - fy), w1 = w * fy;
            // rows and columns: this lane's and the other ones
            const unsigned rm = lower ? rn : ra, ro = lower ? ra : rn;
            const unsigned cm = right ? xn : xi, co = right ? xi : xn;
            // pyr_column
            const unsigned sm = KW4 >= 2 && (rm & W) ? 2u : 0u, so = KW4 >= 2 && (ro & W) ? 2u : 0u;
            const float um = lower ? w1 : w0, uo = lower ? w0 : w1, vm = right ? fx : wl, vo = right ? wl : fx;
            const unsigned i0 = rm | (cm ^ sm);
            const float f0 = um * vm;
            const unsigned i1 = __shfl_xor_sync(0xffffffffu, rm | (co ^ sm), 1);
            const float f1 = __shfl_xor_sync(0xffffffffu, um * vo, 1);
            const unsigned i2 = __shfl_xor_sync(0xffffffffu, ro | (cm ^ so), 2);
            const float f2 = __shfl_xor_sync(0xffffffffu, uo * vm, 2);
            const unsigned i3 = __shfl_xor_sync(0xffffffffu, ro | (co ^ so), 3);
            const float f3 = __shfl_xor_sync(0xffffffffu, uo * vo, 3);
            // one point of the quad a request: each lane its texel of it
            const unsigned j0 = right ? i1 : i0, j1 = right ? i0 : i1, j2 = right ? i3 : i2, j3 = right ? i2 : i3;
            const float g0 = right ? f1 : f0, g1 = right ? f0 : f1, g2 = right ? f3 : f2, g3 = right ? f2 : f3;
            add_texel<K, KW4>(lev, lower ? j2 : j0, lower ? g2 : g0, lower, acc);
            add_texel<K, KW4>(lev, lower ? j3 : j1, lower ? g3 : g1, lower, acc);
            add_texel<K, KW4>(lev, lower ? j0 : j2, lower ? g0 : g2, lower, acc);
            add_texel<K, KW4>(lev, lower ? j1 : j3, lower ? g1 : g3, lower, acc);
        };
        if (FIXED) {
            const int per = max(G / S, 1);  // angles at a time
            for (int g = 0; g < S; g += G) {
                const float2 rs = ring[(lp & (S - 1)) + g];
                const float axr = e.ax * rs.x, ayr = e.ay * rs.x;
#pragma unroll 1
                for (int ic = S < G ? lp / S : 0; ic < S; ic += per) point(axr, ayr, rs.y, angle[ic]);
            }
        } else {
            int ia = lp % S, ic = lp / S;
            const int da = G % S, dc = G / S;
            for (int i = lp; i - lp < S * S; i += G) {  // the same trips for every lane
                const bool in = i < S * S;
                const float2 rs = ring[ia];
                point(e.ax * rs.x, e.ay * rs.x, in ? rs.y : 0.f, angle[in ? ic : 0]);
                ia += da;
                ic += dc;
                if (ia >= S) { ia -= S; ++ic; }
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            sum_all += __shfl_xor_sync(0xffffffffu, sum_all, o);
            sum_inv += __shfl_xor_sync(0xffffffffu, sum_inv, o);
        }
        if (K == 16 && lower) {  // acc[k] holds component k ^ 8
#pragma unroll
            for (int k = 0; k < K / 2; ++k) {
                const float t = acc[k];
                acc[k] = acc[k + K / 2];
                acc[k + K / 2] = t;
            }
        }
        group_sums<K, G>(acc);
        constexpr int kPer = G >= K ? G / K : 1;  // lanes that hold the same sum
        constexpr int kOwn = G >= K ? 1 : K / G;  // sums a lane holds
        if (q < a.npix && lane % G % kPer == 0) {
#pragma unroll
            for (int i = 0; i < kOwn; ++i) {
                const int k = lane % G / kPer * kOwn + i;
                a.p_out[q * K + k] = live ? (k == 0 ? sum_inv + acc[i] : acc[i]) / sum_all : 0.f;
            }
        }
    }
}

template <int K, int G>
cudaError_t launch(const ShadeArgs &a, int num_sms, cudaStream_t s) {
    // several pixels a group once there are warps enough without
    const long want = (long)num_sms * 24 * 4;
    constexpr int kGroups = 32 / G;
    int steps = kMaxSteps;
    while (steps > 1 && a.npix / (kGroups * steps) < want) steps >>= 1;
    const long per_block = (long)kWarps * kGroups * steps;
    const unsigned grid = (unsigned)((a.npix + per_block - 1) / per_block);
    const bool fixed = a.e2S >= 8 && (a.e2S & (a.e2S - 1)) == 0;
    auto kernel = k_e2_probs<K, true, G>;
    if constexpr (K >= 8 || G == 32) {  // (8 lanes take K <= 4 only with a power of two)
        if (!fixed) kernel = k_e2_probs<K, false, G>;
    } else if (!fixed) {
        return cudaErrorInvalidValue;
    }
    return launch_pdl(true, kernel, grid, kWarps * 32, 0, s, a, steps);
}

}  // namespace

cudaError_t glint_launch_e2_probs(const ShadeArgs &a, int K, int lanes, int num_sms, cudaStream_t s) {
    switch (K) {
    case 2: return lanes == 8 ? launch<2, 8>(a, num_sms, s) : launch<2, 32>(a, num_sms, s);
    case 4: return lanes == 8 ? launch<4, 8>(a, num_sms, s) : launch<4, 32>(a, num_sms, s);
    case 8: return lanes == 8 ? launch<8, 8>(a, num_sms, s) : launch<8, 32>(a, num_sms, s);
    case 16: return lanes == 8 ? launch<16, 8>(a, num_sms, s) : launch<16, 32>(a, num_sms, s);
    default: return cudaErrorInvalidValue;
    }
}
