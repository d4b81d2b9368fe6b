// denoise.cu -- the edge-avoiding a-trous wavelet denoiser between the rendered image and the
// loss (Appendix A, "Denoiser"), its adjoint, and the G-buffer it stops at.
//
// Level i smooths c_i into c_{i+1}(p) = sum_q h(q - p) w(p, q) c_i(q) / k(p) over the 5 x 5
// B3-spline taps (1, 4, 6, 4, 1) / 16 placed 2^i pixels apart, with
// w(p, q) = exp(-|c_i(p) - c_i(q)|^2 / sigma_rt_i^2 - |n_p - n_q|^2 / sigma_n^2 - |x_p - x_q|^2 / sigma_x^2),
// sigma_rt_i = sigma_rt / 2^i and k(p) = sum_q h w; taps outside the image are left out. The
// adjoint holds the weights fixed: since h w(p, q) is symmetric in p and q, the transpose of a
// level is the same stencil applied to g / k. Every launch covers a stack of images of one size.
#include <algorithm>

#include "render.h"

namespace {

__constant__ float kB3[5] = {1.0f / 16.0f, 4.0f / 16.0f, 6.0f / 16.0f, 4.0f / 16.0f, 1.0f / 16.0f};
constexpr float kLog2e = 1.44269504088896341f;

__device__ __forceinline__ float exp2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The level kernels read the colour as one float4 a pixel and the G-buffer as one 32-byte record
// (normal.xyz, position.x) (position.yz, -, -): one 16-byte and one 32-byte load per tap (two of 16
// bytes where the record is not 32-byte aligned: ALIGNED = false).
struct Guide {
    float nx, ny, nz, x, y, z;
};
template <bool ALIGNED>
__device__ __forceinline__ Guide guide_at(const float4* __restrict__ g, uint32_t p)
{
    float4 a, b;
    if (ALIGNED) {
        asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
            : "l"(g + 2 * (size_t)p));
    } else {
        a = __ldg(g + 2 * (size_t)p);
        b = __ldg(g + 2 * (size_t)p + 1);
    }
    return Guide{a.x, a.y, a.z, a.w, b.x, b.y};
}

__global__ void __launch_bounds__(256) k_eawt_pack(const float* __restrict__ image, const float* __restrict__ normal,
                                                   const float* __restrict__ position, float4* __restrict__ c,
                                                   float4* __restrict__ g, int64_t npx)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npx; p += (int64_t)gridDim.x * blockDim.x) {
        const float *i = image + 3 * p, *n = normal + 3 * p, *x = position + 3 * p;
        c[p] = make_float4(__ldg(i), __ldg(i + 1), __ldg(i + 2), 0.0f);
        g[2 * p] = make_float4(__ldg(n), __ldg(n + 1), __ldg(n + 2), __ldg(x));
        g[2 * p + 1] = make_float4(__ldg(x + 1), __ldg(x + 2), 0.0f, 0.0f);
    }
}

// the adjoint's input at the last level: d_out with 1 / k beside it
__global__ void __launch_bounds__(256) k_eawt_pack_adjoint(const float* __restrict__ d, const float* __restrict__ ik,
                                                           float4* __restrict__ out, int64_t npx)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npx; p += (int64_t)gridDim.x * blockDim.x) {
        out[p] = make_float4(__ldg(d + 3 * p), __ldg(d + 3 * p + 1), __ldg(d + 3 * p + 2), __ldg(ik + p));
    }
}

__device__ __forceinline__ void store3(float* o3, uint32_t p, float x, float y, float z)
{
    o3[3 * (size_t)p] = x;
    o3[3 * (size_t)p + 1] = y;
    o3[3 * (size_t)p + 2] = z;
}

// One level over a stack of N images of W x H. A thread takes a strip of two output pixels of one
// column `step` rows apart: their 5 x 5 footprints overlap in four of six rows, so the strip reads
// its 6 x 5 taps once each -- 15 tap reads per output instead of 25. A block is 32 columns by 8
// strips (narrower for narrow images, see launch_level), and strips of one residue of the rows mod `step` follow each other, so that neighbouring
// warps share tap rows in L1; block and grid are two- and three-dimensional, as the 64-bit
// divisions of a flat index cost a twelfth of the instructions. The kernel is bound by issue slots
// (about 29 instructions a tap and output: nine differences, the squared distances, one
// exponential, the sums) and its code size: the four rows that both outputs use are a loop, not
// unrolled, as the flat 6 x 5 x 2 body overran the instruction cache (20% of the stalls).
// Calls on 8 images of 800 x 800, three levels, forward / adjoint: 939 / 1125 us with flat strips of two
// (unrolled, three 16-byte loads a tap and 1 / k read per tap), now 687 / 727.
// ADJOINT: gout(q) = sum over taps of h w(q, q + tap) gin(q + tap) / k(q + tap), the weights recomputed
// from the level's recorded input c, 1 / k in gin's fourth word; the output carries the next level's
// (ikio). Forward: cout = sum h w c / k, and 1 / k to ikio.
// Rounding: h multiplies the exponential (as a logarithm in its exponent it would cost the small
// exponents of neighbouring taps three bits: 1.9e-7 instead of 2.6e-8 of a weight, RMS, for differences
// up to 1e-2), the exponent is scaled once, as a sum (scales rounded into its three terms shift every
// tap of an image alike), and 1 / k multiplies the tap's weight (a product per pixel is one more
// rounding of all its taps). Error of d_image against 64 bits on ramps with 1e-2 steps, one level of
// random gradients: 1.91e-7 without the first, 1.22e-7 with all three.
#ifndef MR_EAWT_MINB
#define MR_EAWT_MINB 4  // resident 256-thread blocks per SM the register cap aims at
#endif
constexpr int EAWT_THREADS = 256;

// TILE: blocks of 32 columns by 8 strips (the sizes as constants: 1.5% faster); else as launched
template <bool ADJOINT, bool ALIGNED, bool TILE>
__global__ void __launch_bounds__(EAWT_THREADS, MR_EAWT_MINB)
    k_eawt_level(const float4* __restrict__ c, const float4* __restrict__ gbuf, const float4* __restrict__ gin, int N,
                 int W, int H, int lstep, float inv_rt2, float inv_n2, float inv_x2, float4* __restrict__ out,
                 float* __restrict__ out3, float* __restrict__ ikio)
{
    const int step = 1 << lstep;
    const uint32_t npx = (uint32_t)W * (uint32_t)H;
    const int n_strips = ((H + 2 * step - 1) / (2 * step)) * step;
    const int X = TILE ? 32 : blockDim.x, Y = TILE ? 8 : blockDim.y, Z = TILE ? 1 : blockDim.z;
    const int x = blockIdx.x * X + threadIdx.x;
    if (x >= W) return;
    for (int img = blockIdx.z * Z + (TILE ? 0 : threadIdx.z); img < N; img += gridDim.z * Z)
        for (int sr = blockIdx.y * Y + threadIdx.y; sr < n_strips; sr += gridDim.y * Y) {
            const int y0 = ((sr >> lstep) << (lstep + 1)) + (sr & (step - 1)), y1 = y0 + step;
            if (y0 >= H) continue;
            const uint32_t base = (uint32_t)img * npx;
            const uint32_t p0 = base + (uint32_t)y0 * (uint32_t)W + (uint32_t)x;
            const uint32_t p1 = y1 < H ? p0 + (uint32_t)step * (uint32_t)W : p0;
            const float4 c0 = __ldg(c + p0), c1 = __ldg(c + p1);
            const Guide g0 = guide_at<ALIGNED>(gbuf, p0), g1 = guide_at<ALIGNED>(gbuf, p1);
            float3 a0 = f3(0.f, 0.f, 0.f), a1 = a0;
            float k0 = 0.0f, k1 = 0.0f;
            auto weight = [&](const float4& cp, const Guide& gp, const float4& cq, const Guide& gq, float h) {
                const float dx = cp.x - cq.x, dy = cp.y - cq.y, dz = cp.z - cq.z;
                const float nx = gp.nx - gq.nx, ny = gp.ny - gq.ny, nz = gp.nz - gq.nz;
                const float px = gp.x - gq.x, py = gp.y - gq.y, pz = gp.z - gq.z;
                const float dc = dx * dx + dy * dy + dz * dz, dn = nx * nx + ny * ny + nz * nz,
                            dp = px * px + py * py + pz * pz;
                return h * exp2_approx(-kLog2e * fmaf(dp, inv_x2, fmaf(dn, inv_n2, dc * inv_rt2)));
            };
            // the five taps of one row; h0, h1: the row's B3 weight for either output (the products are exact)
            auto row = [&](int qy, bool use0, bool use1, float h0, float h1) {
                if (qy < 0 || qy >= H) return;
#pragma unroll
                for (int b = 0; b < 5; ++b) {
                    const int qx = x + (b - 2) * step;
                    if (qx < 0 || qx >= W) continue;
                    const uint32_t q = base + (uint32_t)qy * (uint32_t)W + (uint32_t)qx;
                    const float4 cq = __ldg(c + q);
                    const Guide gq = guide_at<ALIGNED>(gbuf, q);
                    const float4 v = ADJOINT ? __ldg(gin + q) : cq;
                    if (use0) {
                        const float w = weight(c0, g0, cq, gq, h0 * kB3[b]) * (ADJOINT ? v.w : 1.0f);
                        a0.x += w * v.x;
                        a0.y += w * v.y;
                        a0.z += w * v.z;
                        if (!ADJOINT) k0 += w;
                    }
                    if (use1) {
                        const float w = weight(c1, g1, cq, gq, h1 * kB3[b]) * (ADJOINT ? v.w : 1.0f);
                        a1.x += w * v.x;
                        a1.y += w * v.y;
                        a1.z += w * v.z;
                        if (!ADJOINT) k1 += w;
                    }
                }
            };
            row(y0 - 2 * step, true, false, kB3[0], 0.0f);
#pragma unroll 1
            for (int m = 1; m < 5; ++m) row(y0 + (m - 2) * step, true, true, kB3[m], kB3[m - 1]);
            if (y1 < H) row(y1 + 2 * step, false, true, 0.0f, kB3[4]);
            auto emit = [&](uint32_t p, const float3& a, float k) {
                if (ADJOINT) {
                    if (out3) store3(out3, p, a.x, a.y, a.z);
                    else out[p] = make_float4(a.x, a.y, a.z, __ldg(ikio + p));
                    return;
                }
                const float f = 1.0f / k;  // k >= (6/16)^2: the centre tap has weight 1
                ikio[p] = f;
                if (out3) store3(out3, p, a.x * f, a.y * f, a.z * f);
                else out[p] = make_float4(a.x * f, a.y * f, a.z * f, 0.0f);
            };
            emit(p0, a0, k0);
            if (y1 < H) emit(p1, a1, k1);
        }
}

// G-buffer: the primary hit through each pixel centre, face normal turned towards the camera
// and hit position; 0 for both where the ray escapes
__global__ void __launch_bounds__(256) k_gbuffer(SceneDev s, ViewDev v, float* __restrict__ nrm, float* __restrict__ pos)
{
    extern __shared__ __align__(16) uint32_t sstk[];
    const int64_t npx = (int64_t)v.width * v.height;
    const float3 o = f3(v.c2w[3], v.c2w[7], v.c2w[11]);
    const float tmin = *s.tmin_dev;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npx; p += (int64_t)gridDim.x * blockDim.x) {
        const int px = (int)(p % v.width), py = (int)(p / v.width);
        const float3 d = camera_dir(v, px, py, 0.5f, 0.5f);
        Hit h;
        trace<false>(s, o, d, -1, tmin, __int_as_float(0x7f800000), h, sstk + threadIdx.x);
        float3 n = f3(0.f, 0.f, 0.f), x = n;
        if (h.tri >= 0) {
            float3 v0, e1, e2;
            int tchk;
            load_tri(s, __ldg(s.leaf_of + h.tri), v0, e1, e2, tchk);
            n = normalize(cross(e1, e2));
            if (dot(n, d) > 0.0f) n = f3(-n.x, -n.y, -n.z);
            x = f3(o.x + h.t * d.x, o.y + h.t * d.y, o.z + h.t * d.z);
        }
        nrm[3 * p] = n.x;
        nrm[3 * p + 1] = n.y;
        nrm[3 * p + 2] = n.z;
        pos[3 * p] = x.x;
        pos[3 * p + 1] = x.y;
        pos[3 * p + 2] = x.z;
    }
}

unsigned grid_for_pixels(int64_t n, int sms)
{
    const int64_t g = (n + 255) / 256;
    const int64_t cap = (int64_t)sms * 8;
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

void mr_launch_eawt_pack(const float* image, const float* normal, const float* position, float4* c, float4* g,
                         int64_t npx, int sms, cudaStream_t st)
{
    k_eawt_pack<<<grid_for_pixels(npx, sms), 256, 0, st>>>(image, normal, position, c, g, npx);
}

void mr_launch_eawt_pack_adjoint(const float* d, const float* ik, float4* out, int64_t npx, int sms, cudaStream_t st)
{
    k_eawt_pack_adjoint<<<grid_for_pixels(npx, sms), 256, 0, st>>>(d, ik, out, npx);
}

template <bool ADJOINT>
static void launch_level(const float4* c, const float4* g, const float4* gin, int N, int W, int H, int lstep,
                         float inv_rt2, float inv_n2, float inv_x2, float4* out, float* out3, float* ikio,
                         cudaStream_t st)
{
    const int64_t step = (int64_t)1 << lstep, strips = (H + 2 * step - 1) / (2 * step) * step;
    // Columns, strips and images of a block: the widest of 32, 16 and 8 columns unless a narrower one leaves a
    // tenth fewer threads beside the image, for images below 8 columns what holds them; as many strips as there
    // are, then images (block.z is at most 64). 32 x 8 x 1 alone left threads idle on small and narrow images:
    // 2048 images of 8 x 8, two levels, 60 us, now 37; 16 of 720 x 40 119 and 103; 64 of 256 x 1 46 and 33.
    int X = W < 8 ? 1 : 32, Y = 1, Z = 1;
    const auto padded = [W](int x) { return (W + x - 1) / x * x; };
    while (X < 8 && X < W) X *= 2;
    for (int x = 16; x >= 8 && W >= 8; x /= 2)
        if (10 * padded(x) <= 9 * padded(X)) X = x;
    while (X * Y < EAWT_THREADS && Y < strips) Y *= 2;
    while (X * Y * Z < EAWT_THREADS && Z < std::min(N, 64)) Z *= 2;
    const bool tile = X == 32 && Y == 8;
    const dim3 block((unsigned)X, (unsigned)Y, (unsigned)Z);
    const dim3 grid((unsigned)((W + X - 1) / X), (unsigned)std::min<int64_t>((strips + Y - 1) / Y, 65535),
                    (unsigned)std::min((N + Z - 1) / Z, 65535));
    const bool aligned = (reinterpret_cast<uintptr_t>(g) & 31) == 0;
    const auto k = tile ? (aligned ? k_eawt_level<ADJOINT, true, true> : k_eawt_level<ADJOINT, false, true>)
                        : (aligned ? k_eawt_level<ADJOINT, true, false> : k_eawt_level<ADJOINT, false, false>);
    k<<<grid, block, 0, st>>>(c, g, gin, N, W, H, lstep, inv_rt2, inv_n2, inv_x2, out, out3, ikio);
}

void mr_launch_eawt_level(const float4* c, const float4* g, int N, int W, int H, int lstep, float inv_rt2, float inv_n2,
                          float inv_x2, float4* cout, float* out3, float* ikout, cudaStream_t st)
{
    launch_level<false>(c, g, nullptr, N, W, H, lstep, inv_rt2, inv_n2, inv_x2, cout, out3, ikout, st);
}

void mr_launch_eawt_level_adjoint(const float4* gin, const float4* c, const float4* g, int N, int W, int H, int lstep,
                                  float inv_rt2, float inv_n2, float inv_x2, float4* gout, float* out3,
                                  const float* ik_next, cudaStream_t st)
{
    launch_level<true>(c, g, gin, N, W, H, lstep, inv_rt2, inv_n2, inv_x2, gout, out3, const_cast<float*>(ik_next), st);
}

void mr_launch_gbuffer(const SceneDev& s, const ViewDev& v, float* nrm, float* pos, int sms, cudaStream_t st)
{
    k_gbuffer<<<grid_for_pixels((int64_t)v.width * v.height, sms), 256, sizeof(uint32_t) * MR_SSTACK * 256, st>>>(
        s, v, nrm, pos);
}
