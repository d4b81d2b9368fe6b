// env.cu -- environment-map importance-sampling tables (the paper's proposal
// q_dir proportional to L_env, drawn from the environment map itself, Sec. 4.1).
//
// Texel weight w = Y(L) sin(theta_row), Y = (r + g + b) / 3 (Appendix A). Per-row conditional
// CDFs and the marginal CDF over rows are FP64 prefix sums (each sum from the left, by one thread,
// so that it has a fixed order), converted to uint32 thresholds
// ceil(cdf * 2^24): for a 24-bit uniform u = k 2^-24, cdf <= u exactly when threshold <= k,
// so the search needs no FP64 arithmetic. The texel table packs (r, g, b, P * W * H).
// The draw inverts the CDF over all texels in row-major order, (rows before + texels before in
// the row) / total, as 53-bit thresholds ceil(cdf * 2^53) for a 53-bit uniform made of two
// random words, through a guide with about eight buckets per texel: one short search instead of
// a row search followed by a column search.
#include <algorithm>

#include "internal.h"

namespace {

__device__ __forceinline__ uint32_t threshold(double cdf)
{
    const double x = ceil(cdf * 16777216.0);
    return x <= 0.0 ? 0u : (x >= 16777216.0 ? 16777216u : (uint32_t)x);
}

// One block per row. The weights and the thresholds are one division each per texel, spread over
// the block; only the prefix sum is serial, as its order is part of the contract (w_0 + w_1 + ...
// from the left): one thread adds ENV_COLS weights at a time out of shared memory. The sums before
// each texel serve both CDFs. One thread per row did all of it before, its loads and divisions in
// one dependent chain: 1253 us (this kernel) + 508 us (the thresholds over all texels) + 266 us
// (the rows) at 1024 x 512, now 82 + 33 + 28 us.
constexpr int ENV_COLS = 1024;

// exclusive prefix sums of s[0 .. n) in place, in order, onto `run`; returns the sum. One thread.
__device__ __forceinline__ double serial_prefix(double* s, int n, double run)
{
    constexpr int B = 8;  // loads in flight ahead of the chain of additions
    int c = 0;
    for (; c + B <= n; c += B) {
        double v[B];
#pragma unroll
        for (int k = 0; k < B; ++k) v[k] = s[c + k];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            s[c + k] = run;
            run += v[k];
        }
    }
    for (; c < n; ++c) {
        const double v = s[c];
        s[c] = run;
        run += v;
    }
    return run;
}

__global__ void __launch_bounds__(256) k_env_rows(const float* __restrict__ env, int W, int H, double* __restrict__ w,
                                                  double* __restrict__ before, double* __restrict__ rowsum,
                                                  uint32_t* __restrict__ cond)
{
    __shared__ double s[ENV_COLS];
    __shared__ double sh[2];  // sin(theta) of the row, the row's sum so far
    const int r = blockIdx.x, tid = threadIdx.x;
    if (tid == 0) {
        sh[0] = sin(3.14159265358979323846 * ((double)r + 0.5) / (double)H);
        sh[1] = 0.0;
    }
    __syncthreads();
    const double st = sh[0];
    const size_t row = (size_t)r * W;
    for (int c0 = 0; c0 < W; c0 += ENV_COLS) {
        const int n = min(ENV_COLS, W - c0);
        for (int c = tid; c < n; c += blockDim.x) {
            const float* p = env + 3 * (row + c0 + c);
            const double y = (((double)p[0] + (double)p[1]) + (double)p[2]) / 3.0 * st;
            w[row + c0 + c] = y;
            s[c] = y;
        }
        __syncthreads();
        if (tid == 0) sh[1] = serial_prefix(s, n, sh[1]);
        __syncthreads();
        for (int c = tid; c < n; c += blockDim.x) before[row + c0 + c] = s[c];
        __syncthreads();
    }
    const double acc = sh[1];
    if (tid == 0) rowsum[r] = acc;
    uint32_t* cr = cond + (size_t)r * (W + 1);
    for (int c = tid; c <= W; c += blockDim.x) {
        double v;
        // (a thread reads back the sums it wrote itself)
        if (acc > 0.0) v = (c == W) ? 1.0 : before[row + c] / acc;
        else v = (double)c / (double)W;
        cr[c] = threshold(v);
    }
}

// one block: the sums of the rows before each row, in order, the total and the marginal CDF
__global__ void __launch_bounds__(256) k_env_marg(const double* __restrict__ rowsum, int H, double* total_out,
                                                  int32_t* ok_out, uint32_t* __restrict__ marg,
                                                  double* __restrict__ rowbase)
{
    __shared__ double s[ENV_COLS];
    __shared__ double sh;
    const int tid = threadIdx.x;
    if (tid == 0) sh = 0.0;
    for (int r0 = 0; r0 < H; r0 += ENV_COLS) {
        const int n = min(ENV_COLS, H - r0);
        for (int r = tid; r < n; r += blockDim.x) s[r] = rowsum[r0 + r];
        __syncthreads();
        if (tid == 0) sh = serial_prefix(s, n, sh);
        __syncthreads();
        for (int r = tid; r < n; r += blockDim.x) rowbase[r0 + r] = s[r];
        __syncthreads();
    }
    const double total = sh;
    const int ok = total > 0.0;
    for (int r = tid; r <= H; r += blockDim.x) {
        double v;
        if (ok) v = (r == H) ? 1.0 : rowbase[r] / total;
        else v = (double)r / (double)H;
        marg[r] = threshold(v);
    }
    if (tid == 0) {
        *total_out = total;
        *ok_out = ok;
    }
}

__device__ __forceinline__ unsigned long long threshold53(double cdf)
{
    const double x = ceil(cdf * 9007199254740992.0);
    return x <= 0.0 ? 0ull : (x >= 9007199254740992.0 ? 9007199254740992ull : (unsigned long long)x);
}

// one thread per texel: the threshold of the CDF over all texels, (rows before + texels before in
// the row) / total, and the packed texel (r, g, b, P W H). The first threads also write the angle
// tables for drawing directions inside a texel without a full-range sin/cos: the row centre
// theta_r = pi (r + 1/2) / H and the column centre psi_c = 2 pi (c + 1/2) / W - pi, plus the
// per-row RIS weight factor. With q = P W H / (2 pi^2 sin theta) and P = Y(L) sin theta_r / total,
// the candidate weight p_hat / q = Y(f_r cos) sin theta 2 pi^2 total / (W H sin theta_r): Y(L)
// cancels, so a candidate needs no texel fetch.
__global__ void __launch_bounds__(256) k_env_tables(const float* __restrict__ env, const double* __restrict__ w,
                                                    const double* __restrict__ before,
                                                    const double* __restrict__ rowbase,
                                                    const double* __restrict__ total, int W, int H,
                                                    unsigned long long* __restrict__ flat, float4* __restrict__ texel,
                                                    float4* __restrict__ row, float2* __restrict__ col)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x, n = (size_t)W * H;
    const double tot = *total;
    if (i < n) {
        const double cdf = tot > 0.0 ? (rowbase[(uint32_t)i / (uint32_t)W] + before[i]) / tot : (double)i / ((double)W * (double)H);
        flat[i] = threshold53(cdf);
        const float p = tot > 0.0 ? (float)(w[i] / tot * ((double)W * (double)H)) : 0.0f;
        texel[i] = make_float4(env[3 * i], env[3 * i + 1], env[3 * i + 2], p);
    } else if (i == n) {
        flat[i] = 9007199254740992ull;
    }
    const double pi = 3.14159265358979323846;
    if (i < (size_t)H) {
        const double th = pi * ((double)i + 0.5) / (double)H;
        const double st = sin(th);
        const double g = tot > 0.0 ? 2.0 * pi * pi * tot / ((double)W * (double)H * st) : 0.0;
        row[i] = make_float4((float)cos(th), (float)st, (float)g, 0.0f);
    }
    if (i < (size_t)W) {
        const double ps = 2.0 * pi * ((double)i + 0.5) / (double)W - pi;
        col[i] = make_float2((float)cos(ps), (float)sin(ps));
    }
}

// largest t in [lo, hi] with a[t] <= k (a[lo] <= k)
template <class T>
__device__ __forceinline__ int search_in(const T& a, int lo, int hi, unsigned long long k)
{
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a[mid] <= k) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// the same by a whole warp, 32 probes a step
__device__ __forceinline__ int search_warp(const unsigned long long* __restrict__ a, int lo, int hi, unsigned long long k)
{
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int stride = (hi - lo) / 32 + 1;
        const int64_t probe = (int64_t)lo + (int64_t)lane * stride;
        const int below = __popc(__ballot_sync(MR_FULL, lane == 0 || (probe <= hi && a[probe] <= k)));
        lo += (below - 1) * stride;
        hi = min(hi, lo + stride - 1);
    }
    return lo;
}

// Guide of the flat CDF (n entries): bucket b answers the search at k = b << shift; entry g is
// n - 1. A block takes GUIDE_TILE consecutive buckets: two searches over the whole table find the
// texels its first and last bucket fall on, the thresholds between them (about an eighth of the
// buckets) go to shared memory and every bucket searches there: ~7 steps instead of 19 through
// L2 at 1024 x 512 (54 us for the 4.2 M buckets before, now 38 with GUIDE_MORE).
constexpr int GUIDE_TILE = 2048, GUIDE_SHARED = 1024;
__global__ void __launch_bounds__(256) k_env_flat_guide(const unsigned long long* __restrict__ flat, int n, int g,
                                                        int shift, uint32_t* __restrict__ guide)
{
    __shared__ unsigned long long s[GUIDE_SHARED];
    __shared__ int sh[2];
    const int b0 = blockIdx.x * GUIDE_TILE, b1 = min(b0 + GUIDE_TILE, g + 1);  // [b0, b1)
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        const int t = search_warp(flat, 0, n - 1, (unsigned long long)(warp ? b1 - 1 : b0) << shift);
        if ((threadIdx.x & 31) == 0) sh[warp] = t;
    }
    __syncthreads();
    const int t0 = sh[0], t1 = sh[1], m = t1 - t0 + 1;
    const bool staged = m >= 1 && m <= GUIDE_SHARED;  // block-uniform
    if (staged)
        for (int t = threadIdx.x; t < m; t += blockDim.x) s[t] = flat[t0 + t];
    __syncthreads();
    for (int b = b0 + (int)threadIdx.x; b < b1; b += blockDim.x) {
        const unsigned long long k = (unsigned long long)b << shift;
        int t;
        if (b == g) t = n - 1;
        else if (staged) t = t0 + search_in(s, 0, m - 1, k);
        else t = search_in(flat, 0, n - 1, k);
        // the bucket's answer may be a later texel: the next threshold is reached before the next bucket
        const unsigned long long next = (unsigned long long)(b + 1) << shift;
        const bool more = t + 1 < n && (staged && t + 1 - t0 < m ? s[t + 1 - t0] : flat[t + 1]) <= next;
        guide[b] = (uint32_t)t | (more ? GUIDE_MORE : 0u);
    }
}

}  // namespace

// guide buckets per texel of the flat CDF: with 8 only ~12% of the draws on config 3's env land
// in a bucket that holds a CDF boundary (and so read a threshold), against ~36% with 2; the
// shade stage measured 85.3 / 82.1 / 80.0 / 81.5 / 85.8 ms per 20-view render at 2 / 4 / 8 / 16 / 32
#ifndef MR_GUIDE_PER_TEXEL
#define MR_GUIDE_PER_TEXEL 8
#endif

mirres_status mr_env_alloc(mirres_scene* s)
{
    const size_t W = (size_t)s->desc.env_w, H = (size_t)s->desc.env_h;
    {
        // about MR_GUIDE_PER_TEXEL guide buckets per texel over the 53-bit uniform
        int lg = 1;
        while (((size_t)1 << lg) < (size_t)MR_GUIDE_PER_TEXEL * W * H && lg < 30) ++lg;
        s->gf = 1 << lg;
        s->gf_shift = 53 - lg;
    }
    cudaError_t e = cudaSuccess;
    e = e ? e : cudaMalloc((void**)&s->env_w, sizeof(double) * W * H);
    e = e ? e : cudaMalloc((void**)&s->env_before, sizeof(double) * W * H);
    e = e ? e : cudaMalloc((void**)&s->env_rowsum, sizeof(double) * H);
    e = e ? e : cudaMalloc((void**)&s->env_total, sizeof(double));
    e = e ? e : cudaMalloc((void**)&s->env_ok, sizeof(int32_t));
    e = e ? e : cudaMalloc((void**)&s->env_marg, sizeof(uint32_t) * (H + 1));
    e = e ? e : cudaMalloc((void**)&s->env_cond, sizeof(uint32_t) * H * (W + 1));
    e = e ? e : cudaMalloc((void**)&s->env_texel, sizeof(float4) * W * H);
    e = e ? e : cudaMalloc((void**)&s->env_row, sizeof(float4) * H);
    e = e ? e : cudaMalloc((void**)&s->env_col, sizeof(float2) * W);
    e = e ? e : cudaMalloc((void**)&s->env_flat, sizeof(unsigned long long) * (W * H + 1));
    e = e ? e : cudaMalloc((void**)&s->env_gflat, sizeof(uint32_t) * ((size_t)s->gf + 1));
    e = e ? e : cudaMalloc((void**)&s->env_rowbase, sizeof(double) * H);
    if (e != cudaSuccess) {
        cudaGetLastError();
        mr_set_error(std::string("env table allocation failed: ") + cudaGetErrorString(e));
        return MIRRES_ERR_OOM;
    }
    return MIRRES_OK;
}

void mr_env_free(mirres_scene* s)
{
    void* ptrs[] = {s->env_w,     s->env_before, s->env_rowsum, s->env_total, s->env_ok,    s->env_marg,
                    s->env_cond,  s->env_texel,  s->env_row,    s->env_col,   s->env_flat,  s->env_gflat,
                    s->env_rowbase};
    for (void* p : ptrs)
        if (p) cudaFree(p);
}

mirres_status mr_env_build(mirres_scene* s, cudaStream_t st)
{
    const int W = s->desc.env_w, H = s->desc.env_h;
    const size_t n = (size_t)W * H;
    k_env_rows<<<H, 256, 0, st>>>(s->desc.env, W, H, s->env_w, s->env_before, s->env_rowsum, s->env_cond);
    k_env_marg<<<1, 256, 0, st>>>(s->env_rowsum, H, s->env_total, s->env_ok, s->env_marg, s->env_rowbase);
    const size_t na = std::max(n + 1, (size_t)std::max(W, H));  // texels, the last threshold, the angle tables
    k_env_tables<<<(unsigned)((na + 255) / 256), 256, 0, st>>>(s->desc.env, s->env_w, s->env_before, s->env_rowbase,
                                                              s->env_total, W, H, s->env_flat, s->env_texel,
                                                              s->env_row, s->env_col);
    k_env_flat_guide<<<(unsigned)(s->gf / GUIDE_TILE + 1), 256, 0, st>>>(s->env_flat, W * H + 1, s->gf, s->gf_shift,
                                                                        s->env_gflat);
    MR_CUDA(cudaGetLastError());
    return MIRRES_OK;
}
