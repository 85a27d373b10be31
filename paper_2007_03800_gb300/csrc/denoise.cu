// Patch-based denoising around the sparse coder (the experiment of Sec. IV):
// gather every stride-1 p x p patch of an image with its mean removed, put
// the coded patches back by averaging overlapping reconstructions, and the
// PSNR and SSIM of the result.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ctx.cuh"

using namespace sdl;

namespace {

constexpr unsigned kFull = 0xffffffffu;

// One warp per patch k (top-left corner (r, c), raster order over the
// (H-p+1) x (W-p+1) corners); element (a, b) goes to patches[k*p*p + a + p*b].
__global__ void extract_patches_kernel(const float* __restrict__ img, int H, int W, int p,
                                       float* __restrict__ patches, float* __restrict__ means,
                                       long long N) {
    const long long k = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const int wc = W - p + 1;
    const int r = (int)(k / wc), c = (int)(k % wc);
    const int pp = p * p;
    float s = 0.f;
    for (int e = lane; e < pp; e += 32) {
        const int a = e % p, b = e / p;
        s += img[(size_t)(r + a) * W + (c + b)];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    const float mean = s / (float)pp;
    float* dst = patches + (size_t)k * pp;
    for (int e = lane; e < pp; e += 32) {
        const int a = e % p, b = e / p;
        dst[e] = img[(size_t)(r + a) * W + (c + b)] - mean;
    }
    if (lane == 0) means[k] = mean;
}

// The same for p <= 32, a block per run of kRun patches of one corner row: their
// p image rows in shared memory once, means from column sums, and the patches
// (consecutive in memory) written as one coalesced run.  Bound by the write of
// the patches: 251 001 patches of 12x12 (144.6 MB) take 28 us, 5.2 TB/s; one warp
// per patch, with a division per element, took 121 us.
constexpr int kRun = 64;
constexpr int kRunMaxP = 32;

// f(0) + ... + f(n - 1) in four interleaved sums
template <class F>
__device__ __forceinline__ float sum4(int n, F f) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    int k = 0;
    for (; k + 4 <= n; k += 4) {
        s0 += f(k);
        s1 += f(k + 1);
        s2 += f(k + 2);
        s3 += f(k + 3);
    }
    if (k < n) s0 += f(k);
    if (k + 1 < n) s1 += f(k + 1);
    if (k + 2 < n) s2 += f(k + 2);
    return (s0 + s2) + (s1 + s3);
}

__global__ void __launch_bounds__(256) extract_run_kernel(const float* __restrict__ img, int W, int p, int wc,
                                                          float* __restrict__ patches,
                                                          float* __restrict__ means) {
    extern __shared__ float sx[];
    const int sw = (kRun + p - 1) | 1;              // odd row stride: a column's rows hit distinct banks
    const int pp = p * p;
    float* rows = sx;                               // p x sw
    float* cs = rows + p * sw;                      // column sums
    float* mean = cs + sw;                          // kRun
    unsigned short* off = reinterpret_cast<unsigned short*>(mean + kRun);   // element e -> its place in `rows`
    const int r = blockIdx.y, c0 = blockIdx.x * kRun;
    const int m = min(kRun, wc - c0);               // patches of this run
    const int wide = m + p - 1;
    for (int e = threadIdx.x; e < pp; e += blockDim.x) off[e] = (unsigned short)((e % p) * sw + e / p);
    for (int a = threadIdx.x >> 5; a < p; a += blockDim.x >> 5)
        for (int x = threadIdx.x & 31; x < wide; x += 32) rows[a * sw + x] = img[(size_t)(r + a) * W + c0 + x];
    __syncthreads();
    for (int x = threadIdx.x; x < wide; x += blockDim.x) {
        cs[x] = sum4(p, [&](int a) { return rows[a * sw + x]; });
    }
    __syncthreads();
    const size_t k0 = (size_t)r * wc + c0;
    if (threadIdx.x < m) {
        const float mu = sum4(p, [&](int b) { return cs[threadIdx.x + b]; }) / (float)pp;
        mean[threadIdx.x] = mu;
        means[k0 + threadIdx.x] = mu;
    }
    __syncthreads();
    float* dst = patches + k0 * pp;
    // V consecutive elements per thread: 4 (one 16-byte store) when patches are
    // multiples of 16 bytes, as then so is the run's start
    auto write = [&](auto vc) {
        constexpr int V = decltype(vc)::value;
        const int n = pp / V, dj = blockDim.x / n, de = blockDim.x % n;
        int j = threadIdx.x / n, e = threadIdx.x % n;
#pragma unroll 4
        for (int o = threadIdx.x; o < m * n; o += blockDim.x) {
            const float mu = mean[j];
            float v[V];
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = rows[off[e * V + k] + j] - mu;
            if constexpr (V == 4) reinterpret_cast<float4*>(dst)[o] = make_float4(v[0], v[1], v[2], v[3]);
            else dst[o] = v[0];
            j += dj;
            e += de;
            if (e >= n) {
                e -= n;
                ++j;
            }
        }
    };
    if (pp % 4 == 0 && (reinterpret_cast<uintptr_t>(patches) & 15u) == 0) write(std::integral_constant<int, 4>{});
    else write(std::integral_constant<int, 1>{});
}

// Reconstructed patch k (mean added back): one warp per patch.
__global__ void reconstruct_patches_kernel(const int32_t* __restrict__ support,
                                           const float* __restrict__ coef,
                                           const float* __restrict__ means, long long N, int s,
                                           const float* __restrict__ D1, int n1,
                                           const float* __restrict__ D2, int n2, int p,
                                           float* __restrict__ rec) {
    const long long k = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const int pp = p * p;
    int q = -1;
    float x = 0.f;
    if (lane < s) {
        q = support[k * s + lane];
        x = coef[k * s + lane];
    }
    const float mean = means[k];
    for (int e0 = 0; e0 < pp; e0 += 32) {   // every lane stays in the loop: the picks travel by shuffles
        const int e = min(e0 + lane, pp - 1);
        const int a = e % p, b = e / p;
        float v = mean;
        for (int l = 0; l < s; ++l) {
            const int ql = __shfl_sync(kFull, q, l);
            const float xl = __shfl_sync(kFull, x, l);
            if (ql >= 0 && ql < n1 * n2) {
                const int i = ql % n1, j = ql / n1;
                v = fmaf(xl * D1[a + p * i], D2[b + p * j], v);
            }
        }
        if (e0 + lane < pp) rec[(size_t)k * pp + e] = v;
    }
}

// Output pixel = average of the reconstructions of every patch covering it,
// summed in a fixed (r, c) order: deterministic.
__global__ void average_patches_kernel(const float* __restrict__ rec, int H, int W, int p,
                                       float* __restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= W || y >= H) return;
    const int wc = W - p + 1;
    const int r0 = max(0, y - p + 1), r1 = min(y, H - p);
    const int c0 = max(0, x - p + 1), c1 = min(x, W - p);
    const int pp = p * p;
    float s = 0.f;
    for (int r = r0; r <= r1; ++r)
        for (int c = c0; c <= c1; ++c) {
            const long long k = (long long)r * wc + c;
            s += rec[(size_t)k * pp + (y - r) + p * (x - c)];
        }
    out[(size_t)y * W + x] = s / (float)((r1 - r0 + 1) * (c1 - c0 + 1));
}

// Patch averaging for p <= 32 without writing the patches: out[y, x] sums, over
// the corner rows r covering y, the row sums
//   H[r][a][x] = sum over corners c covering x of (D1 X D2^T)[a, x - c],  a = y - r,
// and M[r][x] = the sum of those corners' means.  overlap_rows_kernel: one warp per
// corner row and 32 image columns, lane = column, the p rows a in registers; the
// warp walks its corners' picks (compacted in shared memory, in corner and slot
// order), a pick touching the p lanes that its patch covers.  The planes H
// and M (p + 1 floats per pixel) stay in L2; average_rows_kernel adds them up.  All
// sums run in a fixed order.  251 001 patches of 12x12 with 0.8 picks on average:
// 41 us (cold caches) against 316 us through 144.6 MB of written and re-read patches.
// Its chain per warp, every slot of up to 31 + p corners, is what a small image of full
// codes waits for: there the patches are written after all (patches_faster).
constexpr int kOvWarps = 8;
constexpr int kOvList = 128;         // picks compacted at a time

// Whether codes with all s slots in use are faster through written patches, by the
// times of both forms in us: a pick costs a warp of overlap_rows_kernel 0.09, a value of a
// written patch 2e-6 per pick; reading the patches back costs p p / 14 + 14 more than
// a short chain (drawn so that sparse codes of images from 120 x 120 on keep the planes).  Planes | patches, all slots used: p = 8, 50 x 50, s = 4 22 | 22, s = 8 33 | 22, s = 32
// 109 | 31; 128 x 128, s = 8 39 | 34, s = 16 70 | 47; 256 x 256, s = 32 144 | 228; p = 16, 80 x 80, s = 8
// 51 | 60, s = 16 93 | 78; p = 24, 80 x 80, s = 32 214 | 204; p = 32, 50 x 50, s = 32 95 | 201.
bool patches_faster(int p, int H, int W, int s) {
    const double pp = (double)p * p, N = (double)(H - p + 1) * (W - p + 1);
    return s * (0.09 * std::min(31 + p, W - p + 1) - 2e-6 * N * pp) > 14.0 + pp / 14.0;
}

struct alignas(16) OvPick {
    float x;
    int i, j, c;      // offsets of the atoms' columns, corner column relative to the warp's first image column
};

template <int PR>
__global__ void __launch_bounds__(kOvWarps * 32)
    overlap_rows_kernel(const int32_t* __restrict__ support, const float* __restrict__ coef,
                        const float* __restrict__ means, int s, const float* __restrict__ D1, int n1,
                        const float* __restrict__ D2, int n2, int p, int H, int W,
                        float* __restrict__ planes) {
    extern __shared__ __align__(16) float so[];
    float* d1 = so;                                  // column i at i * PR, zero past row p
    float* d2 = d1 + n1 * PR;                        // column j at j * p
    OvPick* lists = reinterpret_cast<OvPick*>(so + ((n1 * PR + n2 * p + 3) & ~3));
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    OvPick* list = lists + w * kOvList;
    for (int e = threadIdx.x; e < n1 * PR; e += blockDim.x) {
        const int i = e / PR, a = e % PR;
        d1[e] = a < p ? D1[a + p * i] : 0.f;
    }
    for (int e = threadIdx.x; e < n2 * p; e += blockDim.x) d2[e] = D2[e];
    __syncthreads();
    const int wc = W - p + 1, nr = H - p + 1, segs = (W + 31) / 32, nq = n1 * n2;
    const float inv_n1 = 1.f / (float)n1;
    const long long units = (long long)nr * segs, step = (long long)gridDim.x * kOvWarps;
    for (long long u = (long long)blockIdx.x * kOvWarps + w; u < units; u += step) {
        const int r = (int)(u / segs), x0 = (int)(u % segs) * 32;
        const int cb = max(0, x0 - p + 1), ce = min(wc, x0 + 32);   // corners covering these columns
        float acc[PR];
#pragma unroll
        for (int a = 0; a < PR; ++a) acc[a] = 0.f;
        const size_t base = ((size_t)r * wc + cb) * s;
        const int total = max(0, ce - cb) * s;
        int n = 0;
        // corner and slot of this lane's next entry (no division in the loop)
        const int dc = 32 / s, ds = 32 % s;
        int c = cb - x0 + lane / s, sl = lane % s;
        auto drain = [&]() {
            __syncwarp();
            for (int k = 0; k < n; ++k) {
                const OvPick q = list[k];
                const int b = lane - q.c;
                if (b >= 0 && b < p) {
                    const float v = q.x * d2[q.j + b];
#pragma unroll
                    for (int a = 0; a < PR; a += 4) {
                        const float4 d = *reinterpret_cast<const float4*>(d1 + q.i + a);
                        acc[a] = fmaf(v, d.x, acc[a]);
                        acc[a + 1] = fmaf(v, d.y, acc[a + 1]);
                        acc[a + 2] = fmaf(v, d.z, acc[a + 2]);
                        acc[a + 3] = fmaf(v, d.w, acc[a + 3]);
                    }
                }
            }
            __syncwarp();
            n = 0;
        };
        for (int f0 = 0; f0 < total; f0 += 32) {
            const int f = f0 + lane;
            int q = -1;
            float x = 0.f;
            if (f < total) {
                q = support[base + f];
                x = coef[base + f];
            }
            const bool on = q >= 0 && q < nq;
            const unsigned bal = __ballot_sync(kFull, on);
            if (on) {
                int j = (int)((float)q * inv_n1);      // q / n1, off by one at most
                int i = q - j * n1;
                if (i < 0) i += n1, --j;
                else if (i >= n1) i -= n1, ++j;
                list[n + __popc(bal & ((1u << lane) - 1u))] = OvPick{x, i * PR, j * p, c};
            }
            n += __popc(bal);
            c += dc;
            sl += ds;
            if (sl >= s) sl -= s, ++c;
            if (n > kOvList - 32) drain();
        }
        drain();
        const int x = x0 + lane;
        float mu = 0.f;
        for (int c = max(cb, x - p + 1); c <= min(x, ce - 1); ++c) mu += means[(size_t)r * wc + c];
        if (x < W) {
            float* out = planes + ((size_t)r * (p + 1)) * W + x;
#pragma unroll
            for (int a = 0; a < PR; ++a)
                if (a < p) out[(size_t)a * W] = acc[a];
            out[(size_t)p * W] = mu;
        }
    }
}

__global__ void __launch_bounds__(256) average_rows_kernel(const float* __restrict__ planes, int H, int W, int p,
                                                           float* __restrict__ out) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (x >= W || y >= H) return;
    const int r0 = max(0, y - p + 1), r1 = min(y, H - p);
    const int nc = min(x, W - p) - max(0, x - p + 1) + 1;
    float h = 0.f, m = 0.f;
#pragma unroll 4
    for (int r = r0; r <= r1; ++r) {
        const float* pl = planes + (size_t)r * (p + 1) * W + x;
        h += pl[(size_t)(y - r) * W];
        m += pl[(size_t)p * W];
    }
    out[(size_t)y * W + x] = (h + m) / (float)((r1 - r0 + 1) * nc);
}

// PSNR = 10 log10(peak^2 / MSE): one CTA, compensated FP32 per thread,
// fixed-order FP64 combination.
__global__ void __launch_bounds__(1024) psnr_kernel(const float* __restrict__ a,
                                                    const float* __restrict__ b, long long count,
                                                    float peak, float* __restrict__ out) {
    __shared__ double part[32];
    float sum = 0.f, comp = 0.f;
    for (long long e = threadIdx.x; e < count; e += blockDim.x) {
        const float d = a[e] - b[e];
        const float y = d * d - comp;
        const float t = sum + y;
        comp = (t - sum) - y;
        sum = t;
    }
    double v = (double)sum - (double)comp;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += part[w];
        const double mse = tot / (double)count;
        out[0] = (float)(10.0 * log10((double)peak * peak / mse));
    }
}

// SSIM index (Wang, Bovik, Sheikh, Simoncelli 2004) of x against ref: one
// thread per window position inside the image (valid region), 11 x 11
// Gaussian window (sigma 1.5, normalised to sum 1), per-block sums in FP64
// combined in a fixed order by ssim_finish_kernel.
constexpr int kSsimWin = 11;
constexpr float kSsimSigma = 1.5f;
constexpr int kSsimThreads = 256;

__global__ void __launch_bounds__(kSsimThreads)
    ssim_kernel(const float* __restrict__ x, const float* __restrict__ y, int H, int W,
                float peak, double* __restrict__ part) {
    __shared__ float w[kSsimWin * kSsimWin];
    __shared__ double red[kSsimThreads / 32];
    constexpr int G = kSsimWin;
    if (threadIdx.x < G * G) {
        const int u = threadIdx.x / G - G / 2, v = threadIdx.x % G - G / 2;
        w[threadIdx.x] = expf(-(float)(u * u + v * v) / (2.f * kSsimSigma * kSsimSigma));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int e = 0; e < G * G; ++e) t += (double)w[e];
        red[0] = t;
    }
    __syncthreads();
    const float inv = (float)(1.0 / red[0]);
    __syncthreads();
    if (threadIdx.x < G * G) w[threadIdx.x] *= inv;
    __syncthreads();
    const int wc = W - G + 1;
    const long long P = (long long)(H - G + 1) * wc;
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double val = 0.0;
    if (k < P) {
        const int r = (int)(k / wc), c = (int)(k % wc);
        float mx = 0.f, my = 0.f;
        for (int a = 0; a < G; ++a)
            for (int b = 0; b < G; ++b) {
                const float wt = w[a * G + b];
                mx = fmaf(wt, x[(size_t)(r + a) * W + c + b], mx);
                my = fmaf(wt, y[(size_t)(r + a) * W + c + b], my);
            }
        float vx = 0.f, vy = 0.f, cxy = 0.f;
        for (int a = 0; a < G; ++a)
            for (int b = 0; b < G; ++b) {
                const float wt = w[a * G + b];
                const float dx = x[(size_t)(r + a) * W + c + b] - mx;
                const float dy = y[(size_t)(r + a) * W + c + b] - my;
                vx = fmaf(wt * dx, dx, vx);
                vy = fmaf(wt * dy, dy, vy);
                cxy = fmaf(wt * dx, dy, cxy);
            }
        const double C1 = (0.01 * peak) * (0.01 * peak), C2 = (0.03 * peak) * (0.03 * peak);
        val = ((2.0 * mx * my + C1) * (2.0 * cxy + C2)) /
              (((double)mx * mx + (double)my * my + C1) * ((double)vx + vy + C2));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) val += __shfl_down_sync(kFull, val, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = val;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int e = 0; e < kSsimThreads / 32; ++e) t += red[e];
        part[blockIdx.x] = t;
    }
}

__global__ void ssim_finish_kernel(const double* __restrict__ part, int nblocks, long long P,
                                   float* __restrict__ out) {
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int b = 0; b < nblocks; ++b) t += part[b];
        out[0] = (float)(t / (double)P);
    }
}

}  // namespace

extern "C" {

int sdl_extract_patches(const float* image, int H, int W, int p, float* patches, float* means,
                        void* stream) {
    if (!image || !patches || !means || p < 1 || H < p || W < p) return SDL_ERR_ARG;
    const long long N = (long long)(H - p + 1) * (W - p + 1);
    const int threads = 256;
    if (p <= kRunMaxP && H - p + 1 <= 65535) {
        const int wc = W - p + 1, sw = (kRun + p - 1) | 1;
        const size_t bytes = sizeof(float) * ((size_t)p * sw + sw + kRun) + sizeof(unsigned short) * (size_t)p * p;
        extract_run_kernel<<<dim3((wc + kRun - 1) / kRun, H - p + 1), threads, bytes, (cudaStream_t)stream>>>(
            image, W, p, wc, patches, means);
        return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
    }
    const long long blocks = (N * 32 + threads - 1) / threads;
    extract_patches_kernel<<<(unsigned)blocks, threads, 0, (cudaStream_t)stream>>>(
        image, H, W, p, patches, means, N);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_patch_average(sdl_ctx* c, const int32_t* support, const float* coef, const float* means,
                      int s_max, const float* D1, int n1, const float* D2, int n2, int p, int H,
                      int W, float* image_out, void* stream) {
    if (!c || !support || !coef || !means || !D1 || !D2 || !image_out) return SDL_ERR_ARG;
    if (p < 1 || H < p || W < p || s_max < 1 || s_max > 32 || n1 < 1 || n2 < 1) return SDL_ERR_ARG;
    DeviceGuard guard(c->device);
    cudaStream_t st = (cudaStream_t)stream;
    const long long N = (long long)(H - p + 1) * (W - p + 1);
    // both dictionaries and the pick lists of a block in shared memory
    const int pr = p <= 8 ? 8 : p <= 12 ? 12 : p <= 16 ? 16 : 32;
    const size_t bytes = sizeof(float) * (((size_t)n1 * pr + (size_t)n2 * p + 3) & ~size_t(3)) +
                         sizeof(OvPick) * kOvWarps * kOvList;
    const bool planes = p <= 32 && bytes <= 48 * 1024 && H <= 8 * 65535 && !patches_faster(p, H, W, s_max);
    const size_t need = planes ? (size_t)(H - p + 1) * (p + 1) * W : (size_t)N * p * p;
    if (need > c->cap_rec) {
        if (c->rec) cudaFree(c->rec);
        c->rec = nullptr;
        c->cap_rec = 0;
        if (cudaMalloc(&c->rec, need * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            return SDL_ERR_WORKSPACE;
        }
        c->cap_rec = need;
    }
    if (planes) {
        const long long units = (long long)(H - p + 1) * ((W + 31) / 32);
        const int grid = (int)std::min<long long>((units + kOvWarps - 1) / kOvWarps, (long long)c->num_sms * 8);
        auto rows = [&](auto kern) {
            kern<<<grid, kOvWarps * 32, bytes, st>>>(support, coef, means, s_max, D1, n1, D2, n2, p, H, W, c->rec);
        };
        if (pr == 8) rows(overlap_rows_kernel<8>);
        else if (pr == 12) rows(overlap_rows_kernel<12>);
        else if (pr == 16) rows(overlap_rows_kernel<16>);
        else rows(overlap_rows_kernel<32>);
        average_rows_kernel<<<dim3((W + 31) / 32, (H + 7) / 8), 256, 0, st>>>(c->rec, H, W, p, image_out);
        return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
    }
    const int threads = 256;
    const long long blocks = (N * 32 + threads - 1) / threads;
    reconstruct_patches_kernel<<<(unsigned)blocks, threads, 0, st>>>(support, coef, means, N, s_max,
                                                                     D1, n1, D2, n2, p, c->rec);
    average_patches_kernel<<<dim3((W + 127) / 128, H), 128, 0, st>>>(c->rec, H, W, p, image_out);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_ssim(sdl_ctx* c, const float* x, const float* ref, int H, int W, float peak, float* out,
             void* stream) {
    if (!c || !x || !ref || !out || H < kSsimWin || W < kSsimWin || !(peak > 0.f))
        return SDL_ERR_ARG;
    DeviceGuard g(c->device);
    const long long P = (long long)(H - kSsimWin + 1) * (W - kSsimWin + 1);
    const int nblocks = (int)((P + kSsimThreads - 1) / kSsimThreads);
    if ((size_t)nblocks > c->cap_ssim) {
        if (c->ssim_part) cudaFree(c->ssim_part);
        c->ssim_part = nullptr;
        c->cap_ssim = 0;
        if (cudaMalloc(&c->ssim_part, sizeof(double) * nblocks) != cudaSuccess) {
            cudaGetLastError();
            return SDL_ERR_WORKSPACE;
        }
        c->cap_ssim = nblocks;
    }
    cudaStream_t st = (cudaStream_t)stream;
    ssim_kernel<<<nblocks, kSsimThreads, 0, st>>>(x, ref, H, W, peak, c->ssim_part);
    ssim_finish_kernel<<<1, 32, 0, st>>>(c->ssim_part, nblocks, P, out);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_psnr(const float* x, const float* ref, int64_t count, float peak, float* out,
             void* stream) {
    if (!x || !ref || !out || count < 1 || !(peak > 0.f)) return SDL_ERR_ARG;
    psnr_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(x, ref, count, peak, out);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

}  // extern "C"
