// Learned support proposal: a two-layer network (p1*p2 -> hidden, GELU ->
// n1*n2 scores) trained on the GPU on (signal, 2D-OMP support) pairs, whose
// top-k scores shortlist the atom pairs that 2D-OMP then searches.
//
//   x = vec(Y)/||Y||,  h = GELU(W1 x + b1),  z = W2 h + b2
//   loss = mean_b sum_q softplus(z) - t z   (t: multi-hot OMP support)
//
// Forward and backward run as tcgen05 GEMMs (tc_gemm.cu) with fused
// epilogues; this file holds the element-wise kernels (input scaling, the
// loss gradient, bias-gradient reductions, Adam), the warp top-k and the deterministic
// compaction of the fallback signals; 2D-OMP on the shortlists with its fallback
// test is omp_group_short.cu.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <utility>
#include <vector>

#include "ctx.cuh"

using namespace sdl;
using bf16 = __nv_bfloat16;

struct sdl_mlp {
    sdl_ctx* ctx = nullptr;
    int P = 0, H = 0, Q = 0, Kp = 0, Bmax = 0, step = 0;
    int rows = 0;                // signals that Xb and Hb hold: a training batch or an inference chunk
    float *W1 = nullptr, *b1 = nullptr, *W2 = nullptr, *b2 = nullptr;
    float *mW1, *vW1, *mb1, *vb1, *mW2, *vW2, *mb2, *vb2;
    float *gW1, *gb1, *gW2, *gb2;
    bf16 *W1b, *W2b, *W2Tb;
    bf16 *Xb, *XTb, *Hb, *HTb, *dZb, *dZTb, *dPreTb;
    float *pre, *Z, *lossp;
    char* mem = nullptr;
};

namespace {

constexpr unsigned kFull = 0xffffffffu;

// x = vec(Y_k)/||Y_k|| as BF16 rows (zero padded to Kp)
__global__ void prep_input_kernel(const float* __restrict__ Y, long long N, int P, int Kp, bf16* __restrict__ X) {
    const long long k = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const float* y = Y + (size_t)k * P;
    float ss = 0.f;
    for (int e = lane; e < P; e += 32) ss = fmaf(y[e], y[e], ss);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(kFull, ss, o);
    const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
    for (int e = lane; e < Kp; e += 32) {
        const bf16 v = __float2bfloat16_rn(e < P ? y[e] * inv : 0.f);
        X[(size_t)k * Kp + e] = v;
    }
}

// The same rows for inference when p1 p2 is a multiple of 4 and Y is 16-byte aligned: 8 lanes
// per signal, 16-byte loads and 8-byte stores, the norm in the same 32 chains and
// order (lane j holds chains 4j .. 4j + 3); one square root per four signals.
// 32 768 x 64: 7.4 us, 13 with a warp per signal (latency of 4-byte loads and of one
// root per signal).
__global__ void __launch_bounds__(256) prep_rows_kernel(const float* __restrict__ Y, long long N, int P, int Kp,
                                                        bf16* __restrict__ X) {
    const int lane = threadIdx.x & 31, j = lane & 7;
    const long long k = ((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5) * 4 + (lane >> 3);
    const float* src = Y + (size_t)k * P;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (k < N) {
#pragma unroll 4
        for (int e = 4 * j; e < P; e += 32) {
            const float4 y = *reinterpret_cast<const float4*>(src + e);
            v[0] = fmaf(y.x, y.x, v[0]);
            v[1] = fmaf(y.y, y.y, v[1]);
            v[2] = fmaf(y.z, y.z, v[2]);
            v[3] = fmaf(y.w, y.w, v[3]);
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(kFull, v[c], o);
    const float ss = (v[0] + v[2]) + (v[1] + v[3]);
    const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
    if (k < N) {
#pragma unroll 4
        for (int e = 4 * j; e < Kp; e += 32) {
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e < P) y = *reinterpret_cast<const float4*>(src + e);   // still in L1
            const __nv_bfloat162 a = __floats2bfloat162_rn(y.x * inv, y.y * inv);
            const __nv_bfloat162 b = __floats2bfloat162_rn(y.z * inv, y.w * inv);
            *reinterpret_cast<uint2*>(X + (size_t)k * Kp + e) =
                make_uint2(*reinterpret_cast<const unsigned*>(&a), *reinterpret_cast<const unsigned*>(&b));
        }
    }
}

// The same for a training batch, with the transposed copy: a block takes 32
// signals, and both copies leave as coalesced rows (the norm, in the same order,
// by one warp per signal).
__global__ void __launch_bounds__(256) prep_batch_kernel(const float* __restrict__ Y, int N, int P, int Kp,
                                                         bf16* __restrict__ X, bf16* __restrict__ XT, int ldt) {
    __shared__ float inv_s[32];
    __shared__ bf16 tile[32][66];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, k0 = blockIdx.x * 32;
    for (int i = w; i < 32; i += 8) {
        float ss = 0.f;
        if (k0 + i < N) {
            const float* y = Y + (size_t)(k0 + i) * P;
            for (int e = lane; e < P; e += 32) ss = fmaf(y[e], y[e], ss);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(kFull, ss, o);
        if (lane == 0) inv_s[i] = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
    }
    __syncthreads();
    for (int e0 = 0; e0 < Kp; e0 += 64) {
        for (int t = threadIdx.x; t < 32 * 64; t += 256) {
            const int i = t >> 6, e = e0 + (t & 63), k = k0 + i;
            bf16 v = __float2bfloat16_rn(0.f);
            if (k < N && e < P) v = __float2bfloat16_rn(Y[(size_t)k * P + e] * inv_s[i]);
            if (k < N && e < Kp) X[(size_t)k * Kp + e] = v;
            tile[i][t & 63] = v;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < 32 * 64; t += 256) {
            const int e = e0 + (t >> 5), k = k0 + (t & 31);
            if (k < N && e < Kp) XT[(size_t)e * ldt + k] = tile[t & 31][t >> 5];
        }
        __syncthreads();
    }
}

// dz = (sigmoid(z) - t) * scale, loss terms softplus(z) - t z; a block takes 32
// signals x 64 scores, so that dZ and its transpose leave as coalesced rows
// (one block per signal wrote the transpose 2 bytes at a time: 29 us for a batch of
// 4096 x 576).  lossp: one sum per (column block, signal).
constexpr int kBceCols = 64;

__global__ void __launch_bounds__(256)
    bce_kernel(const float* __restrict__ Z, int ldz, const int32_t* __restrict__ sup, int s, int B, int Q,
               float scale, bf16* __restrict__ dZ, int lddz, bf16* __restrict__ dZT, int lddt,
               float* __restrict__ lossp) {
    __shared__ unsigned long long hit[32];     // bit c: pair q0 + c is in the signal's support
    __shared__ bf16 tile[32][kBceCols + 2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b0 = blockIdx.x * 32, q0 = blockIdx.y * kBceCols;
    if (threadIdx.x < 32) {
        unsigned long long h = 0;
        if (b0 + lane < B)
            for (int l = 0; l < s; ++l) {
                const int c = sup[(size_t)(b0 + lane) * s + l] - q0;
                if (c >= 0 && c < kBceCols) h |= 1ull << c;
            }
        hit[lane] = h;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = w * 4 + r, b = b0 + i;
        const unsigned long long h = hit[i];
        float acc = 0.f;
#pragma unroll
        for (int c = lane; c < kBceCols; c += 32) {
            const int q = q0 + c;
            if (b < B && q < Q) {
                const float t = (float)((h >> c) & 1ull);
                const float z = Z[(size_t)b * ldz + q];
                acc += fmaxf(z, 0.f) - t * z + log1pf(expf(-fabsf(z)));
                const float g = (1.f / (1.f + expf(-z)) - t) * scale;
                const bf16 gb = __float2bfloat16_rn(g);
                dZ[(size_t)b * lddz + q] = gb;
                tile[i][c] = gb;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (lane == 0 && b < B) lossp[(size_t)blockIdx.y * B + b] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 32 * kBceCols; t += 256) {
        const int q = q0 + (t >> 5), b = b0 + (t & 31);
        if (b < B && q < Q) dZT[(size_t)q * lddt + b] = tile[t & 31][t >> 5];
    }
}

// The bias gradients out[r] = sum_c M[r, c] of two BF16 matrices with the same
// columns (one warp per row, fixed order), and in the last block the mean loss.
__global__ void __launch_bounds__(256)
    row_sums_kernel(const bf16* __restrict__ M1, int R1, float* __restrict__ out1, const bf16* __restrict__ M2,
                    int R2, float* __restrict__ out2, int ld, int C, const float* __restrict__ lossp, int nloss,
                    float scale, float* __restrict__ loss) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float part[8];
        if (!loss) return;
        float acc = 0.f;
#pragma unroll 8
        for (int i = threadIdx.x; i < nloss; i += 256) acc += lossp[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (lane == 0) part[w] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int v = 0; v < 8; ++v) t += part[v];
            loss[0] = t * scale;
        }
        return;
    }
    int r = blockIdx.x * 8 + w;
    const bf16* M = M1;
    float* out = out1;
    if (r >= R1) {
        r -= R1;
        M = M2;
        out = out2;
        if (r >= R2) return;
    }
    float acc = 0.f;
    const bf16* row = M + (size_t)r * ld;
#pragma unroll 16
    for (int c = lane; c < C; c += 32) acc += __bfloat162float(row[c]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    if (lane == 0) out[r] = acc;
}

struct AdamJob {
    float *p, *m, *v;
    const float* g;
    int rows, cols, blocks;  // 32 x 32 blocks
    bf16 *pb, *pbT;          // BF16 copies (row-major, transposed) or null
};
struct AdamJobs {
    AdamJob job[4];
};

// Adam on FP32 master weights for the four parameter arrays in one launch;
// refreshes the BF16 copies (the transposed one through shared memory)
__global__ void __launch_bounds__(256)
    adam_kernel(const __grid_constant__ AdamJobs jobs, float lr, float beta1, float beta2, float eps, float bc1,
                float bc2) {
    __shared__ bf16 tile[32][34];
    int blk = blockIdx.x, k = 0;
    while (k < 3 && blk >= jobs.job[k].blocks) blk -= jobs.job[k++].blocks;
    const AdamJob& q = jobs.job[k];
    const int cb = (q.cols + 31) / 32, r0 = blk / cb * 32, c0 = blk % cb * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = r0 + w + 8 * u, c = c0 + lane;
        if (r >= q.rows || c >= q.cols) continue;
        const size_t i = (size_t)r * q.cols + c;
        const float gi = q.g[i];
        const float mi = beta1 * q.m[i] + (1.f - beta1) * gi;
        const float vi = beta2 * q.v[i] + (1.f - beta2) * gi * gi;
        q.m[i] = mi;
        q.v[i] = vi;
        const float pn = q.p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        q.p[i] = pn;
        const bf16 b = __float2bfloat16_rn(pn);
        if (q.pb) q.pb[i] = b;
        tile[w + 8 * u][lane] = b;
    }
    if (!q.pbT) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int c = c0 + w + 8 * u, r = r0 + lane;
        if (c < q.cols && r < q.rows) q.pbT[(size_t)c * q.rows + r] = tile[lane][w + 8 * u];
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ p, int rows, int cols,
                               bf16* __restrict__ pb, bf16* __restrict__ pbT) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * cols) return;
    const bf16 b = __float2bfloat16_rn(p[i]);
    if (pb) pb[i] = b;
    if (pbT) pbT[(size_t)(i % cols) * rows + i / cols] = b;
}

// ---------------------------------------------------------------- top-k
// order-preserving 16-bit key of a float (larger float -> larger key)
__device__ __forceinline__ unsigned key16(float f) {
    unsigned u = __float_as_uint(f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return u >> 16;
}

// Per signal: the k1 best scores (the shortlist) and the next k2 - k1 (the
// fallback check set), ranked by 16-bit key then by smaller pair index; each
// of the two sets is written in increasing pair index.
// One warp per signal; lane holds scores q = lane + 32 e.
template <int EQ>
__global__ void topk_kernel(const float* __restrict__ Z, int ldz, long long N, int Q, int k1,
                            int k2, int32_t* __restrict__ out) {
    const long long k = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    unsigned key[EQ];
#pragma unroll
    for (int e = 0; e < EQ; ++e) {
        const int q = lane + 32 * e;
        const float z = (q < Q) ? Z[(size_t)k * ldz + q] : 0.f;
        key[e] = (q < Q && z == z) ? key16(z) + 1u : 0u;   // 0 = no entry (past Q, or NaN)
    }
    auto count_ge = [&](unsigned t) {
        int c = 0;
#pragma unroll
        for (int e = 0; e < EQ; ++e) c += key[e] >= t ? 1 : 0;
        return (int)__reduce_add_sync(kFull, (unsigned)c);
    };
    // At least 32 keys reach the smallest of the lanes' maxima: the search for up to
    // 32 of them starts there and ends at the largest key (256 scores, k = 32:
    // 28 -> 23 us per 32 768 signals against bisecting all 17 bits).
    unsigned top = key[0];
#pragma unroll
    for (int e = 1; e < EQ; ++e) top = max(top, key[e]);
    const unsigned low = __reduce_min_sync(kFull, top);
    top = __reduce_max_sync(kFull, top);
    // largest threshold with at least kk keys >= it (0: there are fewer), or the first
    // one met with exactly kk: then no key ties for the last place, and the set is the same
    auto threshold = [&](int kk, bool& exact) {
        unsigned t = kk <= 32 ? low : 0u, hi = top;
        exact = false;
        while (t < hi) {
            const unsigned c = (t + hi + 1u) >> 1;
            const int n = count_ge(c);
            if (n >= kk) t = c;
            else hi = c - 1u;
            if (n == kk) {
                exact = true;
                break;
            }
        }
        return t;
    };
    // membership masks of the top-kk set (ties at the threshold by smaller q)
    auto select = [&](int kk) {
        bool exact;
        const unsigned t = threshold(kk, exact);
        unsigned mask = 0;
        if (exact) {
#pragma unroll
            for (int e = 0; e < EQ; ++e)
                if (key[e] >= t) mask |= 1u << e;
            return mask;
        }
        int above = 0;
#pragma unroll
        for (int e = 0; e < EQ; ++e) {
            if (key[e] > t) mask |= 1u << e;
            above += key[e] > t ? 1 : 0;
        }
        int need = kk - (int)__reduce_add_sync(kFull, (unsigned)above);
#pragma unroll
        for (int e = 0; e < EQ; ++e) {      // q = lane + 32 e ascending: e outer, lane inner
            const bool eq = key[e] == t && t > 0;
            const unsigned bal = __ballot_sync(kFull, eq);
            const int rank = __popc(bal & ((1u << lane) - 1u));
            if (eq && rank < need) mask |= 1u << e;
            need -= min(need, __popc(bal));
        }
        return mask;
    };
    const unsigned m1 = select(k1);
    const unsigned m2 = k2 > k1 ? select(k2) & ~m1 : 0u;   // no check set: one bisection
    int base = 0;
    int32_t* o = out + (size_t)k * k2;
    for (int pass = 0; pass < (k2 > k1 ? 2 : 1); ++pass) {
        const unsigned msk = pass == 0 ? m1 : m2;
        if (pass == 1) base = k1;
        int written = 0;
#pragma unroll
        for (int e = 0; e < EQ; ++e) {
            const bool on = (msk >> e) & 1u;
            const unsigned bal = __ballot_sync(kFull, on);
            if (on) o[base + written + __popc(bal & ((1u << lane) - 1u))] = lane + 32 * e;
            written += __popc(bal);
        }
        const int lim = pass == 0 ? k1 : k2;
        for (int p = base + written + lane; p < lim; p += 32) o[p] = -1;   // fewer valid scores
    }
}

// ---------------------------------------------------------------- compaction
constexpr int kScanBlock = 1024;

__global__ void count_flags_kernel(const int32_t* __restrict__ flag, long long N,
                                   int* __restrict__ blockcnt) {
    __shared__ int wsum[32];
    const long long i = blockIdx.x * (long long)kScanBlock + threadIdx.x;
    const int f = (i < N && flag[i]) ? 1 : 0;
    const int c = __popc(__ballot_sync(kFull, f));
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kScanBlock / 32; ++w) t += wsum[w];
        blockcnt[blockIdx.x] = t;
    }
}

__global__ void scan_counts_kernel(int* __restrict__ blockcnt, int nblocks, int* __restrict__ total) {
    // one warp, 32 counts at a time
    int run = 0;
    for (int b0 = 0; b0 < nblocks; b0 += 32) {
        const int b = b0 + (int)threadIdx.x;
        const int c = b < nblocks ? blockcnt[b] : 0;
        int s = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, s, o);
            if ((int)threadIdx.x >= o) s += v;
        }
        if (b < nblocks) blockcnt[b] = run + s - c;
        run += __shfl_sync(kFull, s, 31);
    }
    if (threadIdx.x == 0) total[0] = run;
}

__global__ void write_index_kernel(const int32_t* __restrict__ flag, long long N,
                                   const int* __restrict__ blockoff, int32_t* __restrict__ idx) {
    __shared__ int woff[32];
    const long long i = blockIdx.x * (long long)kScanBlock + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int f = (i < N && flag[i]) ? 1 : 0;
    const unsigned bal = __ballot_sync(kFull, f);
    if (lane == 0) woff[w] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int ww = 0; ww < kScanBlock / 32; ++ww) {
            const int c = woff[ww];
            woff[ww] = run;
            run += c;
        }
    }
    __syncthreads();
    if (f) idx[blockoff[blockIdx.x] + woff[w] + __popc(bal & ((1u << lane) - 1u))] = (int32_t)i;
}

// ---------------------------------------------------------------- RMSE guard
// The plain coder judges the learned one on a strided sample of the signals:
// if the learned codes' RMSE there exceeds the plain coder's by more than 1 %,
// every signal is coded again by the plain coder.
constexpr double kGuardRmseRatio = 1.01;
constexpr int kGuardThreads = 256;
constexpr long long kGuardMinSample = 4096;

__global__ void sample_index_kernel(int32_t* __restrict__ idx, int m, long long stride,
                                    int* __restrict__ count) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < m) idx[r] = (int32_t)(r * stride);
    if (r == 0) *count = m;
}

// Fixed-order FP64 sums of the two residual energies over the sample, a pair per CTA
// (one CTA alone spends 24 us on 2 x 12 500 of them, FP64 adds at one SM's rate; 13 us
// with the decision in a launch of its own).
constexpr int kGuardCtas = 64;
__global__ void __launch_bounds__(kGuardThreads)
    guard_sums_kernel(const float* __restrict__ plainE, const float* __restrict__ learnedE,
                      const int32_t* __restrict__ idx, int m, double2* __restrict__ part) {
    __shared__ double sp[kGuardThreads / 32], sl[kGuardThreads / 32];
    double a = 0.0, b = 0.0;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < m; r += (long long)gridDim.x * blockDim.x) {
        a += (double)plainE[r];
        b += (double)learnedE[idx[r]];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(kFull, a, o);
        b += __shfl_down_sync(kFull, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sp[threadIdx.x >> 5] = a;
        sl[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < kGuardThreads / 32; ++w) {
            ta += sp[w];
            tb += sl[w];
        }
        part[blockIdx.x] = make_double2(ta, tb);
    }
}

// one warp: the decision from the kGuardCtas pairs
__global__ void guard_kernel(const double2* __restrict__ part, int m, long long N, int P, int* __restrict__ recode_count,
                             int32_t* __restrict__ n_fallback, float* __restrict__ guard_out) {
    double ta = 0.0, tb = 0.0;
    for (int c = threadIdx.x; c < kGuardCtas; c += 32) {
        ta += part[c].x;
        tb += part[c].y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ta += __shfl_down_sync(kFull, ta, o);
        tb += __shfl_down_sync(kFull, tb, o);
    }
    if (threadIdx.x == 0) {
        const bool fail = tb > kGuardRmseRatio * kGuardRmseRatio * ta;
        *recode_count = fail ? (int)N : 0;
        if (fail) *n_fallback = (int32_t)N;
        if (guard_out) {
            const double scale = 1.0 / ((double)m * P);
            guard_out[0] = (float)sqrt(tb * scale);
            guard_out[1] = (float)sqrt(ta * scale);
            guard_out[2] = fail ? 1.f : 0.f;
        }
    }
}

__global__ void mark_all_kernel(const int* __restrict__ recode_count, long long N,
                                int32_t* __restrict__ idx, int32_t* __restrict__ fallback) {
    if (*recode_count == 0) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        idx[i] = (int32_t)i;
        fallback[i] = 1;
    }
}

template <class T>
T* carve(char*& p, size_t n) {
    T* r = reinterpret_cast<T*>(p);
    p += (n * sizeof(T) + 255) & ~size_t(255);
    return r;
}

// The context's second stream and its events, made with its first network.
int side_stream(sdl_ctx* c) {
    if (!c->side && cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess) return SDL_ERR_CUDA;
    for (cudaEvent_t& e : c->side_ev)
        if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return SDL_ERR_CUDA;
    return SDL_OK;
}

int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

// Inference runs in chunks of this many signals: a 4096-signal chunk leaves
// every SM one 128 x 128 tile per GEMM, so that nothing hides the epilogue's GELU
// (23 us per chunk at 64 -> 512; 8 times the signals take 36 us), while the
// activations and scores of a chunk still stay in L2.  The network holds the
// buffers of a chunk from its creation on, so that a forward pass allocates
// nothing and may be captured; wide networks take shorter chunks.
constexpr int kInferChunk = 32768;
constexpr size_t kInferBytes = size_t(64) << 20;

}  // namespace

extern "C" {

int sdl_mlp_create(sdl_ctx* c, int p1, int p2, int n1, int n2, int hidden, int max_batch,
                   sdl_mlp** out) {
    if (!out) return SDL_ERR_ARG;
    *out = nullptr;
    if (!c || p1 < 1 || p2 < 1 || n1 < 1 || n2 < 1 || hidden < 8 || hidden % 8 ||
        max_batch < 8 || max_batch % 8 || (long long)n1 * n2 > 1024 || (long long)n1 * n2 % 8)
        return SDL_ERR_ARG;
    DeviceGuard guard(c->device);
    sdl_mlp* m = new (std::nothrow) sdl_mlp();
    if (!m) return SDL_ERR_WORKSPACE;
    m->ctx = c;
    m->P = p1 * p2;
    m->Kp = (m->P + 7) & ~7;
    m->H = hidden;
    m->Q = n1 * n2;
    m->Bmax = max_batch;
    const size_t H = m->H, Kp = m->Kp, Q = m->Q, B = m->Bmax;
    m->rows = std::max(m->Bmax, (int)std::min<size_t>(kInferChunk, kInferBytes / (2 * (Kp + H)) & ~size_t(127)));
    const size_t R = m->rows;
    const size_t nf = 4 * (H * Kp + H + Q * H + Q) + 1024;     // params, m, v, grads
    const size_t nloss = B * ((Q + kBceCols - 1) / kBceCols);
    const size_t bytes = (nf * 4 + nloss * 4 + (H * Kp + 2 * Q * H) * 2 +
                          (R * Kp + B * Kp + R * H + B * H + 2 * B * Q + B * H) * 2 +
                          (B * H + B * Q + B) * 4) + 64 * 256;
    if (side_stream(c) != SDL_OK) {
        delete m;
        return SDL_ERR_CUDA;
    }
    if (cudaMalloc(&m->mem, bytes) != cudaSuccess) {
        cudaGetLastError();
        delete m;
        return SDL_ERR_WORKSPACE;
    }
    cudaMemset(m->mem, 0, bytes);
    char* p = m->mem;
    m->W1 = carve<float>(p, H * Kp); m->b1 = carve<float>(p, H);
    m->W2 = carve<float>(p, Q * H); m->b2 = carve<float>(p, Q);
    m->mW1 = carve<float>(p, H * Kp); m->vW1 = carve<float>(p, H * Kp);
    m->mb1 = carve<float>(p, H); m->vb1 = carve<float>(p, H);
    m->mW2 = carve<float>(p, Q * H); m->vW2 = carve<float>(p, Q * H);
    m->mb2 = carve<float>(p, Q); m->vb2 = carve<float>(p, Q);
    m->gW1 = carve<float>(p, H * Kp); m->gb1 = carve<float>(p, H);
    m->gW2 = carve<float>(p, Q * H); m->gb2 = carve<float>(p, Q);
    m->W1b = carve<bf16>(p, H * Kp); m->W2b = carve<bf16>(p, Q * H); m->W2Tb = carve<bf16>(p, H * Q);
    m->Xb = carve<bf16>(p, R * Kp); m->XTb = carve<bf16>(p, Kp * B);
    m->Hb = carve<bf16>(p, R * H); m->HTb = carve<bf16>(p, H * B);
    m->dZb = carve<bf16>(p, B * Q); m->dZTb = carve<bf16>(p, Q * B);
    m->dPreTb = carve<bf16>(p, H * B);
    m->pre = carve<float>(p, B * H); m->Z = carve<float>(p, B * Q); m->lossp = carve<float>(p, nloss);
    if ((size_t)(p - m->mem) > bytes) {
        cudaFree(m->mem);
        delete m;
        return SDL_ERR_WORKSPACE;
    }
    *out = m;
    return SDL_OK;
}

int sdl_mlp_destroy(sdl_mlp* m) {
    if (!m) return SDL_OK;
    DeviceGuard guard(m->ctx->device);
    cudaDeviceSynchronize();
    cudaFree(m->mem);
    delete m;
    return SDL_OK;
}

// Host FP32 arrays: W1 [hidden x p1p2], b1 [hidden], W2 [n1n2 x hidden], b2 [n1n2].
// Either direction is synchronous; Adam moments and the step count are reset on set.
int sdl_mlp_set_weights(sdl_mlp* m, const float* W1, const float* b1, const float* W2,
                        const float* b2) {
    if (!m || !W1 || !b1 || !W2 || !b2) return SDL_ERR_ARG;
    DeviceGuard guard(m->ctx->device);
    std::vector<float> w1((size_t)m->H * m->Kp, 0.f);
    for (int h = 0; h < m->H; ++h)
        for (int e = 0; e < m->P; ++e) w1[(size_t)h * m->Kp + e] = W1[(size_t)h * m->P + e];
    const size_t H = m->H, Kp = m->Kp, Q = m->Q;
    if (cudaMemcpy(m->W1, w1.data(), H * Kp * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->b1, b1, H * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->W2, W2, Q * H * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->b2, b2, Q * 4, cudaMemcpyHostToDevice) != cudaSuccess)
        return SDL_ERR_CUDA;
    for (float* z : {m->mW1, m->vW1, m->gW1}) cudaMemset(z, 0, H * Kp * 4);
    for (float* z : {m->mb1, m->vb1, m->gb1}) cudaMemset(z, 0, H * 4);
    for (float* z : {m->mW2, m->vW2, m->gW2}) cudaMemset(z, 0, Q * H * 4);
    for (float* z : {m->mb2, m->vb2, m->gb2}) cudaMemset(z, 0, Q * 4);
    m->step = 0;
    to_bf16_kernel<<<blocks_for(H * Kp, 256), 256>>>(m->W1, (int)H, (int)Kp, m->W1b, nullptr);
    to_bf16_kernel<<<blocks_for(Q * H, 256), 256>>>(m->W2, (int)Q, (int)H, m->W2b, m->W2Tb);
    return cudaDeviceSynchronize() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_mlp_get_weights(sdl_mlp* m, float* W1, float* b1, float* W2, float* b2) {
    if (!m) return SDL_ERR_ARG;
    DeviceGuard guard(m->ctx->device);
    if (cudaDeviceSynchronize() != cudaSuccess) return SDL_ERR_CUDA;
    const size_t H = m->H, Kp = m->Kp, Q = m->Q;
    if (W1) {
        std::vector<float> w1(H * Kp);
        if (cudaMemcpy(w1.data(), m->W1, H * Kp * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
            return SDL_ERR_CUDA;
        for (size_t h = 0; h < H; ++h)
            for (int e = 0; e < m->P; ++e) W1[h * m->P + e] = w1[h * Kp + e];
    }
    if (b1 && cudaMemcpy(b1, m->b1, H * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    if (W2 && cudaMemcpy(W2, m->W2, Q * H * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    if (b2 && cudaMemcpy(b2, m->b2, Q * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    return SDL_OK;
}

// Forward + loss + backward for one batch (gradients left in the network's
// gradient buffers); optionally the Adam step.  Y: B signals (layout of
// sdl_iterate), support: B x s OMP supports (the labels).
static int mlp_batch(sdl_mlp* m, const float* Y, const int32_t* support, int s, int B, bool update,
                     float lr, float* loss_out, cudaStream_t st) {
    sdl_ctx* c = m->ctx;
    const int H = m->H, Kp = m->Kp, Q = m->Q, Bm = m->Bmax;
    int rc;
    {
        Trace tr(c, kMlp, st);
        prep_batch_kernel<<<blocks_for(B, 32), 256, 0, st>>>(Y, B, m->P, Kp, m->Xb, m->XTb, Bm);
        if ((rc = tc_gemm(m->Xb, Kp, m->W1b, Kp, B, H, Kp, 1.f, m->b1, 1, nullptr, 0, 0, m->Hb, H,
                          m->HTb, Bm, m->pre, H, c->err, st)))
            return rc;
        if ((rc = tc_gemm(m->Hb, H, m->W2b, H, B, Q, H, 1.f, m->b2, 0, m->Z, Q, 0, nullptr, 0,
                          nullptr, 0, nullptr, 0, c->err, st)))
            return rc;
        const dim3 bce(blocks_for(B, 32), blocks_for(Q, kBceCols));
        bce_kernel<<<bce, 256, 0, st>>>(m->Z, Q, support, s, B, Q, 1.f / (float)B, m->dZb, Q, m->dZTb, Bm, m->lossp);
        // dW2 = dZ^T H ; dPre = (dZ W2) * GELU'(pre) ; dW1 = dPre^T X.  dW2 (few
        // tiles, a long K) runs beside dPre, which leaves it SMs, and the bias
        // gradients beside dW1; everything joins `st` before the update.
        auto step = [&](cudaError_t e) { return e == cudaSuccess; };
        if (!step(cudaEventRecord(c->side_ev[0], st)) || !step(cudaStreamWaitEvent(c->side, c->side_ev[0], 0))) return SDL_ERR_CUDA;
        rc = tc_gemm(m->dZTb, Bm, m->HTb, Bm, Q, H, B, 1.f, nullptr, 0, m->gW2, H, 0, nullptr, 0, nullptr, 0,
                     nullptr, 0, c->err, c->side);
        if (!rc)
            rc = tc_gemm(m->dZb, Q, m->W2Tb, Q, B, H, Q, 1.f, nullptr, 2, nullptr, 0, 0, nullptr, 0, m->dPreTb, Bm,
                         nullptr, 0, c->err, st, m->pre, H);
        if (!step(cudaEventRecord(c->side_ev[1], st)) || !step(cudaStreamWaitEvent(c->side, c->side_ev[1], 0))) rc = SDL_ERR_CUDA;
        if (!rc)
            row_sums_kernel<<<blocks_for(Q + H, 8) + 1, 256, 0, c->side>>>(m->dZTb, Q, m->gb2, m->dPreTb, H, m->gb1, Bm,
                                                                          B, m->lossp, B * (int)bce.y, 1.f / (float)B,
                                                                          loss_out);
        if (!rc)
            rc = tc_gemm(m->dPreTb, Bm, m->XTb, Bm, H, Kp, B, 1.f, nullptr, 0, m->gW1, Kp, 0, nullptr, 0, nullptr, 0,
                         nullptr, 0, c->err, st);
        // the side stream joins whatever happened above
        if (!step(cudaEventRecord(c->side_ev[2], c->side)) || !step(cudaStreamWaitEvent(st, c->side_ev[2], 0))) rc = SDL_ERR_CUDA;
        if (rc) return rc;
    }
    if (update) {
        Trace tr(c, kAdam, st);
        m->step += 1;
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float bc1 = 1.f - powf(b1, (float)m->step), bc2 = 1.f - powf(b2, (float)m->step);
        auto blocks = [](int rows, int cols) { return blocks_for(rows, 32) * blocks_for(cols, 32); };
        const AdamJobs jobs = {{{m->W2, m->mW2, m->vW2, m->gW2, Q, H, blocks(Q, H), m->W2b, m->W2Tb},
                                {m->W1, m->mW1, m->vW1, m->gW1, H, Kp, blocks(H, Kp), m->W1b, nullptr},
                                {m->b1, m->mb1, m->vb1, m->gb1, 1, H, blocks(1, H), nullptr, nullptr},
                                {m->b2, m->mb2, m->vb2, m->gb2, 1, Q, blocks(1, Q), nullptr, nullptr}}};
        int total = 0;
        for (const AdamJob& j : jobs.job) total += j.blocks;
        adam_kernel<<<total, 256, 0, st>>>(jobs, lr, b1, b2, eps, bc1, bc2);
    }
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_mlp_train_step(sdl_mlp* m, const float* Y, const int32_t* support, int s, int B, float lr,
                       float* loss_out, void* stream) {
    if (!m || !Y || !support || s < 1 || s > 32 || B < 8 || B % 8 || B > m->Bmax || !(lr > 0.f))
        return SDL_ERR_ARG;
    DeviceGuard guard(m->ctx->device);
    return mlp_batch(m, Y, support, s, B, true, lr, loss_out, (cudaStream_t)stream);
}

int sdl_mlp_gradients(sdl_mlp* m, const float* Y, const int32_t* support, int s, int B,
                      float* loss_out, float* gW1, float* gb1, float* gW2, float* gb2,
                      void* stream) {
    if (!m || !Y || !support || s < 1 || s > 32 || B < 8 || B % 8 || B > m->Bmax) return SDL_ERR_ARG;
    DeviceGuard guard(m->ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    int rc = mlp_batch(m, Y, support, s, B, false, 0.f, loss_out, st);
    if (rc) return rc;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SDL_ERR_CUDA;
    const size_t H = m->H, Kp = m->Kp, Q = m->Q;
    if (gW1) {
        std::vector<float> g(H * Kp);
        if (cudaMemcpy(g.data(), m->gW1, H * Kp * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
        for (size_t h = 0; h < H; ++h)
            for (int e = 0; e < m->P; ++e) gW1[h * m->P + e] = g[h * Kp + e];
    }
    if (gb1 && cudaMemcpy(gb1, m->gb1, H * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    if (gW2 && cudaMemcpy(gW2, m->gW2, Q * H * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    if (gb2 && cudaMemcpy(gb2, m->gb2, Q * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SDL_ERR_CUDA;
    return SDL_OK;
}

// Scores of `rows` (<= m->rows) signals.
static int infer_rows(sdl_mlp* m, const float* Y, int64_t rows, float* scores, cudaStream_t st) {
    sdl_ctx* c = m->ctx;
    const int H = m->H, Kp = m->Kp, Q = m->Q, B = (int)rows;
    bf16 *Xb = m->Xb, *Hb = m->Hb;
    if (m->P % 4 == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0)
        prep_rows_kernel<<<blocks_for(rows * 8, 256), 256, 0, st>>>(Y, B, m->P, Kp, Xb);
    else
        prep_input_kernel<<<blocks_for(rows * 32, 256), 256, 0, st>>>(Y, B, m->P, Kp, Xb);
    const int rc = tc_gemm(Xb, Kp, m->W1b, Kp, B, H, Kp, 1.f, m->b1, 1, nullptr, 0, 0, Hb, H, nullptr, 0, nullptr,
                           0, c->err, st);
    if (rc) return rc;
    return tc_gemm(Hb, H, m->W2b, H, B, Q, H, 1.f, m->b2, 0, scores, Q, 0, nullptr, 0, nullptr, 0, nullptr, 0,
                   c->err, st);
}

// Scores of N signals (device FP32 N x n1n2).
int sdl_mlp_forward(sdl_mlp* m, const float* Y, int64_t N, float* scores, void* stream) {
    if (!m || (N > 0 && (!Y || !scores)) || N < 0) return SDL_ERR_ARG;
    DeviceGuard guard(m->ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    sdl_ctx* c = m->ctx;
    const int64_t chunk = m->rows;
    Trace tr(c, kMlp, st);
    for (int64_t r0 = 0; r0 < N; r0 += chunk) {
        const int64_t B = std::min<int64_t>(chunk, N - r0);
        const int rc = infer_rows(m, Y + (size_t)r0 * m->P, B, scores + (size_t)r0 * m->Q, st);
        if (rc) return rc;
    }
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

}  // extern "C"

// ------------------------------------------------------------ learned coder
namespace {

// 2D-OMP on the shortlists and the fallback flags
int launch_shortlist(const float* Y, int p1, int p2, long long N, const float* D1, int n1, const float* D2, int n2,
                     int s, const int32_t* cand, int k1, int k2, int32_t* support, float* coef, int32_t* nnz,
                     float* res, int32_t* flag, int num_sms, cudaStream_t st) {
    PassArgs a{};
    a.Y = Y;
    a.p1 = p1;
    a.p2 = p2;
    a.N = N;
    a.D1 = D1;
    a.D2 = D2;
    a.n1 = n1;
    a.n2 = n2;
    a.s = s;
    a.support = support;
    a.coef = coef;
    a.nnz = nnz;
    a.res_energy = res;
    a.n_slots = 1;
    a.cand = cand;
    a.cand_k = k1;
    a.cand_ld = k2;
    a.flag = flag;
    return launch_code_group_short(a, st, num_sms);
}

}  // namespace

extern "C" int sdl_sparse_code_learned(sdl_ctx* c, sdl_mlp* m, const float* Y, int p1, int p2,
                                       int64_t N, const float* D1, int n1, const float* D2, int n2,
                                       int s_max, int k, int32_t* support, float* coef,
                                       int32_t* nnz, float* res_energy, int32_t* fallback,
                                       int32_t* n_fallback, float* guard_out, void* stream) {
    if (!c || !m || m->ctx != c || !Y || !D1 || !D2 || !support || !coef || !nnz || !fallback ||
        !n_fallback || N < 1 || N > 0x7fffffffLL)
        return SDL_ERR_ARG;
    if (m->P != p1 * p2 || m->Q != n1 * n2 || k < 1 || k > 32) return SDL_ERR_ARG;
    const bool shape_a = p1 == 12 && p2 == 12 && n1 == 24 && n2 == 24 && s_max == 6;
    const bool shape_b = p1 == 8 && p2 == 8 && n1 == 16 && n2 == 16 && s_max == 4;
    if (!shape_a && !shape_b) return SDL_ERR_UNSUPPORTED;
    DeviceGuard guard(c->device);
    cudaStream_t st = (cudaStream_t)stream;
    const int k2 = k, Q = m->Q;     // the shortlist only: the fallback test scans every pair
    // workspace: scores of one chunk, candidates, scan buffers, index list
    const long long chunk = std::min<long long>(N, m->rows);
    const int nblk = (int)((N + kScanBlock - 1) / kScanBlock);
    const long long m_s = std::min<long long>(N, std::max<long long>(kGuardMinSample, N / 16));
    const long long stride_s = N / m_s;
    const size_t need = sizeof(float) * (size_t)chunk * Q + sizeof(int32_t) * (size_t)N * k2 +
                        sizeof(int) * (nblk + 8) +
                        sizeof(int32_t) * (size_t)N + sizeof(int32_t) * (size_t)m_s +
                        sizeof(float) * (size_t)m_s + sizeof(float) * (size_t)N + sizeof(double2) * kGuardCtas +
                        10 * 256;
    if (need > c->cap_learn) {
        if (c->learn) cudaFree(c->learn);
        c->learn = nullptr;
        c->cap_learn = 0;
        if (cudaMalloc(&c->learn, need) != cudaSuccess) {
            cudaGetLastError();
            return SDL_ERR_WORKSPACE;
        }
        c->cap_learn = need;
    }
    int rc;
    char* p = c->learn;
    float* scores = carve<float>(p, (size_t)chunk * Q);
    int32_t* cand = carve<int32_t>(p, (size_t)N * k2);
    int* blockcnt = carve<int>(p, nblk + 8);
    int32_t* idx = carve<int32_t>(p, (size_t)N);
    int32_t* idx_s = carve<int32_t>(p, (size_t)m_s);
    float* plainE = carve<float>(p, (size_t)m_s);
    float* learnedE = res_energy ? res_energy : carve<float>(p, (size_t)N);
    int* cnt_s = carve<int>(p, 2);
    double2* part = carve<double2>(p, kGuardCtas);
    // 1. scores and shortlists, chunk by chunk
    for (int64_t r0 = 0; r0 < N; r0 += chunk) {
        const int B = (int)std::min<int64_t>(chunk, N - r0);
        {
            Trace tr(c, kMlp, st);
            if ((rc = infer_rows(m, Y + (size_t)r0 * p1 * p2, B, scores, st))) return rc;
        }
        Trace tr(c, kTopk, st);
        if (Q <= 256)
            topk_kernel<8><<<blocks_for((long long)B * 32, 256), 256, 0, st>>>(
                scores, Q, B, Q, k, k2, cand + (size_t)r0 * k2);
        else if (Q <= 576)
            topk_kernel<18><<<blocks_for((long long)B * 32, 256), 256, 0, st>>>(
                scores, Q, B, Q, k, k2, cand + (size_t)r0 * k2);
        else
            topk_kernel<32><<<blocks_for((long long)B * 32, 256), 256, 0, st>>>(
                scores, Q, B, Q, k, k2, cand + (size_t)r0 * k2);
    }
    // 2. 2D-OMP on the shortlists, with the fallback test
    {
        Trace tr(c, kShortlist, st);
        rc = launch_shortlist(Y, p1, p2, N, D1, n1, D2, n2, s_max, cand, k, k2, support, coef, nnz, learnedE, fallback,
                              c->num_sms, st);
        if (rc) return rc;
    }
    // 3. compact the flagged signals (fixed order) and re-code them with the full coder
    count_flags_kernel<<<nblk, kScanBlock, 0, st>>>(fallback, N, blockcnt);
    scan_counts_kernel<<<1, 32, 0, st>>>(blockcnt, nblk, n_fallback);
    write_index_kernel<<<nblk, kScanBlock, 0, st>>>(fallback, N, blockcnt, idx);
    PassArgs a{};
    a.Y = Y;
    a.p1 = p1;
    a.p2 = p2;
    a.N = N;
    a.D1 = D1;
    a.D2 = D2;
    a.n1 = n1;
    a.n2 = n2;
    a.s = s_max;
    a.support = support;
    a.coef = coef;
    a.nnz = nnz;
    a.res_energy = learnedE;
    a.n_slots = 1;
    a.err = c->err;
    a.idx = idx;
    a.idx_count = n_fallback;
    {
        Trace tr(c, kCode, st);
        rc = launch_code_group_fixed(a, false, st, c->num_sms);
        if (rc < 0) return rc;
    }
    // 4. the plain coder on the strided sample (residual energies only)
    sample_index_kernel<<<blocks_for(m_s, 256), 256, 0, st>>>(idx_s, (int)m_s, stride_s, cnt_s);
    PassArgs g = a;
    g.support = nullptr;
    g.coef = nullptr;
    g.nnz = nullptr;
    g.res_energy = plainE;
    g.idx = idx_s;
    g.idx_count = cnt_s;
    g.idx_compact = 1;
    {
        Trace tr(c, kCode, st);
        rc = launch_code_group_fixed(g, false, st, c->num_sms);
        if (rc < 0) return rc;
    }
    // 5. RMSE guard; when it trips, every signal is coded again by the plain coder
    guard_sums_kernel<<<kGuardCtas, kGuardThreads, 0, st>>>(plainE, learnedE, idx_s, (int)m_s, part);
    guard_kernel<<<1, 32, 0, st>>>(part, (int)m_s, N, p1 * p2, cnt_s + 1, n_fallback, guard_out);
    mark_all_kernel<<<std::max(1, std::min(blocks_for(N, 256), c->num_sms * 8)), 256, 0, st>>>(
        cnt_s + 1, N, idx, fallback);
    a.idx_count = cnt_s + 1;
    {
        Trace tr(c, kCode, st);
        rc = launch_code_group_fixed(a, false, st, c->num_sms);
    }
    return rc < 0 ? rc : SDL_OK;
}

// The two shortlist steps of sdl_sparse_code_learned on their own (before
// any fallback), so that each can be checked against a reference.
extern "C" int sdl_learned_shortlists(sdl_ctx* c, const float* scores, int64_t N, int Q, int k1,
                                      int k2, int32_t* cand, void* stream) {
    if (!c || N < 0 || N > 0x7fffffffLL || Q < 1 || Q > 1024 || k1 < 1 || k2 < k1 || k2 > Q)
        return SDL_ERR_ARG;
    if (N == 0) return SDL_OK;
    if (!scores || !cand) return SDL_ERR_ARG;
    DeviceGuard guard(c->device);
    cudaStream_t st = (cudaStream_t)stream;
    Trace tr(c, kTopk, st);
    const int blocks = blocks_for(N * 32, 256);
    if (Q <= 256)
        topk_kernel<8><<<blocks, 256, 0, st>>>(scores, Q, N, Q, k1, k2, cand);
    else if (Q <= 576)
        topk_kernel<18><<<blocks, 256, 0, st>>>(scores, Q, N, Q, k1, k2, cand);
    else
        topk_kernel<32><<<blocks, 256, 0, st>>>(scores, Q, N, Q, k1, k2, cand);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

extern "C" int sdl_sparse_code_shortlist(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N,
                                         const float* D1, int n1, const float* D2, int n2,
                                         int s_max, const int32_t* cand, int k1, int k2,
                                         int32_t* support, float* coef, int32_t* nnz,
                                         float* res_energy, int32_t* flag, void* stream) {
    if (!c || !D1 || !D2 || N < 0 || N > 0x7fffffffLL || k1 < 1 || k1 > 32 || k2 < k1)
        return SDL_ERR_ARG;
    const bool shape_a = p1 == 12 && p2 == 12 && n1 == 24 && n2 == 24 && s_max == 6;
    const bool shape_b = p1 == 8 && p2 == 8 && n1 == 16 && n2 == 16 && s_max == 4;
    if (!shape_a && !shape_b) return SDL_ERR_UNSUPPORTED;
    if (N == 0) return SDL_OK;
    if (!Y || !cand || !support || !coef || !nnz || !flag) return SDL_ERR_ARG;
    DeviceGuard guard(c->device);
    cudaStream_t st = (cudaStream_t)stream;
    Trace tr(c, kShortlist, st);
    return launch_shortlist(Y, p1, p2, N, D1, n1, D2, n2, s_max, cand, k1, k2, support, coef, nnz, res_energy, flag,
                            c->num_sms, st);
}
