// Error-driven coding: the signals already within the error target, found and
// given their empty code before the coder runs, and the list of the others.
//
// Most patches of a denoising call take no atom, and they come in clusters
// (smooth regions), so a coder that meets them one by one spends its time
// loading them at a coder's occupancy and its warps finish unevenly.  This pass
// reads the signals at the memory's rate and the coder's units are then full
// and evenly dealt.  Measured on the patches of a 512 x 512 image (13-19 % of them
// over the target): 8x8 84 -> 39 us, 12x12 158 -> 94, 16x16 397 -> 221; the
// three sizes as one batch 630-750 -> 360-385 by board.  The same scan inside the coder
// (32 signals at a time per warp, the others queued) took 90, 444 and 518 us.
#include <algorithm>
#include <type_traits>

#include "sdl_internal.cuh"

namespace sdl {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = 8;           // a block scans 8 x 4 ITS signals

// A group of 8 lanes sums one signal, 4 signals per warp and step, ITS (1, 2, 4 or
// 8) steps per warp: few signals spread over more blocks (up to 8000 of 32x32 values
// in blocks of 256 took 33 us, most of it one warp's chain of loads).  The partial
// sums and their combining tree are the coders' (32 strided chains, then xor
// 16, 8, 4, 2, 1), so the comparison with the target comes out the same: lane j
// holds chains 4j .. 4j+3.  VEC: 16-byte loads (p1 p2 a multiple of 4, Y
// 16-byte aligned).
// `word` starts at zero: blocks that have come in the upper half, signals listed in
// the lower.  The last block to come moves the total to *count and clears the
// word for the next scan, which costs no launch of its own (a memset costs the host
// 3 us).  A scan of 8 steps per warp, whose time the host does not feel, adds to a cleared
// *count instead, and blocks that list nothing skip the atomic (three scans of 250 000
// signals: 363 us with their coders, 381 through the word).
template <bool VEC, int ITS>
__global__ void __launch_bounds__(kWarps * 32)
    energy_scan_kernel(const float* __restrict__ Y, int pp, long long N, float eps2, int s,
                       int32_t* __restrict__ support, float* __restrict__ coef, int32_t* __restrict__ nnz,
                       float* __restrict__ res_energy, int32_t* __restrict__ list, int* __restrict__ count,
                       unsigned long long* __restrict__ word) {
    __shared__ int wcount[kWarps], base_s;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane >> 3, j = lane & 7;
    const long long first = ((long long)blockIdx.x * kWarps + w) * (4 * ITS);
    const int m = (int)max(0LL, min(4LL * ITS, N - first));
    float mine = 0.f;
#pragma unroll 2
    for (int it = 0; it < ITS; ++it) {
        const int i = it * 4 + grp;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (i < m) {
            const float* src = Y + (size_t)(first + i) * pp;
            if constexpr (VEC) {
#pragma unroll 4
                for (int e = 4 * j; e < pp; e += 32) {
                    const float4 y = __ldg(reinterpret_cast<const float4*>(src + e));
                    v[0] = fmaf(y.x, y.x, v[0]);
                    v[1] = fmaf(y.y, y.y, v[1]);
                    v[2] = fmaf(y.z, y.z, v[2]);
                    v[3] = fmaf(y.w, y.w, v[3]);
                }
            } else {
                for (int e = 4 * j; e < pp; e += 32)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (e + c < pp) {
                            const float y = __ldg(src + e + c);
                            v[c] = fmaf(y, y, v[c]);
                        }
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(kFull, v[c], o);
        const float ss = (v[0] + v[2]) + (v[1] + v[3]);
        const float mv = __shfl_sync(kFull, ss, (lane & 3) * 8);
        if ((lane >> 2) == it) mine = mv;
    }
    // lane i holds signal i of the warp
    const bool have = lane < m;
    const bool done = have && isfinite(mine) && mine <= eps2;
    const unsigned dm = __ballot_sync(kFull, done), todo = __ballot_sync(kFull, have && !done);
    if (done) {
        if (nnz) nnz[first + lane] = 0;
        if (res_energy) res_energy[first + lane] = mine;
    }
    if (support && dm) {
        const unsigned inv_s = (65536u + s - 1) / s;   // e / s for e < 1024
        for (int e = lane; e < 4 * ITS * s; e += 32)
            if ((dm >> ((unsigned)e * inv_s >> 16)) & 1u) {
                support[(size_t)first * s + e] = -1;
                coef[(size_t)first * s + e] = 0.f;
            }
    }
    if (lane == 0) wcount[w] = __popc(todo);
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int v = 0; v < kWarps; ++v) {
            const int c = wcount[v];
            wcount[v] = tot;
            tot += c;
        }
        // the list's order does not matter
        if constexpr (ITS == 8) {
            base_s = tot ? atomicAdd(count, tot) : 0;
        } else {
            const unsigned long long old = atomicAdd(word, (1ULL << 32) | (unsigned)tot);
            base_s = (int)(unsigned)old;
            if ((unsigned)(old >> 32) + 1 == gridDim.x) {   // every other block has come
                *count = base_s + tot;
                *word = 0;
            }
        }
    }
    __syncthreads();
    if (have && !done) list[base_s + wcount[w] + __popc(todo & ((1u << lane) - 1u))] = (int32_t)(first + lane);
}

}  // namespace

// The list fits the scratch in at most kSegments parts (4 floats hold the count).
constexpr long long kSegments = 8;
// Calls up to both sizes are coded without a scan: the coder stops at a signal
// within the target by itself, and a second launch costs more than it saves.  Coder
// alone | scan and coder | one warp per signal, us per call, most and fewest signals
// over the target: 8000 x 16x16, 32x32 pairs 47 | 59 | 64 and 18 | 24 | 22; 16 000 80 | 92 |
// 115 and 27 | 25 | 22; 16 000 x 12x12 37 | 47 | 53 and 18 | 25 | 22, 64 000 111 | 123 | 163 and
// 41 | 25 | 27; 64 000 x 4x4 31 | 41 | 82 and 21 | 25 | 22 (the first of each pair's lines
// is within, the second past; scans then with a memset of the count, 3 us more).
constexpr long long kUnscannedSignals = 32768, kUnscannedFloats = 1 << 21;
bool unscanned(const PassArgs& a) {
    return !(a.eps2 > 0.f) || (a.N <= kUnscannedSignals && a.N * a.p1 * a.p2 <= kUnscannedFloats);
}
long long list_capacity(size_t ws_n) {
    return ws_n < 64 ? 0 : std::min<long long>((long long)(ws_n - 4) & ~3LL, 1LL << 30);
}

// Code-only passes that the lane-group coder takes, given ws_n floats of scratch
// for the list of an error-driven call.  (Every accepted signal size fits a CTA's
// shared memory in each of its tiles: the largest, 64x16 signals with s = 32 on
// the 32 x 128 tile, need 126 KB for one team.)
bool code_lanes_take(const PassArgs& a, size_t ws_n) {
    // correlations from the tensor cores, a pinned tiling and wider dictionaries
    // have coders of their own
    if (a.c0ext || a.tiling_forced || a.n1 > 32 || a.n2 > 128) return false;
    // the scan's sums are those of the coders with 32 chains
    if (!(a.eps2 > 0.f)) return true;
    return !a.idx && a.n2 <= 32 && (unscanned(a) || a.N <= kSegments * list_capacity(ws_n));
}

// ws: ws_n floats of scratch (null: none), scan_word: a device word that is zero
// between scans.  SDL_ERR_UNSUPPORTED, with nothing launched, for a call that it
// does not take.
int launch_code_lanes(const PassArgs& a, float* ws, size_t ws_n, unsigned long long* scan_word, cudaStream_t st,
                      int num_sms) {
    if (!code_lanes_take(a, ws && scan_word ? ws_n : 0)) return SDL_ERR_UNSUPPORTED;
    const bool aligned = (reinterpret_cast<uintptr_t>(a.Y) & 15u) == 0;
    auto code = [&](const PassArgs& q) -> int {
        // the compiled shapes keep their tilings' arithmetic, which they have
        // only with aligned signals
        const int r = aligned ? launch_code_group_fixed(q, false, st, num_sms) : SDL_ERR_UNSUPPORTED;
        return r != SDL_ERR_UNSUPPORTED ? r : launch_code_group_any(q, st, num_sms);
    };
    if (unscanned(a)) return code(a);
    const long long cap = list_capacity(ws_n);
    const int pp = a.p1 * a.p2;
    int* count = reinterpret_cast<int*>(ws);
    int32_t* list = reinterpret_cast<int32_t*>(ws + 4);
    for (long long k0 = 0; k0 < a.N; k0 += cap) {
        PassArgs q = a;
        q.N = std::min(cap, a.N - k0);
        q.Y = a.Y + (size_t)k0 * pp;
        q.support = a.support ? a.support + (size_t)k0 * a.s : nullptr;
        q.coef = a.coef ? a.coef + (size_t)k0 * a.s : nullptr;
        q.nnz = a.nnz ? a.nnz + k0 : nullptr;
        q.res_energy = a.res_energy ? a.res_energy + k0 : nullptr;
        // four blocks per SM before a warp takes more signals
        int its = 8;
        while (its > 1 && q.N < (long long)kWarps * 4 * its * 4 * num_sms) its /= 2;
        if (its == 8 && cudaMemsetAsync(count, 0, sizeof(int), st) != cudaSuccess) return SDL_ERR_CUDA;
        const unsigned blocks = (unsigned)((q.N + kWarps * 4 * its - 1) / (kWarps * 4 * its));
        auto scan = [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            return aligned && pp % 4 == 0 ? energy_scan_kernel<true, I> : energy_scan_kernel<false, I>;
        };
        auto kern = its == 8   ? scan(std::integral_constant<int, 8>{})
                    : its == 4 ? scan(std::integral_constant<int, 4>{})
                    : its == 2 ? scan(std::integral_constant<int, 2>{})
                               : scan(std::integral_constant<int, 1>{});
        kern<<<blocks, kWarps * 32, 0, st>>>(q.Y, pp, q.N, a.eps2, a.s, q.support, q.coef, q.nnz, q.res_energy,
                                             list, count, scan_word);
        if (cudaGetLastError() != cudaSuccess) return SDL_ERR_CUDA;
        q.idx = list;
        q.idx_count = count;
        const int r = code(q);
        if (r != SDL_OK) return r == SDL_ERR_UNSUPPORTED ? SDL_ERR_CUDA : r;   // the scan has run
    }
    return SDL_OK;
}

}  // namespace sdl
