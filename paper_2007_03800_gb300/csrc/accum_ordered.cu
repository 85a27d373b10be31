// Partial sums of a learning iteration from codes just written, in the order of
// the fused coders (omp_fast.cu): at the compiled shapes an iteration runs the
// lane-group coder (omp_group.cuh) and then this pass, instead of one warp per
// signal for both.
//
// The first dictionary's rounding decides near-tied picks of the second coding
// pass, so the sums keep the fused epilogue's exact order: warp w of CTA b takes
// signals b WPC + w, + grid WPC, ..., adds (pick, row) and (pick, pick) terms to its
// private accumulators, terms that meet in one entry in increasing pick order, and
// the warps are combined in warp order.  (The fused epilogue adds with
// shared-memory atomics in rounds of 32 lanes.  No document says in which order those
// of one warp reach one address; the boards measured take increasing lane order, as
// B here does, and the P half uses the same atomics, so that the two forms give the same
// bits there.)  Two warps share a sequence, one for B and
// one for P: a sequence is a serial chain and they are as many as the fused
// kernel had warps.  B: lane = row r of pick l = G t + g, the G picks of a
// round added one after the other; P: lane = (pick, pick), by the same atomics.
// z = (Y D2)[r, j_l] (D1 side) or (Y^T D1)[b, i_l] (D2 side) is formed for the
// picks alone, by the coders' FMA chain, a row of Y in registers.
// Measured: 200 000 x 12x12, 24x24 atoms, s = 6: 77 us per side, so that a learning
// pass takes 329 + 77 us against 546 fused; with atomics for both and one warp
// per sequence 101 and 145 us; terms told apart by rank, without atomics, 142 us.
#include <algorithm>

#include "sdl_internal.cuh"

namespace sdl {
namespace {

constexpr unsigned kFull = 0xffffffffu;
__host__ __device__ constexpr int up4(int x) { return (x + 3) & ~3; }

// WPC: warps per CTA, CPS: CTAs per SM of the fused kernel whose order is kept
template <int P1_, int P2_, int N1_, int N2_, int S_, int WPC_, int CPS_>
struct OrderedShape {
    static constexpr int P1 = P1_, P2 = P2_, N1 = N1_, N2 = N2_, S = S_, WPC = WPC_, CPS = CPS_, PP = P1 * P2;
    static_assert(N1 <= 64 && N2 <= 64, "packed pick fields");
    static_assert(P1 % 4 == 0 && P2 % 4 == 0 && S <= 32, "16-byte columns, one lane per pick");
};

template <class Sh, int SIDE>
struct OrderedLayout {
    static constexpr bool kD1 = SIDE == kSideD1;
    static constexpr int PC = kD1 ? Sh::P2 : Sh::P1, NC = kD1 ? Sh::N2 : Sh::N1;   // the other dictionary
    static constexpr int PA = kD1 ? Sh::P1 : Sh::P2, NA = kD1 ? Sh::N1 : Sh::N2;   // the updated one
    static constexpr int nf = NA * NA + PA * NA;
    static constexpr int AS = NA | 1;                 // row stride of the accumulators: rows in different banks
    static constexpr int nfa = up4(NA * AS + PA * AS);
    // strides of an odd number of 16-byte pieces: columns start in different banks
    static constexpr int odd4(int x) { return x / 4 % 2 ? x : x + 4; }
    static constexpr int DS = odd4(PC);
    static constexpr int YS = kD1 ? Sh::P1 : odd4(Sh::P1);
    static constexpr int dc = 0, g = dc + DS * NC, acc = g + up4(NC * NC), warp0 = acc + nfa * Sh::WPC;
    static constexpr int ybuf = up4(YS * Sh::P2), stride = 2 * ybuf, total = warp0 + Sh::WPC * stride;
};

template <class Sh, int SIDE>
__global__ void __launch_bounds__(Sh::WPC * 64, Sh::CPS) accum_ordered_kernel(PassArgs a) {
    using L = OrderedLayout<Sh, SIDE>;
    constexpr bool kD1 = L::kD1;
    constexpr int P1 = Sh::P1, N1 = Sh::N1, S = Sh::S, PP = Sh::PP, PA = L::PA, PC = L::PC, NA = L::NA, NC = L::NC;
    extern __shared__ __align__(16) float sm[];
    // two warps per sequence of signals: one adds to B, one to P
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = wid % Sh::WPC;
    const bool for_b = wid < Sh::WPC;
    float* dc = sm + L::dc;
    float* gs = sm + L::g;
    float* acc = sm + L::acc;
    float* wP = acc + w * L::nfa;
    float* wB = wP + NA * L::AS;
    float* ybuf = sm + L::warp0 + w * L::stride;
    const float* Dc = kD1 ? a.D2 : a.D1;
    for (int e = threadIdx.x; e < PC * NC; e += blockDim.x) dc[e / PC * L::DS + e % PC] = Dc[e];
    for (int e = threadIdx.x; e < L::nfa * Sh::WPC; e += blockDim.x) acc[e] = 0.f;
    __syncthreads();
    for (int e = threadIdx.x; e < NC * NC; e += blockDim.x) {   // one FMA chain, as the Gram kernels
        const int i = e / NC, j = e % NC;
        float v = 0.f;
        for (int c = 0; c < PC; ++c) v = fmaf(dc[i * L::DS + c], dc[j * L::DS + c], v);
        gs[e] = v;
    }
    __syncthreads();

    auto fetch = [&](long long k, int buf) {
        if (!for_b) return;
        const float* src = a.Y + (size_t)k * PP;
        float* dst = ybuf + buf * L::ybuf;
#pragma unroll
        for (int e0 = 0; e0 < PP; e0 += 128) {
            const int e = e0 + lane * 4;
            if (e < PP)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(dst + e / P1 * L::YS + e % P1)),
                             "l"(src + e)
                             : "memory");
        }
    };
    const long long step = (long long)gridDim.x * Sh::WPC;
    long long k = (long long)blockIdx.x * Sh::WPC + w;
    int qn = -1;
    float xn = 0.f;
    auto load = [&](long long kk, int buf) {   // codes to registers, Y to a buffer
        qn = -1;
        if (kk < a.N) {
            fetch(kk, buf);
            if (lane < S) {
                qn = a.in_support[(size_t)kk * S + lane];
                xn = a.in_coef[(size_t)kk * S + lane];
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(k, 0);
    constexpr int G = 32 / PA, T = (S + G - 1) / G;        // picks per round, rounds (B)
    const int g = lane / PA, r = lane % PA;                // lanes past G PA idle
    for (int it = 0; k < a.N; ++it, k += step) {
        const int q = qn;
        const float x = xn;
        const int cnt = __popc(__ballot_sync(kFull, q >= 0));   // the picks come first
        const int j = q >= 0 ? q / N1 : 0, i = q >= 0 ? q - j * N1 : 0;
        const int pk = kD1 ? i | j << 8 : j | i << 8;           // updated side | other side
        load(k + step, (it + 1) & 1);
        if (for_b) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            const float* Y = ybuf + (it & 1) * L::ybuf;
            float y[PC], v[T];
            int at[T];
            if constexpr (kD1) {
#pragma unroll
                for (int c = 0; c < PC; ++c) y[c] = Y[r + L::YS * c];
            } else {
#pragma unroll
                for (int c = 0; c < PC; c += 4) {
                    const float4 u = *reinterpret_cast<const float4*>(Y + L::YS * r + c);
                    y[c] = u.x; y[c + 1] = u.y; y[c + 2] = u.z; y[c + 3] = u.w;
                }
            }
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const int l = G * t + g;
                const int p = __shfl_sync(kFull, pk, l & 31);
                const float xl = __shfl_sync(kFull, x, l & 31);
                const float* d = dc + (p >> 8) * L::DS;
                float z = 0.f;
#pragma unroll
                for (int c = 0; c < PC; c += 4) {
                    const float4 u = *reinterpret_cast<const float4*>(d + c);
                    z = fmaf(y[c], u.x, z);
                    z = fmaf(y[c + 1], u.y, z);
                    z = fmaf(y[c + 2], u.z, z);
                    z = fmaf(y[c + 3], u.w, z);
                }
                v[t] = __fmul_rn(xl, z);
                at[t] = g < G && l < cnt ? r * L::AS + (p & 255) : -1;
            }
#pragma unroll
            for (int t = 0; t < T; ++t)
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    if (g == h && at[t] >= 0) wB[at[t]] = __fadd_rn(wB[at[t]], v[t]);
                    __syncwarp();
                }
        } else {
#pragma unroll
            for (int e0 = 0; e0 < S * S; e0 += 32) {
                const int e = e0 + lane, l = e / S, m = e % S;
                const int pl = __shfl_sync(kFull, pk, l & 31), pm = __shfl_sync(kFull, pk, m);
                const float xl = __shfl_sync(kFull, x, l & 31), xm = __shfl_sync(kFull, x, m);
                if (l < cnt && m < cnt)
                    atomicAdd(&wP[(pl & 255) * L::AS + (pm & 255)],
                              __fmul_rn(__fmul_rn(xl, xm), gs[(pl >> 8) * NC + (pm >> 8)]));
            }
        }
        __syncwarp();   // the buffers' next fetch
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    float* dst = a.part_f + (size_t)blockIdx.x * L::nf;
    for (int e = threadIdx.x; e < L::nf; e += blockDim.x) {
        const int at = e < NA * NA ? e / NA * L::AS + e % NA
                                   : NA * L::AS + (e - NA * NA) / NA * L::AS + (e - NA * NA) % NA;
        float v = 0.f;
        for (int ww = 0; ww < Sh::WPC; ++ww) v += acc[ww * L::nfa + at];
        dst[e] = v;
    }
}

template <class Sh, int SIDE>
int launch(const PassArgs& a, cudaStream_t st, int num_sms) {
    using L = OrderedLayout<Sh, SIDE>;
    constexpr size_t bytes = sizeof(float) * (size_t)L::total;
    static_assert(bytes * Sh::CPS + 1024 * Sh::CPS <= 228 * 1024, "shared memory");
    auto kern = accum_ordered_kernel<Sh, SIDE>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
        return SDL_ERR_CUDA;
    kern<<<ordered_slots(a, num_sms), Sh::WPC * 64, bytes, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

// the shapes whose fused kernels' default tilings these are
using O8x16s4 = OrderedShape<8, 8, 16, 16, 4, 8, 3>;
using O12x24s6 = OrderedShape<12, 12, 24, 24, 6, 8, 2>;
using O16x32s8 = OrderedShape<16, 16, 32, 32, 8, 6, 2>;

template <class F>
int with_shape(const PassArgs& a, F&& f) {
    auto is = [&](auto sh) {
        using Sh = decltype(sh);
        return a.p1 == Sh::P1 && a.p2 == Sh::P2 && a.n1 == Sh::N1 && a.n2 == Sh::N2 && a.s == Sh::S;
    };
    if (is(O8x16s4{})) return f(O8x16s4{});
    if (is(O12x24s6{})) return f(O12x24s6{});
    if (is(O16x32s8{})) return f(O16x32s8{});
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace

int ordered_slots(const PassArgs& a, int num_sms) {
    return with_shape(a, [&](auto sh) {
        using Sh = decltype(sh);
        const long long need = (a.N + Sh::WPC - 1) / Sh::WPC;
        return (int)std::max<long long>(1, std::min<long long>(need, (long long)num_sms * Sh::CPS));
    });
}

int launch_accumulate_ordered(const PassArgs& a, int side, cudaStream_t st, int num_sms) {
    return with_shape(a, [&](auto sh) {
        using Sh = decltype(sh);
        return side == kSideD1 ? launch<Sh, kSideD1>(a, st, num_sms) : launch<Sh, kSideD2>(a, st, num_sms);
    });
}

}  // namespace sdl
