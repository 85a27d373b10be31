// Three-mode coding (no partial sums) with 16 lanes per signal, two signals per
// warp, at the shapes of tmod3_fast.cu and in its arithmetic: every entry of the
// contractions, the scores, the Cholesky rows and the solves is the same chain,
// so the codes are bit-identical.
//
// As in omp_group.cuh, the pass is bound by warp instructions and shared-memory
// bandwidth: the scalar work of a greedy step is issued once for two signals, a
// lane's block is all n1 rows of RJ x RL columns (j, l), so that one row of G1
// feeds RJ RL columns, the maximum goes down the columns with three-input |max|,
// and only the Cholesky row is unrolled per step.  50 000 cubes of 4x4x16, 8x8x16
// atoms, s = 8: 353 us with one warp per signal, 230 us here (2645 instead of 4264
// warp instructions per signal).
#include "omp_group.cuh"

namespace sdl {
namespace {

using group::cp16;
using group::cp_wait;
using group::kFull;
using group::ld;
using group::max3abs;
using group::rank1;
using group::Rec;
using group::st;
using group::up4;

template <int P1_, int P2_, int P3_, int N1_, int N2_, int N3_, int S_, int RJ_, int RL_>
struct Shape3G {
    static constexpr int P1 = P1_, P2 = P2_, P3 = P3_, N1 = N1_, N2 = N2_, N3 = N3_, S = S_, RJ = RJ_, RL = RL_;
    static constexpr int LJ = N2 / RJ, LL = N3 / RL, C = RJ * RL, E = N1 * C;
    static constexpr int PP = P1 * P2 * P3, P12 = P1 * P2, BL = P2 * N3;
    static constexpr int WARPS = 8;
    static constexpr int EP = (E / 4) % 2 ? E : E + 4;       // lane stride of the C0 blocks: odd x 4
    static_assert(LJ * LL == 16 && LJ * RJ == N2 && LL * RL == N3, "16 lanes tile the columns");
    static_assert(N1 == 8 && P12 == 16 && N3 % 4 == 0 && S <= 8 && PP % 64 == 0, "stage tilings");
    // T1: 4 (a, b) x TL l per lane; T2: 8 rows x TB (b, l) columns per lane
    static constexpr int TL = N3 / 4, TB = BL / 16;
    static_assert(TB % 2 == 0, "T2 columns");
    // shared memory (floats)
    static constexpr int d1 = 0, d2 = d1 + P1 * N1, d3 = d2 + P2 * N2, g1 = d3 + P3 * N3, g2 = g1 + N1 * N1,
                         g3 = g2 + N2 * N2, warp0 = g3 + N3 * N3;
    // per signal: Y | T1 (P1 x BL), T2 (BL x N1), then the C0 blocks | ...
    static constexpr int y = 0, t1 = PP, t2 = t1 + P1 * BL, c0 = t1;
    static constexpr int body = P1 * BL + BL * N1 > 16 * EP ? P1 * BL + BL * N1 : 16 * EP;
    static constexpr int col = c0 + body, rec = col + 8, lf = rec + up4(2 * S), iv = lf + up4(S * (S - 1) / 2),
                         yv = iv + up4(S), raw = yv + up4(S);
    static constexpr int sig = raw + (raw % 32 <= 8 ? 8 - raw % 32 : 40 - raw % 32);   // 8 banks apart
    static constexpr int total = warp0 + WARPS * 2 * sig;
    static_assert(raw % 4 == 0, "16-byte regions");
};

template <class Sh>
__global__ void __launch_bounds__(Sh::WARPS * 32, 2)
    code3_group_kernel(const float* __restrict__ Y, long long N, const float* __restrict__ D1,
                       const float* __restrict__ D2, const float* __restrict__ D3, int32_t* __restrict__ support,
                       float* __restrict__ coef, int32_t* __restrict__ nnz, float* __restrict__ res_energy,
                       int* err) {
    constexpr int P1 = Sh::P1, P2 = Sh::P2, P3 = Sh::P3, N1 = Sh::N1, N2 = Sh::N2, N3 = Sh::N3, S = Sh::S;
    constexpr int RJ = Sh::RJ, RL = Sh::RL, C = Sh::C, E = Sh::E, PP = Sh::PP, BL = Sh::BL, LJ = Sh::LJ;
    extern __shared__ __align__(16) float sm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, gl = lane & 15;
    const int lj = gl % LJ, ll = gl / LJ, j0 = lj * RJ, l0 = ll * RL;
    float* d1 = sm + Sh::d1;   // rows a
    float* d2 = sm + Sh::d2;   // rows b
    float* d3 = sm + Sh::d3;   // rows c
    float* g1 = sm + Sh::g1;
    float* g2 = sm + Sh::g2;
    float* g3 = sm + Sh::g3;
    float* sb = sm + Sh::warp0 + (2 * w + half) * Sh::sig;
    float* Ys = sb + Sh::y;
    float* T1 = sb + Sh::t1;   // T1[a BL + b + P2 l]
    float* T2 = sb + Sh::t2;   // T2[i + N1 (b + P2 l)]
    float* C0s = sb + Sh::c0;
    float* myc0 = C0s + gl * Sh::EP;
    float* col = sb + Sh::col;
    Rec* rec = reinterpret_cast<Rec*>(sb + Sh::rec);
    float* lf = sb + Sh::lf;
    float* iv = sb + Sh::iv;
    float* yv = sb + Sh::yv;

    for (int e = threadIdx.x; e < P1 * N1; e += blockDim.x) d1[e] = D1[e / N1 + P1 * (e % N1)];
    for (int e = threadIdx.x; e < P2 * N2; e += blockDim.x) d2[e] = D2[e / N2 + P2 * (e % N2)];
    for (int e = threadIdx.x; e < P3 * N3; e += blockDim.x) d3[e] = D3[e / N3 + P3 * (e % N3)];
    if (gl < S) rec[gl] = Rec{0.f, 0u};   // a finished signal's lanes run along on valid records
    __syncthreads();
    auto gram_of = [&](float* g, const float* d, int p, int n) {   // as the Gram kernels form it
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const int i = e / n, j = e % n;
            float v = 0.f;
            for (int r = 0; r < p; ++r) v = fmaf(d[r * n + i], d[r * n + j], v);
            g[e] = v;
        }
    };
    gram_of(g1, d1, P1, N1);
    gram_of(g2, d2, P2, N2);
    gram_of(g3, d3, P3, N3);
    __syncthreads();

    const long long units = (N + 1) / 2, step = (long long)gridDim.x * Sh::WARPS;
    auto fetch = [&](long long k) {
        const float* src = Y + (size_t)k * PP;
#pragma unroll
        for (int e = gl * 4; e < PP; e += 64) cp16(Ys + e, src + e);
    };
    long long u = (long long)w * gridDim.x + blockIdx.x;
    if (u < units && 2 * u + half < N) fetch(2 * u + half);
    for (; u < units; u += step) {
        const long long k = 2 * u + half;
        const bool act = k < N;
        cp_wait();
        __syncwarp();
        // ||Y||^2: the one-warp coder's lane v takes elements 4v .. 4v + 3 (or 2v, 2v + 1)
        // of every 128 (64); here a lane stands for v = gl and gl + 16
        float ss = 0.f;
        if (act) {
            constexpr int V = PP >= 128 ? 4 : 2;
            float part[2] = {0.f, 0.f};
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < PP; e += 32 * V)
#pragma unroll
                    for (int c = 0; c < V; ++c) {
                        const float v = Ys[e + V * (gl + 16 * h) + c];
                        part[h] = fmaf(v, v, part[h]);
                    }
            ss = part[0] + part[1];
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(kFull, ss, o);
        const bool finite = act && isfinite(ss);
        bool go = finite;

        // ---- T1 = Y x_3 D3^T: 4 (a, b) x TL l per lane
        {
            const int ab = (gl & 3) * 4, lt = (gl >> 2) * Sh::TL;
            float t[4 * Sh::TL];
#pragma unroll
            for (int e = 0; e < 4 * Sh::TL; ++e) t[e] = 0.f;
#pragma unroll
            for (int c = 0; c < P3; ++c) {
                float x[4], v[Sh::TL];
                ld<4>(x, Ys + ab + Sh::P12 * c);
                if constexpr (Sh::TL == 4) ld<4>(v, d3 + c * N3 + lt);
                else group::ld2<Sh::TL>(v, d3 + c * N3 + lt);
                rank1<4, Sh::TL>(t, x, v);
            }
#pragma unroll
            for (int l = 0; l < Sh::TL; ++l)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int a = (ab + r) % P1, b = (ab + r) / P1;
                    T1[a * BL + b + P2 * (lt + l)] = t[l * 4 + r];
                }
        }
        __syncwarp();
        // Y is consumed: fetch the next unit's signals
        if (u + step < units && 2 * (u + step) + half < N) fetch(2 * (u + step) + half);
        // ---- T2 = T1 x_1 D1^T: N1 rows x TB (b, l) columns per lane
        {
            const int b0 = gl * Sh::TB;
            float t[N1 * Sh::TB];
#pragma unroll
            for (int e = 0; e < N1 * Sh::TB; ++e) t[e] = 0.f;
#pragma unroll
            for (int a = 0; a < P1; ++a) {
                float x[N1], v[Sh::TB];
                ld<N1>(x, d1 + a * N1);
                if constexpr (Sh::TB % 4 == 0) ld<Sh::TB>(v, T1 + a * BL + b0);
                else group::ld2<Sh::TB>(v, T1 + a * BL + b0);
                rank1<N1, Sh::TB>(t, x, v);
            }
#pragma unroll
            for (int c = 0; c < Sh::TB; ++c) {
                float v[N1];
#pragma unroll
                for (int r = 0; r < N1; ++r) v[r] = t[c * N1 + r];
                st<N1>(T2 + (b0 + c) * N1, v);
            }
        }
        __syncwarp();
        // ---- C0 = T2 x_2 D2^T on the lane's columns c = rl RJ + rj
        float sc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) sc[e] = 0.f;
#pragma unroll
        for (int b = 0; b < P2; ++b) {
            float v[RJ];
            ld<RJ>(v, d2 + b * N2 + j0);
#pragma unroll
            for (int rl = 0; rl < RL; ++rl) {
                float x[N1];
                ld<N1>(x, T2 + N1 * (b + P2 * (l0 + rl)));
#pragma unroll
                for (int rj = 0; rj < RJ; ++rj)
#pragma unroll
                    for (int r = 0; r < N1; r += 2) {
                        float* s2 = sc + (rl * RJ + rj) * N1 + r;
                        group::ffma2(s2[0], s2[1], x[r], x[r + 1], v[rj], v[rj]);
                    }
            }
        }
        __syncwarp();   // T1 and T2 are read: their place takes the C0 blocks
        st<E>(myc0, sc);
        __syncwarp();

        int cnt = 0;
        float E2 = ss;
#pragma unroll 1
        for (int t = 0; t < S; ++t) {
            if (!__any_sync(kFull, go)) break;
            if (t > 0) {
                ld<E>(sc, myc0);
                Rec next = rec[0];   // one ahead of the loop
#pragma unroll 1
                for (int m = 0; m < t; ++m) {
                    const Rec q = next;
                    if (m + 1 < S) next = rec[m + 1];
                    float x[N1], v[RJ], wl[RL], vw[C];
                    ld<N1>(x, g1 + (q.o & 255u) * N1);
                    ld<RJ>(v, g2 + ((q.o >> 8) & 255u) * N2 + j0);
                    if constexpr (RL == 2) group::ld2<2>(wl, g3 + (q.o >> 16) * N3 + l0);
                    else wl[0] = g3[(q.o >> 16) * N3 + l0];
#pragma unroll
                    for (int rl = 0; rl < RL; ++rl) {
                        const float wx = -q.x * wl[rl];
#pragma unroll
                        for (int rj = 0; rj < RJ; ++rj) vw[rl * RJ + rj] = v[rj] * wx;
                    }
                    rank1<N1, C>(sc, x, vw);
                }
            }
            // the lane's largest |score| and its first column
            float best = 0.f;
            int bc = 0;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                float m = 0.f;
#pragma unroll
                for (int r = 0; r < N1; r += 2) m = max3abs(m, sc[c * N1 + r], sc[c * N1 + r + 1]);
                if (m > best) { best = m; bc = c; }
            }
            // the signal's largest, its smallest column j + N2 l
            float M = best;
            int key = j0 + bc % RJ + N2 * (l0 + bc / RJ);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                const float mo = __shfl_xor_sync(kFull, M, o);
                const int ko = __shfl_xor_sync(kFull, key, o);
                if (mo > M || (mo == M && ko < key)) { M = mo; key = ko; }
            }
            const bool pick = go && M != 0.f;
            const int jt = key % N2, lt = key / N2;
            const int owner = jt / RJ + LJ * (lt / RL), oc = (lt % RL) * RJ + jt % RJ;
            if (gl == owner) {
#pragma unroll
                for (int c = 0; c < C; ++c)
                    if (bc == c) {
                        float v[N1];
#pragma unroll
                        for (int r = 0; r < N1; ++r) v[r] = sc[c * N1 + r];
                        st<N1>(col, v);
                    }
            }
            __syncwarp();
            const unsigned bal = __ballot_sync(kFull, gl < N1 && fabsf(col[gl & (N1 - 1)]) == M);
            const unsigned rows = (bal >> (16 * half)) & 0xffffu;
            const int it = rows ? __ffs(rows) - 1 : 0;
            float* cq = C0s + owner * Sh::EP + oc * N1 + it;
            const float b = *cq;
            const Rec pk{0.f, (unsigned)it | (unsigned)jt << 8 | (unsigned)lt << 16};
            auto gram = [&](const Rec& r) {
                return g1[it * N1 + (r.o & 255u)] * g2[jt * N2 + ((r.o >> 8) & 255u)] * g3[lt * N3 + (r.o >> 16)];
            };
            const float Att = gram(pk);
            __syncwarp();
            const bool wr = gl == 0;
            if (wr && pick) *cq = __int_as_float(0x7fc00000);   // mask the pick
            bool ok = false;
            auto stepf = [&](auto tc) {
                ok = group::chol_step<decltype(tc)::value, true>(pick, wr, rec, lf, iv, yv, gram, Att, b, pk, E2);
            };
            switch (t) {
                case 0: stepf(std::integral_constant<int, 0>{}); break;
                case 1: if constexpr (S > 1) stepf(std::integral_constant<int, 1>{}); break;
                case 2: if constexpr (S > 2) stepf(std::integral_constant<int, 2>{}); break;
                case 3: if constexpr (S > 3) stepf(std::integral_constant<int, 3>{}); break;
                case 4: if constexpr (S > 4) stepf(std::integral_constant<int, 4>{}); break;
                case 5: if constexpr (S > 5) stepf(std::integral_constant<int, 5>{}); break;
                case 6: if constexpr (S > 6) stepf(std::integral_constant<int, 6>{}); break;
                default: if constexpr (S > 7) stepf(std::integral_constant<int, 7>{}); break;
            }
            if (ok) cnt = t + 1;
            go = ok;
            __syncwarp();   // the step's state and the masked entry are visible
        }
        if (act) {
            if (gl < S) {
                const Rec q = rec[gl];
                const int qi = (int)(q.o & 255u) + N1 * ((int)((q.o >> 8) & 255u) + N2 * (int)(q.o >> 16));
                support[(size_t)k * S + gl] = gl < cnt ? qi : -1;
                coef[(size_t)k * S + gl] = gl < cnt ? q.x : 0.f;
            }
            if (gl == 0) {
                nnz[k] = cnt;
                if (res_energy) res_energy[k] = finite ? fmaxf(E2, 0.f) : __int_as_float(0x7fc00000);
                if (!finite) record_error(err, SDL_ERR_NONFINITE);
            }
        }
        __syncwarp();   // records are read before the next unit writes them
    }
}

template <class Sh>
int run(const float* Y, long long N, const float* D1, const float* D2, const float* D3, int32_t* support, float* coef,
        int32_t* nnz, float* res, int* err, int num_sms, cudaStream_t st) {
    constexpr size_t bytes = sizeof(float) * (size_t)Sh::total;
    static_assert(2 * (bytes + 1024) <= 228 * 1024, "two CTAs per SM");
    auto kern = code3_group_kernel<Sh>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
        return SDL_ERR_CUDA;
    const long long grid = std::max<long long>(1, std::min<long long>((N + 1) / 2, 2LL * num_sms));
    kern<<<(int)grid, Sh::WARPS * 32, bytes, st>>>(Y, N, D1, D2, D3, support, coef, nnz, res, err);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

using G3cube = Shape3G<4, 4, 16, 8, 8, 16, 8, 4, 2>;
using G3small = Shape3G<4, 4, 4, 8, 8, 8, 4, 4, 1>;

// the compiled shape of these sizes, if any
template <class F>
int with_shape(int p1, int p2, int p3, int n1, int n2, int n3, int s, F&& f) {
    auto is = [&](auto sh) {
        using Sh = decltype(sh);
        return p1 == Sh::P1 && p2 == Sh::P2 && p3 == Sh::P3 && n1 == Sh::N1 && n2 == Sh::N2 && n3 == Sh::N3 &&
               s == Sh::S;
    };
    if (is(G3cube{})) return f(G3cube{});
    if (is(G3small{})) return f(G3small{});
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace

bool code3_group_takes(const float* Y, int p1, int p2, int p3, int n1, int n2, int n3, int s) {
    return (reinterpret_cast<uintptr_t>(Y) & 15u) == 0 &&
           with_shape(p1, p2, p3, n1, n2, n3, s, [](auto) { return (int)SDL_OK; }) == SDL_OK;
}

int launch_code3_group(const float* Y, int p1, int p2, int p3, int n1, int n2, int n3, long long N, const float* D1,
                       const float* D2, const float* D3, int s, int32_t* support, float* coef, int32_t* nnz,
                       float* res, int* err, int num_sms, cudaStream_t st) {
    if ((reinterpret_cast<uintptr_t>(Y) & 15u) != 0) return SDL_ERR_UNSUPPORTED;
    return with_shape(p1, p2, p3, n1, n2, n3, s, [&](auto sh) {
        return run<decltype(sh)>(Y, N, D1, D2, D3, support, coef, nnz, res, err, num_sms, st);
    });
}

}  // namespace sdl
