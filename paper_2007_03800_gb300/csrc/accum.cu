// Partial sums of a dictionary update from given codes, n <= 32 atoms and p <= 32
// rows on the side that is updated, without atomics.
//
// Naming for either side (r, i: rows and atoms of the dictionary being updated;
// c, j: of the other one): B[r, i_l] += x_l z_l[r] with z_l = sum_c y[r, c] D[c, j_l],
// and P[i_l, i_m] += x_l x_m G[j_l, j_m].
//
// One warp per signal.  Lane = row r for the projections z_l (a row of Y in
// registers, PA lanes per pick, 32 / PA picks at once); then lane = atom i for
// the sums: a lane adds the picks of its own atom, so no two lanes touch one
// entry.  B stays in registers (PA per lane), P in a warp-private n x n block of
// shared memory, added up over the warps in a fixed order at the end: the
// sums are deterministic.  Bound by issue (61 % of the slots, 750 warp
// instructions per signal): 100 000 signals of 16x16, 32x32 atoms, s = 8 take 92 us
// (D1) and 90 us (D2), against 287 and 430 us with one block-wide accumulator
// under shared-memory atomics and the residual energy always formed (206 and 199 with it).
// Registers for two 12-warp CTAs per SM; the Gram matrix is formed here, so an
// update needs no launch for it.
#include <algorithm>
#include <type_traits>

#include "sdl_internal.cuh"

namespace sdl {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = 12;
constexpr int kMinCtas = 2;
constexpr int kChunk = 16;          // contraction terms held in registers at a time

__host__ __device__ constexpr int up4(int x) { return (x + 3) & ~3; }

struct AccumLayout {
    int ys;        // stride of a staged signal's columns (a)
    int dc, ds, g, gs, warp0;
    int y, z, pick, p, ps, stride, total;
    __host__ __device__ AccumLayout(int p1, int p2, int pa, int pc, int na, int nc, int s, int PA, int side, int warps) {
        // side D2 reads a column as 16-byte pieces, one column per lane: a stride
        // of an odd number of pieces spreads the lanes over the banks
        ys = side == kSideD1 ? p1 : up4(p1) + (up4(p1) / 4 % 2 ? 0 : 4);
        // rows of D and of G: an odd number of 16-byte pieces, so that eight lanes on
        // eight rows hit distinct banks (with up4(64) = 64 all 32 lanes of the Gram
        // product met in one: 16x64 signals, 32x128 atoms, 92 us per CTA)
        ds = up4(pc) + (up4(pc) / 4 % 2 ? 0 : 4);
        gs = nc | 1;
        dc = 0;                              // D[c, j] at j * ds + c, zero-padded
        g = dc + up4(ds * nc);               // G
        warp0 = g + up4(gs * nc);
        y = 0;
        z = y + up4(ys * up4(p2));           // columns past p2 stay zero
        const int body = z + up4(s * PA);
        const int dump = up4(na * PA);       // B of the warp, at the end
        pick = body > dump ? body : dump;
        ps = na | 1;
        p = pick + 4 * s;
        stride = p + up4(na * ps);
        total = warp0 + warps * stride;
        (void)pa;
    }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

struct alignas(16) AccumPick {
    float x;
    int i, j, g;   // atoms of the updated and of the other side, offset of the latter's row of G
};

// ENERGY: the residual energy too (a kernel of its own, for its registers)
template <int PA, int SIDE, bool ENERGY>
__global__ void __launch_bounds__(kWarps * 32, kMinCtas) accum_lane_kernel(PassArgs a) {
    extern __shared__ __align__(16) float sm[];
    constexpr bool kD1 = SIDE == kSideD1;
    constexpr int LG = 32 / PA;              // picks projected at once
    const int p1 = a.p1, p2 = a.p2, pp = p1 * p2, s = a.s;
    const int pa = kD1 ? p1 : p2, pc = kD1 ? p2 : p1;
    const int na = kD1 ? a.n1 : a.n2, nc = kD1 ? a.n2 : a.n1;
    const float* Dc = kD1 ? a.D2 : a.D1;
    const float* Da = kD1 ? a.D1 : a.D2;
    const int warps = blockDim.x >> 5;
    const AccumLayout L(p1, p2, pa, pc, na, nc, s, PA, SIDE, warps);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* ds = sm + L.dc;
    float* gs = sm + L.g;
    float* wb = sm + L.warp0 + w * L.stride;
    float* Ys = wb + L.y;
    float* zs = wb + L.z;
    AccumPick* pk = reinterpret_cast<AccumPick*>(wb + L.pick);
    float* Pw = wb + L.p;

    for (int e = threadIdx.x; e < L.ds * nc; e += blockDim.x) {
        const int j = e / L.ds, c = e - j * L.ds;
        ds[e] = c < pc ? Dc[c + pc * j] : 0.f;
    }
    for (int e = lane; e < na * L.ps; e += 32) Pw[e] = 0.f;
    for (int e = lane; e < L.z; e += 32) Ys[e] = 0.f;
    __syncthreads();
    for (int e = threadIdx.x; e < nc * nc; e += blockDim.x) {   // as the Gram kernels form it
        const int i = e / nc, j = e - i * nc;
        float g = 0.f;
#pragma unroll 2
        for (int c = 0; c < pc; c += 4) {   // (zeros past pc)
            const float4 u = *reinterpret_cast<const float4*>(ds + i * L.ds + c);
            const float4 v = *reinterpret_cast<const float4*>(ds + j * L.ds + c);
            g = fmaf(u.x, v.x, g);
            g = fmaf(u.y, v.y, g);
            g = fmaf(u.z, v.z, g);
            g = fmaf(u.w, v.w, g);
        }
        gs[i * L.gs + j] = g;
    }
    __syncthreads();

    const bool vec = (reinterpret_cast<uintptr_t>(a.Y) & 15u) == 0 && (kD1 ? pp % 4 == 0 : p1 % 4 == 0);
    const unsigned inv_p1 = (65536u + p1 - 1) / p1;   // e / p1 for e < 1024
    auto fetch = [&](long long k) {
        const float* src = a.Y + (size_t)k * pp;
        if (vec) {
            for (int e = lane * 4; e < pp; e += 128) {
                int at = e;
                if constexpr (!kD1) {
                    const int b = (int)((unsigned)e * inv_p1 >> 16);
                    at = b * L.ys + (e - b * p1);
                }
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(Ys + at)),
                             "l"(src + e)
                             : "memory");
            }
        } else {
            for (int e = lane; e < pp; e += 32) {
                const int b = (int)((unsigned)e * inv_p1 >> 16);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(Ys + b * L.ys + (e - b * p1))),
                             "l"(src + e)
                             : "memory");
            }
        }
    };
    const int nq = a.n1 * a.n2;
    float bacc[PA];                          // B[:, lane]
#pragma unroll
    for (int r = 0; r < PA; ++r) bacc[r] = 0.f;
    double energy = 0.0;
    const long long step = (long long)gridDim.x * warps;
    long long k = (long long)w * gridDim.x + blockIdx.x;
    int qn = -1;
    float xn = 0.f;
    auto codes = [&](long long kk) {
        qn = -1;
        if (lane < s) {
            qn = a.in_support[(size_t)kk * s + lane];
            xn = a.in_coef[(size_t)kk * s + lane];
        }
    };
    if (k < a.N) {
        fetch(k);
        codes(k);
    }
    const int r = lane % PA, g = lane / PA, rc = min(r, pa - 1);   // rows past pa repeat the last (unused)
    const float inv_n1 = 1.f / (float)a.n1;
    for (; k < a.N; k += step) {
        // ---- the used picks, compacted
        const bool valid = lane < s && qn >= 0 && qn < nq && xn != 0.f;
        const unsigned vm = __ballot_sync(kFull, valid);
        const int cnt = __popc(vm);
        if (valid) {
            const int pos = __popc(vm & ((1u << lane) - 1u));
            int j = (int)((float)qn * inv_n1), i = qn - j * a.n1;   // q / n1, off by one at most
            if (i < 0) i += a.n1, --j;
            else if (i >= a.n1) i -= a.n1, ++j;
            const int o = kD1 ? j : i;
            pk[pos] = AccumPick{xn, kD1 ? i : j, o, o * L.gs};
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        // ---- ||Y||^2 (a non-finite signal is left out)
        float y2 = 0.f;
        if (vec && kD1) {
            for (int e = lane * 4; e < pp; e += 128) {
                const float4 v = *reinterpret_cast<const float4*>(Ys + e);
                y2 = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, y2))));
            }
        } else {
            for (int e = lane; e < pp; e += 32) {
                const int b = (int)((unsigned)e * inv_p1 >> 16);
                const float v = Ys[b * L.ys + (e - b * p1)];
                y2 = fmaf(v, v, y2);
            }
        }
        // 32 partial sums below 1e37 cannot add up to infinity
        const bool finite = __all_sync(kFull, y2 < 1e37f) || isfinite(warp_sum(y2));
        if (!finite && lane == 0) record_error(a.err, SDL_ERR_NONFINITE);
        if (ENERGY && finite) {
            // exact residual energy with the current dictionaries, U entries of a lane
            // at a time (one at a time, a pick's loads are a chain of their own).  Per update
            // with the objective, us, block-wide kernel | U = 1 | 2 | 4: 40 000 of 32x32 439 | 409 | 358 |
            // 326, of 16x64 with 32x128 atoms 770 | 549 | 453 | 430; 40 000 of 16x16 157 | 115 | 110 | 111,
            // of 12x12 103 | 86 | 86 | 92.
            float e2 = 0.f;
            auto residual = [&](auto uc) {
                constexpr int U = decltype(uc)::value;
                for (int e0 = lane; e0 < pp; e0 += 32 * U) {
                    float rec[U];
                    int at[U], oa[U], oc[U];   // in the signal, the updated and the other dictionary's columns
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int e = min(e0 + 32 * u, pp - 1);
                        const int b = (int)((unsigned)e * inv_p1 >> 16), aa = e - b * p1;
                        at[u] = b * L.ys + aa;
                        oa[u] = kD1 ? aa : b;
                        oc[u] = kD1 ? b : aa;
                        rec[u] = 0.f;
                    }
                    for (int l = 0; l < cnt; ++l) {
                        const AccumPick q = pk[l];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const float da = __ldg(Da + oa[u] + pa * q.i);
                            const float dc = ds[q.j * L.ds + oc[u]];
                            rec[u] = kD1 ? fmaf(q.x * da, dc, rec[u]) : fmaf(q.x * dc, da, rec[u]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (e0 + 32 * u < pp) {
                            const float res = Ys[at[u]] - rec[u];
                            e2 = fmaf(res, res, e2);
                        }
                }
            };
            if (pp <= 64) residual(std::integral_constant<int, 1>{});
            else if (pp < 512) residual(std::integral_constant<int, 2>{});
            else residual(std::integral_constant<int, 4>{});
            e2 = warp_sum(e2);
            energy += (double)e2;
        }
        // ---- projections z_l[r]
        if (finite) {
            for (int c0 = 0; c0 < pc; c0 += kChunk) {
                float y[kChunk];
#pragma unroll
                for (int c = 0; c < kChunk; c += 4) {
                    if (c0 + c < pc) {   // terms past pc are zero in both factors
                        if constexpr (kD1) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) y[c + u] = Ys[rc + L.ys * (c0 + c + u)];
                        } else {
                            const float4 v = *reinterpret_cast<const float4*>(Ys + rc * L.ys + c0 + c);
                            y[c] = v.x; y[c + 1] = v.y; y[c + 2] = v.z; y[c + 3] = v.w;
                        }
                    }
                }
                for (int l = g; l < cnt; l += LG) {
                    const float* d = ds + pk[l].j * L.ds + c0;
                    float z = c0 ? zs[l * PA + r] : 0.f;
#pragma unroll
                    for (int c = 0; c < kChunk; c += 4)
                        if (c0 + c < pc) {
                            const float4 v = *reinterpret_cast<const float4*>(d + c);
                            z = fmaf(y[c], v.x, z);
                            z = fmaf(y[c + 1], v.y, z);
                            z = fmaf(y[c + 2], v.z, z);
                            z = fmaf(y[c + 3], v.w, z);
                        }
                    zs[l * PA + r] = z;
                }
            }
        }
        __syncwarp();   // Y is consumed: fetch the next signal
        const long long kn = k + step;
        if (kn < a.N) {
            fetch(kn);
            codes(kn);
        }
        // ---- sums, lane = atom
        if (finite) {
            unsigned mine = 0;
            for (int l = 0; l < cnt; ++l) mine |= (pk[l].i == lane ? 1u : 0u) << l;
            for (unsigned m = mine; __any_sync(kFull, m != 0u); m &= m - 1)
                if (m) {
                    const int l = __ffs(m) - 1;
                    const float x = pk[l].x;
#pragma unroll
                    for (int e = 0; e < PA; e += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(zs + l * PA + e);
                        bacc[e] = fmaf(x, v.x, bacc[e]);
                        bacc[e + 1] = fmaf(x, v.y, bacc[e + 1]);
                        bacc[e + 2] = fmaf(x, v.z, bacc[e + 2]);
                        bacc[e + 3] = fmaf(x, v.w, bacc[e + 3]);
                    }
                }
            // row `lane` of P: the first two picks of the lane's atom from
            // registers, further ones (rare) in rounds of their own
            for (unsigned m = mine; m;) {
                const AccumPick q0 = pk[__ffs(m) - 1];
                m &= m - 1;
                AccumPick q1 = q0;
                q1.x = 0.f;
                if (m) q1 = pk[__ffs(m) - 1];
                m &= m - 1;
                const int j0 = q0.j, j1 = q1.j;
                float* row = Pw + lane * L.ps;
                for (int l = 0; l < cnt; ++l) {
                    const AccumPick q = pk[l];
                    const float u = fmaf(q1.x, gs[q.g + j1], q0.x * gs[q.g + j0]);
                    row[q.i] = fmaf(q.x, u, row[q.i]);
                }
            }
        }
        __syncwarp();   // picks and projections are read before the next signal's
    }

    // ---- this CTA's slot: the warps' sums in warp order
    __shared__ double se[kWarps];
    float* bw = wb;                          // B of the warp, over its signal and projections
#pragma unroll
    for (int e = 0; e < PA; ++e)
        if (lane < na) bw[lane * PA + e] = bacc[e];
    if (lane == 0) se[w] = energy;
    __syncthreads();
    const int nf = na * na + pa * na;
    float* dst = a.part_f + (size_t)blockIdx.x * nf;
    for (int e = threadIdx.x; e < nf; e += blockDim.x) {
        int off;
        if (e < na * na) {
            const int i = e / na;
            off = L.p + i * L.ps + (e - i * na);
        } else {
            const int f = e - na * na, rr = f / na;
            off = (f - rr * na) * PA + rr;
        }
        float v = 0.f;
        for (int ww = 0; ww < warps; ++ww) v += sm[L.warp0 + ww * L.stride + off];
        dst[e] = v;
    }
    if (threadIdx.x == 0) {
        double d = 0.0;
        for (int ww = 0; ww < warps; ++ww) d += se[ww];
        a.part_d[2 * blockIdx.x] = d;
        a.part_d[2 * blockIdx.x + 1] = 0.0;
    }
}

template <int PA, int SIDE>
int launch(const PassArgs& a, bool want_energy, cudaStream_t st, int num_sms, size_t bytes, int warps) {
    auto kern = want_energy ? accum_lane_kernel<PA, SIDE, true> : accum_lane_kernel<PA, SIDE, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 1024) != cudaSuccess)
        return SDL_ERR_CUDA;
    const int bps = std::max(1, std::min<int>(kMinCtas, (int)((228 * 1024) / (bytes + 2048))));
    const long long grid = std::max<long long>(1, std::min<long long>((a.N + warps - 1) / warps, (long long)num_sms * bps));
    kern<<<(int)grid, warps * 32, bytes, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? (int)grid : SDL_ERR_CUDA;
}

// Rows per lane block, warps per CTA (0: the pass does not take these sizes) and
// shared memory of a CTA.
struct AccumPlan {
    int PA = 0, warps = 0;
    size_t bytes = 0;
};
AccumPlan plan(const PassArgs& a, int side) {
    const int pa = side == kSideD1 ? a.p1 : a.p2, pc = side == kSideD1 ? a.p2 : a.p1;
    const int na = side == kSideD1 ? a.n1 : a.n2, nc = side == kSideD1 ? a.n2 : a.n1;
    AccumPlan q;
    if (na > 32 || pa > 32) return q;
    q.PA = pa <= 8 ? 8 : pa <= 16 ? 16 : 32;
    for (int warps = kWarps; warps >= 4; --warps) {
        q.bytes = sizeof(float) * (size_t)AccumLayout(a.p1, a.p2, pa, pc, na, nc, a.s, q.PA, side, warps).total;
        if (q.bytes <= 200 * 1024) {
            q.warps = warps;
            break;
        }
    }
    return q;
}

template <int SIDE>
int run(const PassArgs& a, bool want_energy, cudaStream_t st, int num_sms) {
    const AccumPlan q = plan(a, SIDE);
    if (q.warps == 0) return SDL_ERR_UNSUPPORTED;
    switch (q.PA) {
        case 8: return launch<8, SIDE>(a, want_energy, st, num_sms, q.bytes, q.warps);
        case 16: return launch<16, SIDE>(a, want_energy, st, num_sms, q.bytes, q.warps);
        default: return launch<32, SIDE>(a, want_energy, st, num_sms, q.bytes, q.warps);
    }
}

}  // namespace

bool accumulate_lanes_take(const PassArgs& a, int side) { return plan(a, side).warps > 0; }

int launch_accumulate_lanes(const PassArgs& a, int side, bool want_energy, cudaStream_t st, int num_sms) {
    return side == kSideD1 ? run<kSideD1>(a, want_energy, st, num_sms) : run<kSideD2>(a, want_energy, st, num_sms);
}

}  // namespace sdl
