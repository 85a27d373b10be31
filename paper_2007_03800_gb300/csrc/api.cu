// C ABI of the library (declared in include/sdl.h): argument checks, the
// context workspace, and the launch sequences of the entry points.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "ctx.cuh"

using namespace sdl;

namespace {

template <class T>
int grow(T*& ptr, size_t& cap, size_t need) {
    if (need <= cap && ptr) return SDL_OK;
    if (ptr) cudaFree(ptr);
    ptr = nullptr;
    cap = 0;
    const size_t n = std::max<size_t>(need, 1);
    if (cudaMalloc(&ptr, n * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return SDL_ERR_WORKSPACE;
    }
    cap = n;
    return SDL_OK;
}

int ensure_workspace(sdl_ctx* c, int p1, int p2, int n1, int n2) {
    const size_t nmax = (size_t)std::max(n1, n2);
    const size_t nf = std::max<size_t>((size_t)n1 * n1 + (size_t)p1 * n1,
                                       (size_t)n2 * n2 + (size_t)p2 * n2);
    const size_t slots = (size_t)max_partial_slots(c->num_sms);
    int rc;
    if ((rc = grow(c->G1, c->cap_g1, nmax * nmax)) != SDL_OK) return rc;
    if ((rc = grow(c->G2, c->cap_g2, nmax * nmax)) != SDL_OK) return rc;
    if ((rc = grow(c->part_f, c->cap_part, slots * nf)) != SDL_OK) return rc;
    if ((rc = grow(c->part_d, c->cap_slots, slots * 2)) != SDL_OK) return rc;
    if ((rc = grow(c->red_f, c->cap_red, nf)) != SDL_OK) return rc;
    if ((rc = grow(c->red_d, c->cap_redd, (size_t)2)) != SDL_OK) return rc;
    if ((rc = grow(c->norms, c->cap_norms, nmax)) != SDL_OK) return rc;
    return SDL_OK;
}

bool valid_common(const sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, int n1, int n2,
                  int s) {
    if (!c || p1 < 1 || p2 < 1 || n1 < 1 || n2 < 1 || N < 0 || s < 1) return false;
    if (N > 0 && !Y) return false;
    return true;
}

int check_shape(int p1, int p2, int n1, int n2, int s) {
    if (s > kMaxS || s > p1 * p2 || s > n1 * n2) return SDL_ERR_ARG;
    if (!code_shape_supported(p1, p2, n1, n2, s)) return SDL_ERR_UNSUPPORTED;
    return SDL_OK;
}

sdl_ctx::Pin* find_pin(sdl_ctx* c, int p1, int p2, int n1, int n2, int s) {
    for (auto& pin : c->pins)
        if (pin.p1 == p1 && pin.p2 == p2 && pin.n1 == n1 && pin.n2 == n2 && pin.s == s) return &pin;
    return nullptr;
}

PassArgs base_args(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, const float* D1, int n1,
                   const float* D2, int n2, int s) {
    PassArgs a;
    std::memset(&a, 0, sizeof(a));
    a.Y = Y;
    a.p1 = p1;
    a.p2 = p2;
    a.N = N;
    a.D1 = D1;
    a.D2 = D2;
    a.G1 = c->G1;
    a.G2 = c->G2;
    a.n1 = n1;
    a.n2 = n2;
    a.s = s;
    a.part_f = c->part_f;
    a.part_d = c->part_d;
    a.n_slots = 1;
    a.err = c->err;
    if (const sdl_ctx::Pin* pin = find_pin(c, p1, p2, n1, n2, s)) {
        a.tiling = pin->id + 1;
        a.tiling_cps = pin->cps;
        a.tiling_forced = pin->forced ? 1 : 0;
    }
    return a;
}

void pin_tiling(sdl_ctx* c, const sdl_ctx::Pin& p) {
    if (sdl_ctx::Pin* old = find_pin(c, p.p1, p.p2, p.n1, p.n2, p.s)) *old = p;
    else c->pins.push_back(p);
}

void grams(sdl_ctx* c, const float* D1, int p1, int n1, const float* D2, int p2, int n2,
           cudaStream_t st) {
    Trace tr(c, kGram, st);
    launch_gram2(D1, p1, n1, c->G1, D2, p2, n2, c->G2, st);
}

// Tensor-core correlations for a coding pass (precision extension): fills
// ctx->C0 and points the pass at it.
int prepare_tc_pass(sdl_ctx* c, PassArgs& a, bool fill_y, cudaStream_t st) {
    const long long N = a.N;
    const int Kp = (a.p1 * a.p2 + 7) & ~7, Q = a.n1 * a.n2;
    int rc;
    // hi and lo BF16 parts of the signals and of the Kronecker dictionary
    if ((rc = grow(reinterpret_cast<char*&>(c->Yb), c->cap_yb, (size_t)N * Kp * 4)) != SDL_OK) return rc;
    if ((rc = grow(reinterpret_cast<char*&>(c->KT), c->cap_kt, (size_t)Q * Kp * 4)) != SDL_OK) return rc;
    if ((rc = grow(c->C0, c->cap_c0, (size_t)N * Q)) != SDL_OK) return rc;
    if (!c->rescored) {
        if (cudaMalloc(&c->rescored, sizeof(unsigned long long)) != cudaSuccess) return SDL_ERR_WORKSPACE;
        cudaMemset(c->rescored, 0, sizeof(unsigned long long));
    }
    {
        Trace tr(c, kTcCorr, st);
        rc = tc_correlations(a.Y, N, a.p1, a.p2, a.D1, a.n1, a.D2, a.n2,
                             static_cast<__nv_bfloat16*>(c->Yb), fill_y,
                             static_cast<__nv_bfloat16*>(c->KT), c->C0, c->err, st);
    }
    if (rc) return rc;
    a.c0ext = c->C0;
    a.ldc0 = Q;
    a.c0_err_rel = (c->prec & SDL_PREC_NO_RESCORE) ? 0.f : c0_split_err_rel(a.p1 * a.p2);
    a.rescored = c->rescored;
    return SDL_OK;
}

// Partial-sum slots of a learning pass that runs as the lane-group coder followed
// by the ordered sums (compiled shapes, fixed sparsity, aligned signals, no tiling
// forced or tuned to be faster), or 0: the fused kernels.  Two launches instead of one pay off from
// about 2.1M correlations on: an iteration (us, split / fused) at 8x8 x 4000 78 / 75,
// x 16000 95 / 99, x 64000 169 / 202; at 12x12 x 2000 94 / 88, x 4000 97 / 100,
// x 64000 332 / 421; at 16x16 x 1000 110 / 101, x 4000 130 / 137, x 64000 688 / 987.
constexpr long long kSplitPairs = 2100000;
int split_pass_slots(const PassArgs& a, bool tc, int num_sms) {
    if (a.N * a.n1 * a.n2 < kSplitPairs) return 0;
    if (tc || a.tiling_forced || a.eps2 > 0.f || a.N < 1 || (reinterpret_cast<uintptr_t>(a.Y) & 15u)) return 0;
    return std::max(0, ordered_slots(a, num_sms));
}

// One such pass: codes to the caller's arrays (both passes: the second rewrites
// them), residual energies to the slots of part_d, sums to those of part_f.
int split_pass(sdl_ctx* c, const PassArgs& a0, int side, int slots, int32_t* support, float* coef, int32_t* nnz,
               cudaStream_t st) {
    PassArgs a = a0;
    a.support = support;
    a.coef = coef;
    a.nnz = nnz;
    a.esum = c->part_d;
    a.esum_slots = slots;
    int rc;
    {
        Trace tr(c, side == kSideD1 ? kCodeD1 : kCodeD2, st);
        rc = launch_code_group_fixed(a, side == kSideD2, st, c->num_sms, slots);
    }
    if (rc != SDL_OK) return rc;
    a.in_support = support;
    a.in_coef = coef;
    Trace tr(c, side == kSideD1 ? kAccD1 : kAccD2, st);
    rc = launch_accumulate_ordered(a, side, st, c->num_sms);
    return rc == SDL_OK ? slots : rc;
}

// reduce -> solve for one dictionary side, using the partial sums in slots.
int finish_update(sdl_ctx* c, int slots, int side, float* D, int p1, int p2, int64_t N, int n1,
                  int n2, double* objective_out, double* rmse_out, cudaStream_t st,
                  float* G_out = nullptr) {
    const int p = side == kSideD1 ? p1 : p2;
    const int n = side == kSideD1 ? n1 : n2;
    const int nf = n * n + p * n;
    {
        Trace tr(c, kReduce, st);
        launch_reduce_partials(c->part_f, c->part_d, slots, nf, c->red_f, c->red_d, st);
    }
    const double inv_count = N > 0 ? 1.0 / ((double)p1 * p2 * (double)N) : 0.0;
    Trace tr(c, kSolve, st);
    if (c->prec & SDL_PREC_FP64_SOLVE)
        return launch_solve64(c->red_f, c->red_d, D, p, n, c->norms, inv_count, objective_out,
                              rmse_out, c->err, st, G_out);
    return launch_solve(c->red_f, c->red_d, D, p, n, c->norms, inv_count, objective_out, rmse_out,
                        c->err, st, G_out);
}

}  // namespace

namespace sdl {
int ctx_workspace(sdl_ctx* c, int p1, int p2, int n1, int n2) {
    return ensure_workspace(c, p1, p2, n1, n2);
}
}  // namespace sdl

extern "C" {

const char* sdl_strerror(int code) {
    switch (code) {
        case SDL_OK: return "ok";
        case SDL_ERR_ARG: return "invalid argument";
        case SDL_ERR_CUDA: return "CUDA runtime error";
        case SDL_ERR_NONFINITE: return "non-finite value in the data or a normal matrix";
        case SDL_ERR_SINGULAR: return "normal matrix not positive definite";
        case SDL_ERR_TIMEOUT: return "device-side wait timed out";
        case SDL_ERR_WORKSPACE: return "workspace allocation failed";
        case SDL_ERR_UNSUPPORTED: return "shape not supported by the compiled kernels";
        case SDL_ERR_CAPACITY: return "problem exceeds the static scratch capacity";
        default: return "unknown error";
    }
}

int sdl_create(sdl_ctx** out, int device) {
    if (!out) return SDL_ERR_ARG;
    *out = nullptr;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) {
        cudaGetLastError();
        return SDL_ERR_CUDA;
    }
    if (cudaSetDevice(device) != cudaSuccess) return SDL_ERR_CUDA;
    sdl_ctx* c = new (std::nothrow) sdl_ctx();
    if (!c) return SDL_ERR_WORKSPACE;
    c->device = device;
    if (cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
        delete c;
        return SDL_ERR_CUDA;
    }
    if (cudaMalloc(&c->err, sizeof(int)) != cudaSuccess || cudaMemset(c->err, 0, sizeof(int)) != cudaSuccess ||
        cudaMalloc(&c->scan_word, sizeof(unsigned long long)) != cudaSuccess ||
        cudaMemset(c->scan_word, 0, sizeof(unsigned long long)) != cudaSuccess ||
        cudaStreamSynchronize(nullptr) != cudaSuccess) {   // calls on any stream find them cleared
        cudaGetLastError();
        cudaFree(c->err);
        cudaFree(c->scan_word);
        delete c;
        return SDL_ERR_WORKSPACE;
    }
    *out = c;
    return SDL_OK;
}

int sdl_destroy(sdl_ctx* c) {
    if (!c) return SDL_OK;
    DeviceGuard g(c->device);
    cudaDeviceSynchronize();
    cudaFree(c->err);
    cudaFree(c->scan_word);
    cudaFree(c->G1);
    cudaFree(c->G2);
    cudaFree(c->part_f);
    cudaFree(c->part_d);
    cudaFree(c->red_f);
    cudaFree(c->red_d);
    cudaFree(c->norms);
    cudaFree(c->rec);
    cudaFree(c->learn);
    cudaFree(c->ssim_part);
    cudaFree(c->G3);
    cudaFree(c->Yb);
    cudaFree(c->KT);
    cudaFree(c->C0);
    cudaFree(c->rescored);
    for (cudaEvent_t e : c->side_ev)
        if (e) cudaEventDestroy(e);
    if (c->side) cudaStreamDestroy(c->side);
    for (auto& r : c->recs) {
        cudaEventDestroy(r.beg);
        cudaEventDestroy(r.end);
    }
    delete c;
    return SDL_OK;
}

int sdl_status(sdl_ctx* c, void* stream) {
    if (!c) return SDL_ERR_ARG;
    DeviceGuard g(c->device);
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) {
        cudaGetLastError();
        return SDL_ERR_CUDA;
    }
    int h = 0;
    if (cudaMemcpy(&h, c->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemset(c->err, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return SDL_ERR_CUDA;
    }
    return h;
}

int sdl_shape_supported(int p1, int p2, int n1, int n2, int s) {
    return check_shape(p1, p2, n1, n2, s) == SDL_OK && p1 >= 1 && p2 >= 1 ? 1 : 0;
}

int sdl_reserve(sdl_ctx* c, int p1, int p2, int n1, int n2, int s) {
    if (!c || p1 < 1 || p2 < 1 || n1 < 1 || n2 < 1 || s < 1) return SDL_ERR_ARG;
    int rc = check_shape(p1, p2, n1, n2, s);
    if (rc != SDL_OK) return rc;
    DeviceGuard g(c->device);
    return ensure_workspace(c, p1, p2, n1, n2);
}

int sdl_sparse_code(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, const float* D1, int n1,
                    const float* D2, int n2, int s, float eps, int32_t* support, float* coef,
                    int32_t* nnz, float* res_energy, void* stream) {
    if (!valid_common(c, Y, p1, p2, N, n1, n2, s) || !D1 || !D2) return SDL_ERR_ARG;
    if (N > 0 && (!support || !coef || !nnz)) return SDL_ERR_ARG;
    int rc = check_shape(p1, p2, n1, n2, s);
    if (rc != SDL_OK) return rc;
    if (N == 0) return SDL_OK;
    DeviceGuard g(c->device);
    if ((rc = ensure_workspace(c, p1, p2, n1, n2)) != SDL_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    PassArgs a = base_args(c, Y, p1, p2, N, D1, n1, D2, n2, s);
    a.eps2 = eps > 0.f ? eps * eps : 0.f;
    a.support = support;
    a.coef = coef;
    a.nnz = nnz;
    a.res_energy = res_energy;
    if (!(c->prec & SDL_PREC_BF16_CORR) && code_lanes_take(a, c->cap_part)) {
        Trace tr(c, kCode, st);
        return launch_code_lanes(a, c->part_f, c->cap_part, c->scan_word, st, c->num_sms);
    }
    grams(c, D1, p1, n1, D2, p2, n2, st);
    if ((c->prec & SDL_PREC_BF16_CORR) && (rc = prepare_tc_pass(c, a, true, st)) != SDL_OK) return rc;
    {
        Trace tr(c, kCode, st);
        rc = launch_code_pass(a, kCodeOnly, st, c->num_sms);
    }
    return rc < 0 ? rc : SDL_OK;
}

static int update_common(sdl_ctx* c, int side, const float* Y, int p1, int p2, int64_t N,
                         const float* D1, float* D1w, int n1, const float* D2, float* D2w, int n2,
                         int s, const int32_t* support, float* coef, double* objective_out,
                         void* stream) {
    if (!valid_common(c, Y, p1, p2, N, n1, n2, s) || !D1 || !D2) return SDL_ERR_ARG;
    if (N > 0 && (!support || !coef)) return SDL_ERR_ARG;
    int rc = check_shape(p1, p2, n1, n2, s);
    if (rc != SDL_OK) return rc;
    DeviceGuard g(c->device);
    if ((rc = ensure_workspace(c, p1, p2, n1, n2)) != SDL_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    PassArgs a = base_args(c, Y, p1, p2, N, D1, n1, D2, n2, s);
    a.in_support = support;
    a.in_coef = coef;
    const bool lanes = accumulate_lanes_take(a, side);
    if (!lanes) grams(c, D1, p1, n1, D2, p2, n2, st);
    int slots;
    {
        // the residual energy before the update goes to objective_out alone
        Trace tr(c, side == kSideD1 ? kAccD1 : kAccD2, st);
        slots = lanes ? launch_accumulate_lanes(a, side, objective_out != nullptr, st, c->num_sms)
                      : launch_accumulate_pass(a, side, st, c->num_sms);
    }
    if (slots < 0) return slots;
    float* D = side == kSideD1 ? D1w : D2w;
    rc = finish_update(c, slots, side, D, p1, p2, N, n1, n2, objective_out, nullptr, st);
    if (rc != SDL_OK) return rc;
    if (N > 0) {
        Trace tr(c, kRescale, st);
        launch_rescale(support, coef, N * (long long)s, n1, n2, side, c->norms, st);
    }
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_update_D1(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, float* D1, int n1,
                  const float* D2, int n2, int s, const int32_t* support, float* coef,
                  double* objective_out, void* stream) {
    return update_common(c, kSideD1, Y, p1, p2, N, D1, D1, n1, D2, nullptr, n2, s, support, coef,
                         objective_out, stream);
}

int sdl_update_D2(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, const float* D1, int n1,
                  float* D2, int n2, int s, const int32_t* support, float* coef,
                  double* objective_out, void* stream) {
    return update_common(c, kSideD2, Y, p1, p2, N, D1, nullptr, n1, D2, D2, n2, s, support, coef,
                         objective_out, stream);
}

int sdl_iterate(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, float* D1, int n1, float* D2,
                int n2, int s, float eps, int32_t* support, float* coef, int32_t* nnz,
                double* rmse_out, void* stream) {
    if (!valid_common(c, Y, p1, p2, N, n1, n2, s) || !D1 || !D2) return SDL_ERR_ARG;
    if (N > 0 && (!support || !coef || !nnz)) return SDL_ERR_ARG;
    int rc = check_shape(p1, p2, n1, n2, s);
    if (rc != SDL_OK) return rc;
    DeviceGuard g(c->device);
    if ((rc = ensure_workspace(c, p1, p2, n1, n2)) != SDL_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const float eps2 = eps > 0.f ? eps * eps : 0.f;

    PassArgs a = base_args(c, Y, p1, p2, N, D1, n1, D2, n2, s);
    a.eps2 = eps2;
    const bool tc = (c->prec & SDL_PREC_BF16_CORR) != 0;
    const sdl_ctx::Pin* pin = find_pin(c, p1, p2, n1, n2, s);
    if (pin && N <= pin->fused_n) a.tiling_forced = 1;
    const int ordered = split_pass_slots(a, tc, c->num_sms);
    // one coding pass with its sums: the number of partial-sum slots
    auto code_side = [&](int side) -> int {
        if (ordered > 0) return split_pass(c, a, side, ordered, support, coef, nnz, st);
        Trace tr(c, side == kSideD1 ? kCodeD1 : kCodeD2, st);
        return launch_code_pass(a, side, st, c->num_sms);
    };

    // steps 1-2: code with (D1, D2) accumulating P, B1; solve for D1
    if (ordered <= 0) grams(c, D1, p1, n1, D2, p2, n2, st);
    if (tc && (rc = prepare_tc_pass(c, a, true, st)) != SDL_OK) return rc;
    int slots = code_side(kSideD1);
    if (slots < 0) return slots;
    // the solve also refreshes G1 for the new D1
    rc = finish_update(c, slots, kSideD1, D1, p1, p2, N, n1, n2, nullptr, rmse_out, st,
                       ordered > 0 ? nullptr : c->G1);
    if (rc != SDL_OK) return rc;
    // steps 3-4: code with the new D1 accumulating M, B2; solve for D2
    a.support = support;
    a.coef = coef;
    a.nnz = nnz;
    if (tc && (rc = prepare_tc_pass(c, a, false, st)) != SDL_OK) return rc;   // new D1
    slots = code_side(kSideD2);
    if (slots < 0) return slots;
    rc = finish_update(c, slots, kSideD2, D2, p1, p2, N, n1, n2, nullptr,
                       rmse_out ? rmse_out + 1 : nullptr, st);
    if (rc != SDL_OK) return rc;
    if (N > 0) {
        Trace tr(c, kRescale, st);
        launch_rescale(support, coef, N * (long long)s, n1, n2, kSideD2, c->norms, st);
    }
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_tilings(int p1, int p2, int n1, int n2, int s, int* ids, int max_ids) {
    if (max_ids < 0) return SDL_ERR_ARG;
    int all[64];
    const int n = fast_shape_variants(p1, p2, n1, n2, s, all, 64);
    for (int v = 0; v < n && v < max_ids; ++v)
        if (ids) ids[v] = all[v];
    return n;
}

int sdl_set_tiling(sdl_ctx* c, int p1, int p2, int n1, int n2, int s, int tiling, int ctas_per_sm) {
    if (!c || ctas_per_sm < 0 || ctas_per_sm > 8) return SDL_ERR_ARG;
    if (tiling < 0) {
        for (size_t k = 0; k < c->pins.size(); ++k)
            if (c->pins[k].p1 == p1 && c->pins[k].p2 == p2 && c->pins[k].n1 == n1 &&
                c->pins[k].n2 == n2 && c->pins[k].s == s) {
                c->pins.erase(c->pins.begin() + (long)k);
                break;
            }
        return SDL_OK;
    }
    int all[64];
    const int n = fast_shape_variants(p1, p2, n1, n2, s, all, 64);
    for (int v = 0; v < n; ++v)
        if (all[v] == tiling) {
            pin_tiling(c, sdl_ctx::Pin{p1, p2, n1, n2, s, tiling, ctas_per_sm, true, 0});
            return SDL_OK;
        }
    return SDL_ERR_UNSUPPORTED;
}

int sdl_tune_tiling(sdl_ctx* c, const float* Y, int p1, int p2, int64_t N, const float* D1, int n1,
                    const float* D2, int n2, int s, int* tiling_out, void* stream) {
    if (!valid_common(c, Y, p1, p2, N, n1, n2, s) || !D1 || !D2 || N < 1) return SDL_ERR_ARG;
    int rc = check_shape(p1, p2, n1, n2, s);
    if (rc != SDL_OK) return rc;
    if ((reinterpret_cast<uintptr_t>(Y) & 15u) != 0) return SDL_ERR_UNSUPPORTED;
    int ids[64];
    const int n = fast_shape_variants(p1, p2, n1, n2, s, ids, 64);
    if (n == 0) return SDL_ERR_UNSUPPORTED;
    DeviceGuard g(c->device);
    if ((rc = ensure_workspace(c, p1, p2, n1, n2)) != SDL_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    grams(c, D1, p1, n1, D2, p2, n2, st);
    PassArgs a = base_args(c, Y, p1, p2, N, D1, n1, D2, n2, s);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return SDL_ERR_CUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return SDL_ERR_CUDA;
    }
    // one untimed run, then the mean of three, in us (negative: did not run)
    bool failed = false;
    auto timed = [&](auto&& run) -> float {
        if (run() < 0) return -1.f;
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) run();
        cudaEventRecord(e1, st);
        float ms = 0.f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            failed = true;
            return -1.f;
        }
        return ms * 1000.f / 3.f;
    };
    c->tune_log.clear();
    int best_id = -1, best_cps = 0;
    float best = 1e30f;
    // the fused tilings: D1-side passes, the heavier of the two epilogues
    for (int v = 0; v < n && !failed; ++v) {
        for (int cps = 1; cps <= 2 && !failed; ++cps) {
            const float us =
                timed([&] { return launch_code_pass_variant(a, kSideD1, ids[v], cps, st, c->num_sms); });
            if (us < 0.f) continue;
            c->tune_log.push_back(sdl_ctx::TuneRec{ids[v], cps, us});
            if (us < best) {
                best = us;
                best_id = ids[v];
                best_cps = cps;
            }
        }
    }
    // The same pass by lane groups, where a learning iteration on N signals would
    // run so: it keeps that form unless the best tiling beats it here.
    sdl_ctx::Pin pin{p1, p2, n1, n2, s, best_id, best_cps, false, 0};
    a.tiling_forced = 0;
    const int slots = failed ? 0 : split_pass_slots(a, false, c->num_sms);
    char* codes = nullptr;
    const size_t words = (size_t)N * s;
    if (slots > 0 && cudaMalloc(&codes, 4 * (2 * words + (size_t)N)) == cudaSuccess) {
        int32_t* sup = reinterpret_cast<int32_t*>(codes);
        float* coef = reinterpret_cast<float*>(sup + words);
        int32_t* nnz = reinterpret_cast<int32_t*>(coef + words);
        int64_t kept[SDL_NUM_KERNEL_KINDS];   // timing runs are not counted
        std::copy(c->launches, c->launches + SDL_NUM_KERNEL_KINDS, kept);
        const bool traced = c->timing;
        c->timing = false;
        const float us = timed([&] { return split_pass(c, a, kSideD1, slots, sup, coef, nnz, st); });
        c->timing = traced;
        std::copy(kept, kept + SDL_NUM_KERNEL_KINDS, c->launches);
        if (us < 0.f || us > best) pin.fused_n = N;
        cudaFree(codes);
    } else {
        cudaGetLastError();
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (failed || best_id < 0) return SDL_ERR_CUDA;
    pin_tiling(c, pin);
    if (tiling_out) *tiling_out = best_id;
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

int sdl_tune_log(const sdl_ctx* c, int* tiling, int* ctas_per_sm, float* cost_us, int max_entries) {
    if (!c || max_entries < 0) return SDL_ERR_ARG;
    const int n = (int)c->tune_log.size();
    for (int e = 0; e < n && e < max_entries; ++e) {
        if (tiling) tiling[e] = c->tune_log[e].id;
        if (ctas_per_sm) ctas_per_sm[e] = c->tune_log[e].cps;
        if (cost_us) cost_us[e] = c->tune_log[e].us;
    }
    return n;
}

int sdl_set_precision(sdl_ctx* c, int flags) {
    if (!c || (flags & ~(SDL_PREC_BF16_CORR | SDL_PREC_NO_RESCORE | SDL_PREC_FP64_SOLVE))) return SDL_ERR_ARG;
    c->prec = flags;
    return SDL_OK;
}

int sdl_precision_stats(sdl_ctx* c, uint64_t* rescored) {
    if (!c || !rescored) return SDL_ERR_ARG;
    DeviceGuard g(c->device);
    *rescored = 0;
    if (!c->rescored) return SDL_OK;
    unsigned long long h = 0;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(&h, c->rescored, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemset(c->rescored, 0, sizeof(h)) != cudaSuccess) {
        cudaGetLastError();
        return SDL_ERR_CUDA;
    }
    *rescored = (uint64_t)h;
    return SDL_OK;
}

int sdl_profile_enable(sdl_ctx* c, int enable) {
    if (!c) return SDL_ERR_ARG;
    c->timing = enable != 0;
    return SDL_OK;
}

int sdl_profile_collect(sdl_ctx* c, double* total_ms, int64_t* launches, int max_kinds) {
    if (!c || max_kinds < 0) return SDL_ERR_ARG;
    DeviceGuard g(c->device);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return SDL_ERR_CUDA;
    }
    double tot[SDL_NUM_KERNEL_KINDS] = {};
    for (size_t r = 0; r < c->n_recs; ++r) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, c->recs[r].beg, c->recs[r].end) == cudaSuccess)
            tot[c->recs[r].kind] += ms;
        else
            cudaGetLastError();
    }
    c->n_recs = 0;
    const int m = std::min(max_kinds, (int)SDL_NUM_KERNEL_KINDS);
    for (int k = 0; k < m; ++k) {
        if (total_ms) total_ms[k] = tot[k];
        if (launches) launches[k] = c->launches[k];
    }
    for (int k = 0; k < SDL_NUM_KERNEL_KINDS; ++k) c->launches[k] = 0;
    return SDL_NUM_KERNEL_KINDS;
}

const char* sdl_kernel_name(int kind) {
    static const char* names[SDL_NUM_KERNEL_KINDS] = {
        "gram", "code", "code_D1", "code_D2", "accum_D1", "accum_D2",
        "reduce", "solve", "rescale", "memset", "batch_graph", "mlp", "adam", "topk",
        "shortlist", "tc_corr", "ortho_code", "procrustes"};
    return (kind >= 0 && kind < SDL_NUM_KERNEL_KINDS) ? names[kind] : "?";
}

}  // extern "C"
