// 2D-OMP coding pass with a small group of lanes per signal: a warp codes
// 32 / GL signals at once, GL = 8 or 16 lanes each; wide dictionaries take a whole warp
// (32) or a team of two (64) per signal.
//
// Same method and arithmetic as the one-warp-per-signal coders (omp_fast.cu,
// omp_pass.cu): every entry of Z, C0 and of the scores, the Cholesky rows and
// both triangular solves are the same FMA chains in the same order, so the
// codes are bit-identical to theirs.  What bounds a coding pass here is the
// number of warp instructions, not the FMAs among them (about one in six in the
// one-warp form).  With GL lanes per signal:
//   * the per-signal scalar work (pick, Cholesky row, solves), which every lane
//     of a signal repeats, is issued once for 32 / GL signals;
//   * a lane's RI x RJ block is large, so each operand load feeds more FMAs;
//   * the argmax takes three-input |max| (two entries per instruction) down
//     the columns of the block and a compare/select only per column; the row
//     comes from one read-back of the winning column;
//   * the greedy loop is a loop over t, with only the Cholesky row unrolled per
//     t, so that the code of all steps fits the instruction cache.
// Scores are recomputed from C0 every step, as in the other coders.
//
// Measured (GB300, us per call, one warp per signal -> this kernel): 200 000 x
// 12x12, 24x24 pairs, s = 6: 472 -> 318 (of the compiled tilings the fastest,
// two signals per warp, takes 410); 247 009 x 16x16, 32x32, s = 8: 1636 -> 1003;
// 99 991 x 10x9, 20x18, s = 5 (generic kernel before): 493 -> 161.  At 12x12 a
// signal takes 1106 warp instructions (1877 before); 71 % of the shared-memory
// bandwidth (operands of the rank-one updates, and C0 read back every step) and
// 51 % of the issue slots are in use; the serial chain of a greedy step (argmax,
// read-back, Cholesky row) sets the rest: a copy of C0 in tensor memory that took
// the read-back off the shared memory left the time as it was (330 us).
#pragma once

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "sdl_internal.cuh"

namespace sdl {
namespace group {

constexpr unsigned kFull = 0xffffffffu;

__host__ __device__ constexpr int up4(int x) { return (x + 3) & ~3; }

// GL lanes per signal in a grid of LI x GL / LI, RI x RJ entries of C0 per lane, WARPS
// per CTA, MINB CTAs per SM.
// P1 .. N2, S: sizes fixed at compile time (0: taken from the call).
// FAST: 1/sqrt by rsqrtf and back substitution in increasing row order
// (the compiled tilings' forms); else 1/sqrtf and decreasing order (the
// generic kernel's).  W: C0 = (D1^T Y) D2 rather than D1^T (Y D2).
// ORTHO_: 0, or the orthonormal variant (n = p; a pick's coefficient is its
// correlation and leaves the others alone) with ||Y||^2 in that many chains.
template <int GL_, int LI_, int RI_, int RJ_, int WARPS_, int MINB_, bool FAST_, bool W_, int P1_ = 0,
          int P2_ = 0, int N1_ = 0, int N2_ = 0, int S_ = 0, int ORTHO_ = 0, int CHAINS_ = 32,
          bool TM_ = false, bool SHORT_ = false>
struct Cfg {
    // the C0 blocks live in tensor memory instead of shared memory: they are read
    // back whole every step, at a bandwidth of its own, and leave the shared memory
    // to more signals in flight (one signal per warp or team, 8 x 8 blocks)
    static constexpr bool kTM = TM_;
    // picks from a list of candidates only (the others are masked in the C0 blocks),
    // then a scan of all pairs, whose correlations wait in tensor memory meanwhile.
    // A rank-one update scales its G1 row, and the back substitution runs down the rows.
    static constexpr bool kShort = SHORT_;
    static constexpr bool kTmem = kTM || kShort;
    static constexpr bool kAsc = FAST_ && !SHORT_;
    static constexpr int MW = (RI_ * RJ_ + 31) / 32;   // words of a lane's candidate marks
    static constexpr int TUSED = kTmem ? WARPS_ / 4 * RI_ * RJ_ : 0;
    static constexpr int TCOLS = TUSED <= 64 ? TUSED : TUSED <= 128 ? 128 : TUSED <= 256 ? 256 : 512;   // of a CTA
    static_assert(!kTM || (GL_ >= 32 && RI_ == 8 && RJ_ == 8), "one signal per warp");
    static_assert(!kShort || (GL_ <= 32 && RI_ * RJ_ % 8 == 0 && FAST_ && N1_ > 0 && ORTHO_ == 0 && !TM_), "shortlists");
    static_assert(!kTmem || (WARPS_ % 4 == 0 && (TCOLS & (TCOLS - 1)) == 0 && TCOLS >= 32 && TCOLS * MINB_ <= 512),
                  "tensor memory");
    static constexpr bool kOrtho = ORTHO_ > 0;
    static constexpr int CHAINS = ORTHO_ > 0 ? ORTHO_ : CHAINS_;   // of ||Y||^2 (128: four warps' worth)
    static constexpr int CPL = CHAINS / GL_;                       // per lane
    // a group of 64 lanes is a team of two warps that meet at a named barrier
    static constexpr int TW = GL_ > 32 ? GL_ / 32 : 1;
    // exchange slots between them; or the candidates (32) and the lanes' marks
    static constexpr int XS = TW > 1 ? 16 : kShort ? 32 + up4(GL_ * MW) : 0;
    static_assert(CHAINS == 128 || CPL == 1 || CPL == 2 || CPL == 4, "chains");
    static_assert(TW == 1 || CHAINS == 128, "a team's chains");
    static constexpr int GL = GL_, LI = LI_, LJ = GL_ / LI_, RI = RI_, RJ = RJ_;
    static constexpr int WARPS = WARPS_, MINB = MINB_;
    static constexpr bool kFast = FAST_, kW = W_;
    static constexpr int P1 = P1_, P2 = P2_, N1 = N1_, N2 = N2_, S = S_;
    static constexpr int SPW = GL < 32 ? 32 / GL : 1;   // signals per warp (or team)
    static constexpr int N1P = LI * RI, N2P = LJ * RJ;
    static constexpr int RIP = up4(RI), RJP = up4(RJ);  // padded block lengths (16-byte loads)
    static constexpr int LD1 = LI * RIP, LD2 = LJ * RJP;
    static constexpr int E = RI * RJ;
    // lane stride of the C0 blocks: an odd multiple of 4 floats, so that the 8
    // lanes of a 128-bit load phase hit distinct banks
    static constexpr int EP = (up4(E) / 4) % 2 ? up4(E) : up4(E) + 4;
    static constexpr int CS = kTM ? 2 * RI : up4(RI);   // the winning column's read-back buffer (and its C0)
    // rows per lane and block of the Z stage (Y D2), columns of the W stage
    static constexpr int ZA = P1 ? (P1 / LI) : 4;
    static constexpr int WB = P2 ? (P2 / LJ) : 4;
    static constexpr int SMAX = S ? S : TW > 1 ? 10 : 8;   // unrolled Cholesky rows
    static_assert(N1P * LD1 <= 65536 && N2P * LD2 <= 65536, "16-bit row offsets");
    static_assert(E % 2 == 0 && RI % 2 == 0, "row pairs, 16-byte block stores");
    static_assert((LI & (LI - 1)) == 0 && LI * LJ == GL, "lane grid");
    static_assert(!kW || P2 > 0, "the W stage is compiled for fixed sizes");
    static_assert(!FAST_ || S_ > 0, "steps past the unrolled ones take the generic kernel's forms");
    static_assert(P1 == 0 || (P1 % LI == 0 && ZA % 2 == 0 && P1 % 4 == 0 && P2 % LJ == 0), "fixed sizes");
    static_assert(N1 == 0 || (N1 == N1P && N2 == N2P), "fixed sizes fill the tile");
};

// Shared memory of a CTA, in floats; every region starts 16-byte aligned.
struct Layout {
    int p1s;       // row stride of a staged signal's columns (p1 rounded up to 4)
    int d1, d2, g1, g2, warp0;
    int y, c0, col, xs, rec, lf, iv, yv, sig_stride;   // per signal
    int total;
};

template <class C>
__host__ __device__ inline Layout layout(int p1, int p2, int s, int warps) {
    Layout L;
    L.p1s = up4(p1);
    L.d1 = 0;
    L.d2 = L.d1 + p1 * C::LD1;
    L.g1 = L.d2 + p2 * C::LD2;
    L.g2 = L.g1 + (C::kOrtho ? 0 : C::N1P * C::LD1);
    L.warp0 = L.g2 + (C::kOrtho ? 0 : C::N2P * C::LD2);
    L.y = 0;
    L.c0 = L.y + L.p1s * p2;
    const int z = C::kW ? p2 * C::LD1 : up4(p1) * C::LD2;   // Z or W shares the C0 blocks' place
    const int c = C::kTM ? 0 : C::GL * C::EP;
    L.col = L.c0 + (z > c ? z : c);
    L.xs = L.col + C::CS;
    L.rec = L.xs + C::XS;
    L.lf = L.rec + up4(2 * s);
    L.iv = L.lf + (C::kOrtho ? 0 : up4(s * (s - 1) / 2));
    L.yv = L.iv + (C::kOrtho ? 0 : up4(s));
    int st = L.yv + (C::kOrtho ? 0 : up4(s));
    // neighbouring signals of a warp start 8 banks apart where they read the
    // same offsets together
    while (st % 32 != 8 && st % 32 != 24) st += 4;
    L.sig_stride = st;
    L.total = L.warp0 + warps * 32 / C::GL * st + (C::kTmem ? 4 : 0);   // (the tensor-memory address)
    return L;
}

// ------------------------------------------------------------------ helpers
template <int R>
__device__ __forceinline__ void ld(float (&v)[R], const float* p) {   // 16-byte aligned p
#pragma unroll
    for (int k = 0; k + 4 <= R; k += 4) {
        const float4 t = *reinterpret_cast<const float4*>(p + k);
        v[k] = t.x; v[k + 1] = t.y; v[k + 2] = t.z; v[k + 3] = t.w;
    }
    constexpr int k0 = R & ~3;
    if constexpr (R - k0 >= 2) {
        const float2 t = *reinterpret_cast<const float2*>(p + k0);
        v[k0] = t.x; v[k0 + 1] = t.y;
    }
    if constexpr ((R - k0) & 1) v[R - 1] = p[R - 1];
}
template <int R>
__device__ __forceinline__ void ld2(float (&v)[R], const float* p) {   // 8-byte aligned p, R even
#pragma unroll
    for (int k = 0; k < R; k += 2) {
        const float2 t = *reinterpret_cast<const float2*>(p + k);
        v[k] = t.x; v[k + 1] = t.y;
    }
}
template <int R>
__device__ __forceinline__ void st(float* p, const float (&v)[R]) {   // 16-byte aligned p
#pragma unroll
    for (int k = 0; k + 4 <= R; k += 4)
        *reinterpret_cast<float4*>(p + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    constexpr int k0 = R & ~3;
    if constexpr (R - k0 >= 2) *reinterpret_cast<float2*>(p + k0) = make_float2(v[k0], v[k0 + 1]);
    if constexpr ((R - k0) & 1) p[R - 1] = v[R - 1];
}

// d = a * b + d on two FP32 lanes at once (each half rounds as fmaf)
__device__ __forceinline__ void ffma2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
    const unsigned long long A = ((unsigned long long)__float_as_uint(a1) << 32) | __float_as_uint(a0);
    const unsigned long long B = ((unsigned long long)__float_as_uint(b1) << 32) | __float_as_uint(b0);
    const unsigned long long C = ((unsigned long long)__float_as_uint(d1) << 32) | __float_as_uint(d0);
    unsigned long long D;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(D) : "l"(A), "l"(B), "l"(C));
    d0 = __uint_as_float((unsigned)(D & 0xffffffffu));
    d1 = __uint_as_float((unsigned)(D >> 32));
}
// blk[c * R + r] += a[r] * b[c]
template <int R, int N>
__device__ __forceinline__ void rank1(float (&blk)[R * N], const float (&a)[R], const float (&b)[N]) {
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
        for (int r = 0; r < R; r += 2) ffma2(blk[c * R + r], blk[c * R + r + 1], a[r], a[r + 1], b[c], b[c]);
}
// the same with the pairs along b (blk[r * N + c] += a[r] * b[c]); odd N leaves one scalar column
template <int R, int N>
__device__ __forceinline__ void rank1_rows(float (&blk)[R * N], const float (&a)[R], const float (&b)[N]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int c = 0; c + 2 <= N; c += 2) ffma2(blk[r * N + c], blk[r * N + c + 1], a[r], a[r], b[c], b[c + 1]);
        if constexpr (N & 1) blk[r * N + N - 1] = fmaf(a[r], b[N - 1], blk[r * N + N - 1]);
    }
}
__device__ __forceinline__ float max3abs(float a, float b, float c) {   // NaN operands are ignored
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ unsigned sptr(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sptr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sptr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------ tensor memory
// Each warp reaches the 32 TMEM lanes of its quarter (warp % 4); thread = lane,
// columns hold its floats.
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_ld8(unsigned ta, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(ta));
}
__device__ __forceinline__ void tm_st8(unsigned ta, const float* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"(ta)
                 : "memory");
}
__device__ __forceinline__ void tm_ld32(unsigned ta, float* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]),
          "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]),
          "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
        : "r"(ta));
}

template <int E>
__device__ __forceinline__ void tm_ld_block(unsigned ta, float (&v)[E]) {
#pragma unroll
    for (int k = 0; k + 32 <= E; k += 32) tm_ld32(ta + k, v + k);
#pragma unroll
    for (int k = E & ~31; k < E; k += 8) tm_ld8(ta + k, v + k);
}
template <int E>
__device__ __forceinline__ void tm_st_block(unsigned ta, const float (&v)[E]) {
#pragma unroll
    for (int k = 0; k < E; k += 8) tm_st8(ta + k, v + k);
}

// One pick of a signal: its coefficient, and the offsets of its rows of G1
// (low half) and G2 (high half) in shared memory, one 8-byte load.
struct alignas(8) Rec {
    float x;
    unsigned o;
    __device__ __forceinline__ int o1() const { return (int)(o & 0xffffu); }
    __device__ __forceinline__ int o2() const { return (int)(o >> 16); }
};

// A signal whose final residual correlates with some unpicked pair more strongly
// than this fraction of its weakest greedy score is flagged: plain 2D-OMP might
// have taken a pair that the shortlist missed.
constexpr float kCheckMargin = 0.7f;

// One greedy step's Cholesky row T and the coefficients of the T + 1 picks
// (every lane of the signal holds the same values; `writer` stores them).
// Returns false (state untouched) when the pick is degenerate or !live.
// gram(r): the product of the Gram entries of the new pick and pick r.
// kAsc: back substitution in increasing row order.
template <int T, bool kFast, bool kAsc = kFast, class Gram>
__device__ __forceinline__ bool chol_step(bool live, bool writer, Rec* rec, float* lf, float* iv, float* yv,
                                          Gram gram, float Att, float b, const Rec& pick, float& E) {
    constexpr int NL = T * (T - 1) / 2;
    float L[NL > 0 ? up4(NL) : 1], io[T > 0 ? up4(T) : 1], yo[T > 0 ? up4(T) : 1], am[T > 0 ? T : 1];
    if constexpr (T > 0) {
#pragma unroll
        for (int m = 0; m < T; ++m) am[m] = gram(rec[m]);
#pragma unroll
        for (int k = 0; k < NL; k += 4) {
            const float4 t = *reinterpret_cast<const float4*>(lf + k);
            L[k] = t.x; L[k + 1] = t.y; L[k + 2] = t.z; L[k + 3] = t.w;
        }
#pragma unroll
        for (int k = 0; k < T; k += 4) {
            const float4 t = *reinterpret_cast<const float4*>(iv + k);
            const float4 u = *reinterpret_cast<const float4*>(yv + k);
            io[k] = t.x; io[k + 1] = t.y; io[k + 2] = t.z; io[k + 3] = t.w;
            yo[k] = u.x; yo[k + 1] = u.y; yo[k + 2] = u.z; yo[k + 3] = u.w;
        }
    }
    float w[T > 0 ? T : 1];
    float ww = 0.f, wy = 0.f;
#pragma unroll
    for (int m = 0; m < T; ++m) {
        float v = am[m];
#pragma unroll
        for (int l = 0; l < m; ++l) v = fmaf(-L[m * (m - 1) / 2 + l], w[l], v);
        w[m] = v * io[m];
        ww = fmaf(w[m], w[m], ww);
        wy = fmaf(w[m], yo[m], wy);
    }
    const float d = Att - ww;
    const bool ok = live && d > kPivotRel * Att;
    const float inv = kFast ? rsqrtf(d) : 1.f / sqrtf(d);
    const float yt = (b - wy) * inv;
    float x[T + 1];
    x[T] = yt * inv;
#pragma unroll
    for (int k = T - 1; k >= 0; --k) {
        float v = yo[k];
        if constexpr (kAsc) {
#pragma unroll
            for (int l = k + 1; l < T; ++l) v = fmaf(-L[l * (l - 1) / 2 + k], x[l], v);
            v = fmaf(-w[k], x[T], v);
        } else {
            v = fmaf(-w[k], x[T], v);
#pragma unroll
            for (int l = T - 1; l > k; --l) v = fmaf(-L[l * (l - 1) / 2 + k], x[l], v);
        }
        x[k] = v * io[k];
    }
    if (ok && writer) {
#pragma unroll
        for (int m = 0; m < T; ++m) {
            lf[NL + m] = w[m];
            rec[m].x = x[m];
        }
        iv[T] = inv;
        yv[T] = yt;
        Rec r = pick;
        r.x = x[T];
        rec[T] = r;
    }
    if (ok) E = fmaf(-yt, yt, E);
    return ok;
}

// The same for any t < 32 (the generic kernel's forms): W lanes share the rows of
// the factor, row m with lane m % W, and the unknowns travel by shuffle, so that a
// step is a chain of t shuffles down and t back.  Every chain keeps its order: a
// row takes the unknowns one after the other.  A step that every lane computed by
// itself, loads of the factor in the chain, cost t^2 of them: 64 signals of 8x8 with
// s = 32 picks took 224 us, 105 in the one-warp coder and 90 so; 8000 of them 515, 432 and
// 213.
// All lanes of the warp (of both warps of a team, which agree) call it together;
// `t` is the same for all of them.
template <int W, class Gram>
__device__ __forceinline__ bool chol_step_any(int t, bool live, bool writer, Rec* rec, float* lf, float* iv,
                                              float* yv, Gram gram, float Att, float b, const Rec& pick, float& E) {
    constexpr int R = 32 / W;          // rows per lane
    const int j = threadIdx.x % W;
    const float* row[R];               // own rows of the factor
    float v[R], inv_m[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int m = r * W + j, mm = m < t ? m : 0;   // rows past t run along on row 0
        row[r] = lf + mm * (mm - 1) / 2;
        v[r] = gram(rec[mm]);
        inv_m[r] = iv[mm];
    }
    // ---- row t of the factor: w_m = (a_m - sum_{l < m} L_ml w_l) / L_mm
    float ww = 0.f, wy = 0.f;
#pragma unroll
    for (int q = 0; q < R; ++q)
        for (int i = 0; i < W && q * W + i < t; ++i) {
            const int l = q * W + i;
            const float wl = __shfl_sync(kFull, v[q] * inv_m[q], i, W);
            ww = fmaf(wl, wl, ww);
            wy = fmaf(wl, yv[l], wy);
#pragma unroll
            for (int r = q; r < R; ++r)
                if (r * W + j > l && r * W + j < t) v[r] = fmaf(-row[r][l], wl, v[r]);
        }
    float w[R];
#pragma unroll
    for (int r = 0; r < R; ++r) w[r] = v[r] * inv_m[r];
    const float d = Att - ww;
    const bool ok = live && d > kPivotRel * Att;
    const float inv = 1.f / sqrtf(d);
    const float yt = (b - wy) * inv;
    const float xt = yt * inv;
    // ---- back substitution, pick t first
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int m = r * W + j;
        v[r] = fmaf(-w[r], xt, m < t ? yv[m] : 0.f);
    }
#pragma unroll
    for (int q = R - 1; q >= 0; --q)
        for (int i = min(W, t - q * W) - 1; i >= 0; --i) {
            const int l = q * W + i;
            const float xl = __shfl_sync(kFull, v[q] * inv_m[q], i, W);
            const float* Ll = lf + l * (l - 1) / 2;
#pragma unroll
            for (int r = 0; r <= q; ++r)
                if (r * W + j < l) v[r] = fmaf(-Ll[r * W + j], xl, v[r]);
        }
    if (ok) {
        float* wrow = lf + t * (t - 1) / 2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int m = r * W + j;
            if (m < t) {
                wrow[m] = w[r];
                rec[m].x = v[r] * inv_m[r];
            }
        }
        if (writer) {
            iv[t] = inv;
            yv[t] = yt;
            Rec r = pick;
            r.x = xt;
            rec[t] = r;
        }
        E = fmaf(-yt, yt, E);
    }
    return ok;
}

// G (row i: the products with every position of a lane-block row) of the
// dictionary whose rows are d, by the whole CTA; wide ones in 4 x 4 blocks
// (128 atoms x 64 rows: a plain loop reads two words per multiply-add)
template <int R, int RP, int NP, int LD>
__device__ __forceinline__ void gram(const float* d, int p, float* G) {
    if constexpr (R % 4 == 0 && NP >= 64) {
        for (int e = threadIdx.x; e < NP / 4 * (LD / 4); e += blockDim.x) {
            const int i0 = e / (LD / 4) * 4, pos = e % (LD / 4) * 4;
            const float* di = d + i0 / R * RP + i0 % R;
            float g[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) g[k] = 0.f;
#pragma unroll 2
            for (int r = 0; r < p; ++r) {
                float x[4], y[4];
                ld<4>(x, d + r * LD + pos);
                ld<4>(y, di + r * LD);
                rank1<4, 4>(g, x, y);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float v[4] = {g[4 * k], g[4 * k + 1], g[4 * k + 2], g[4 * k + 3]};
                st<4>(G + (i0 + k) * LD + pos, v);
            }
        }
    } else {
        for (int e = threadIdx.x; e < NP * LD; e += blockDim.x) {
            const int i = e / LD, pos = e % LD;
            const float* di = d + i / R * RP + i % R;
            float g = 0.f;
            for (int r = 0; r < p; ++r) g = fmaf(di[r * LD], d[r * LD + pos], g);
            G[e] = g;
        }
    }
}

// compensated running sum
__device__ __forceinline__ void ksum(float& s, float& c, float v) {
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// ------------------------------------------------------------------- kernel
// Positions 0 .. count-1 (signals, or entries of the index list) are coded in
// units of SPW: warp w of CTA b takes units w gridDim + b, + gridDim warps, ...
// (a small call spreads over the SMs).
// MANY: sparsities past the unrolled steps (a kernel of its own: that path's registers
// cost the others 1 to 2 % in spills).
template <class C, bool MANY>
__global__ void __launch_bounds__(C::WARPS * 32, C::MINB) code_group_kernel(PassArgs a) {
    constexpr int GL = C::GL, LI = C::LI, LJ = C::LJ, RI = C::RI, RJ = C::RJ, E = C::E, SPW = C::SPW;
    constexpr int LD1 = C::LD1, LD2 = C::LD2, RIP = C::RIP, RJP = C::RJP, ZA = C::ZA, WB = C::WB;
    extern __shared__ __align__(16) float sm[];
    const int p1 = C::P1 ? C::P1 : a.p1, p2 = C::P2 ? C::P2 : a.p2;
    const int n1 = C::N1 ? C::N1 : a.n1, n2 = C::N2 ? C::N2 : a.n2;
    const int s = C::S ? C::S : a.s;
    const int pp = p1 * p2;
    const bool error_driven = a.eps2 > 0.f;
    constexpr int TW = C::TW;
    const int warps = blockDim.x >> 5, workers = warps / TW;
    const Layout L = layout<C>(p1, p2, s, warps);
    const int p1s = L.p1s;

    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = GL < 32 ? lane / GL : 0, gl = threadIdx.x % GL;
    const int worker = threadIdx.x / (32 * TW);   // warp or team
    const int li = gl % LI, lj = gl / LI;
    float* D1s = sm + L.d1;    // row a: D1[a, :] in lane blocks
    float* D2s = sm + L.d2;    // row b: D2[b, :] in lane blocks
    float* G1s = sm + L.g1;
    float* G2s = sm + L.g2;
    float* sb = sm + L.warp0 + (threadIdx.x / GL) * L.sig_stride;
    // the lanes of a signal (and the other signals of its warp) meet
    auto sync = [&]() {
        if constexpr (TW == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(worker + 1), "r"(32 * TW) : "memory");
    };
    // whether any signal of the warp (the one of the team, whose lanes agree) goes on
    auto any = [&](bool v) { return TW == 1 ? __any_sync(kFull, v) != 0 : v; };
    float* Ys = sb + L.y;
    float* Zs = sb + L.c0;     // Z (rows a) or W (rows b), then the C0 blocks
    float* C0s = sb + L.c0;
    float* myc0 = C0s + gl * C::EP;
    float* col = sb + L.col;
    Rec* rec = reinterpret_cast<Rec*>(sb + L.rec);
    float* lf = sb + L.lf;
    float* iv = sb + L.iv;
    float* yv = sb + L.yv;

    // ---- dictionaries in lane-block rows, then their Gram matrices (each
    // entry one FMA chain over the rows, as the Gram kernels form it: no
    // separate launch, and no difference)
    for (int e = threadIdx.x; e < p1 * LD1; e += blockDim.x) {
        const int r = e / LD1, pos = e % LD1, off = pos % RIP, i = (pos / RIP) * RI + off;
        D1s[e] = (off < RI && i < n1) ? a.D1[r + p1 * i] : 0.f;
    }
    for (int e = threadIdx.x; e < p2 * LD2; e += blockDim.x) {
        const int r = e / LD2, pos = e % LD2, off = pos % RJP, j = (pos / RJP) * RJ + off;
        D2s[e] = (off < RJ && j < n2) ? a.D2[r + p2 * j] : 0.f;
    }
    // a signal's records start valid: a finished signal's lanes run along with
    // the others of the warp on whatever its records hold
    for (int l = gl; l < s; l += GL) rec[l] = Rec{0.f, 0u};
    int* cands = reinterpret_cast<int*>(sb + L.xs);          // shortlists only
    unsigned* marks = reinterpret_cast<unsigned*>(sb + L.xs + 32);
    if constexpr (C::kShort)
        for (int m = 0; m < C::MW; ++m) marks[gl * C::MW + m] = 0u;
    __syncthreads();
    if constexpr (!C::kOrtho) {
        gram<RI, RIP, C::N1P, LD1>(D1s, p1, G1s);
        gram<RJ, RJP, C::N2P, LD2>(D2s, p2, G2s);
        __syncthreads();
    }

    // tensor memory of the CTA, and this warp's place in it
    unsigned tbase = 0, tmine = 0;
    unsigned* tslot = reinterpret_cast<unsigned*>(sm + L.total - 4);
    if constexpr (C::kTmem) {
        if (w == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sptr(tslot)),
                         "r"(C::TCOLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tbase = *static_cast<volatile unsigned*>(tslot);
        tmine = tbase + ((unsigned)(w % 4) << 21) + (unsigned)(w / 4 * E);
    }

    const long long count = a.idx ? (long long)*a.idx_count : a.N;
    const long long units = (count + SPW - 1) / SPW;
    const long long ustep = (long long)gridDim.x * workers;
    long long u = (long long)worker * gridDim.x + blockIdx.x;   // next unit

    // signals start on 16-byte boundaries and columns stay 16-byte aligned
    const bool vec = (reinterpret_cast<uintptr_t>(a.Y) & 15u) == 0 && (C::P1 ? true : p1 % 4 == 0);
    const unsigned inv_p1 = (65536u + p1 - 1) / p1;   // e / p1 = e inv_p1 >> 16 for e < 1024
    auto fetch = [&](long long k) {   // this lane group's signal k into Ys (cp.async)
        const float* src = a.Y + (size_t)k * pp;
        if (vec) {
            for (int e = gl * 4; e < pp; e += GL * 4) cp16(Ys + e, src + e);
        } else {
            for (int e = gl; e < pp; e += GL) {
                const int b = (int)((unsigned)e * inv_p1 >> 16);
                cp4(Ys + b * p1s + (e - b * p1), src + e);
            }
        }
        if constexpr (C::kShort)
            for (int c = gl; c < a.cand_k; c += GL)
                cp4(reinterpret_cast<float*>(cands + c),
                    reinterpret_cast<const float*>(a.cand + (size_t)k * a.cand_ld + c));
    };

    float es = 0.f, ec = 0.f;      // this lane's residual-energy sum (compensated)
    // the position of this group in the next unit; -1 when it has none.  The
    // warp's units end when all groups have none.
    auto next_pos = [&]() -> long long {
        const long long p = u < units ? u * SPW + grp : count;
        u += ustep;
        return p < count ? p : -1;
    };

    long long pos = next_pos();
    if (pos >= 0) fetch(a.idx ? (long long)a.idx[pos] : pos);
    while (any(pos >= 0)) {
        const bool act = pos >= 0;
        const long long ko = !act ? 0 : (a.idx && !a.idx_compact) ? (long long)a.idx[pos] : pos;
        cp_wait();
        sync();
        if constexpr (C::kShort) {   // a mark for each candidate, with the lane that owns its entry
            for (int c = gl; c < (act ? a.cand_k : 0); c += GL) {
                const int q = cands[c], i = q % C::N1, j = q / C::N1, e = j % RJ * RI + i % RI;
                if (q >= 0 && j < C::N2)
                    atomicOr(marks + (j / RJ * LI + i / RI) * C::MW + e / 32, 1u << (e % 32));
            }
        }
        // ---- ||Y||^2: the strided partial sums of the one-signal-per-warp (or half
        // warp) coders (this lane takes CPL of them) and their combining tree
        float part[C::CPL];
#pragma unroll
        for (int v = 0; v < C::CPL; ++v) part[v] = 0.f;
        if (act) {
#pragma unroll
            for (int v = 0; v < C::CPL; ++v)
                for (int e = gl + GL * v; e < pp; e += C::CHAINS) {
                    int at = e;
                    if (!(C::P1 ? true : p1 % 4 == 0)) {
                        const int b = (int)((unsigned)e * inv_p1 >> 16);
                        at = b * p1s + (e - b * p1);
                    }
                    part[v] = fmaf(Ys[at], Ys[at], part[v]);
                }
        }
        float ss;
        if constexpr (C::CHAINS == 128) {
            // four warps' sums, added in order; chain GL v + gl belongs to lane
            // (GL v + gl) % 32 of warp (GL v + gl) / 32
            float ws[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if constexpr (GL == 16) ws[v] = part[2 * v] + part[2 * v + 1];
                else if constexpr (GL == 32) ws[v] = part[v];
                else ws[v] = part[v / 2];
#pragma unroll
                for (int o = GL < 32 ? GL / 2 : 16; o > 0; o >>= 1) ws[v] += __shfl_xor_sync(kFull, ws[v], o);
            }
            if constexpr (TW > 1) {   // this warp has warps w % 2 and w % 2 + 2
                const int h = w % TW;
                float* xs = sb + L.xs + 8;
                if (lane == 0) {
                    xs[h] = ws[0];
                    xs[h + 2] = ws[2];
                }
                sync();
#pragma unroll
                for (int v = 0; v < 4; ++v) ws[v] = xs[v];
            }
            ss = ((ws[0] + ws[1]) + ws[2]) + ws[3];
        } else {
            if constexpr (C::CPL == 4) ss = (part[0] + part[2]) + (part[1] + part[3]);
            else if constexpr (C::CPL == 2) ss = part[0] + part[1];
            else ss = part[0];
#pragma unroll
            for (int o = GL / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(kFull, ss, o);
        }
        const bool finite = act && isfinite(ss);
        bool go = finite && !(error_driven && ss <= a.eps2);

        // ---- first contraction into shared memory: Z = Y D2 (lane (li, lj):
        // rows li ZA.., columns of block lj) or W = D1^T Y (rows of block li,
        // columns b of lane lj)
        if constexpr (!C::kW) {
            for (int a0 = li * ZA; a0 < (C::P1 ? C::P1 : p1); a0 += LI * ZA) {
                float z[ZA * RJ];
#pragma unroll
                for (int e = 0; e < ZA * RJ; ++e) z[e] = 0.f;
#pragma unroll 4
                for (int b = 0; b < p2; ++b) {
                    float y[ZA], d[RJ];
                    if constexpr (ZA % 4 == 0) ld<ZA>(y, Ys + b * p1s + a0);
                    else ld2<ZA>(y, Ys + b * p1s + a0);
                    ld<RJ>(d, D2s + b * LD2 + lj * RJP);
                    rank1_rows<ZA, RJ>(z, y, d);
                }
#pragma unroll
                for (int r = 0; r < ZA; ++r) {
                    if (C::P1 || a0 + r < p1) {
                        float v[RJ];
#pragma unroll
                        for (int c = 0; c < RJ; ++c) v[c] = z[r * RJ + c];
                        st<RJ>(Zs + (a0 + r) * LD2 + lj * RJP, v);
                    }
                }
            }
        } else {
            float z[RI * WB];
#pragma unroll
            for (int e = 0; e < RI * WB; ++e) z[e] = 0.f;
#pragma unroll 4
            for (int r = 0; r < p1; ++r) {
                float d[RI], y[WB];
                ld<RI>(d, D1s + r * LD1 + li * RIP);
#pragma unroll
                for (int c = 0; c < WB; ++c) y[c] = Ys[(lj + LJ * c) * p1s + r];
                rank1<RI, WB>(z, d, y);
            }
#pragma unroll
            for (int c = 0; c < WB; ++c) {
                float v[RI];
#pragma unroll
                for (int r = 0; r < RI; ++r) v[r] = z[c * RI + r];
                st<RI>(Zs + (lj + LJ * c) * LD1 + li * RIP, v);
            }
        }
        sync();
        // Y is consumed: fetch the next unit's signals
        const long long pos_next = next_pos();
        if (pos_next >= 0) fetch(a.idx ? (long long)a.idx[pos_next] : pos_next);

        // ---- C0 on the lane's RI x RJ block (flat index c * RI + r)
        float sc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) sc[e] = 0.f;
        if constexpr (!C::kW) {
#pragma unroll 2
            for (int r = 0; r < p1; ++r) {
                float x[RI], v[RJ];
                ld<RI>(x, D1s + r * LD1 + li * RIP);
                ld<RJ>(v, Zs + r * LD2 + lj * RJP);
                rank1<RI, RJ>(sc, x, v);
            }
        } else {
#pragma unroll 2
            for (int b = 0; b < p2; ++b) {
                float x[RI], v[RJ];
                ld<RI>(x, Zs + b * LD1 + li * RIP);
                ld<RJ>(v, D2s + b * LD2 + lj * RJP);
                rank1<RI, RJ>(sc, x, v);
            }
        }
        if constexpr (C::N1 == 0) {   // entries past the dictionaries never win
#pragma unroll
            for (int c = 0; c < RJ; ++c)
#pragma unroll
                for (int r = 0; r < RI; ++r)
                    if (li * RI + r >= n1 || lj * RJ + c >= n2) sc[c * RI + r] = __int_as_float(0x7fc00000);
        }
        sync();   // every lane has read Z: its place takes the C0 blocks
        if constexpr (C::kTmem) {
            tm_st_block<E>(tmine, sc);
            tm_wait_st();
        }
        if constexpr (C::kShort) {   // only the candidates stay
#pragma unroll
            for (int m = 0; m < C::MW; ++m) {
                const unsigned mk = marks[gl * C::MW + m];
                marks[gl * C::MW + m] = 0u;
#pragma unroll
                for (int e = 32 * m; e < (32 * m + 32 < E ? 32 * m + 32 : E); ++e)
                    if (!((mk >> (e - 32 * m)) & 1u)) sc[e] = __int_as_float(0x7fc00000);
            }
        }
        if constexpr (!C::kTM) {
            st<E>(myc0, sc);
            sync();
        }

        // a pick's coefficient goes to one of its two rows
        auto scale = [&](float (&x)[RI], float (&v)[RJ], float f) {
            if constexpr (C::kShort) {
#pragma unroll
                for (int r = 0; r < RI; ++r) x[r] *= -f;
            } else {
#pragma unroll
                for (int c = 0; c < RJ; ++c) v[c] *= -f;
            }
        };
        // ---- greedy steps
        int cnt = 0;
        float E2 = ss, weakest = __int_as_float(0x7f800000);   // (the smallest score of a pick)
        float* masked = nullptr;
#pragma unroll 1
        for (int t = 0; t < s; ++t) {
            const bool live = go && !(error_driven && E2 <= a.eps2);
            if (!any(live)) break;
            if (t > 0) {
                // the last pick leaves the search: its owner masks it here, after
                // every lane has read the entry
                if constexpr (C::kTM) {
                    __syncwarp();
                    tm_ld_block<E>(tmine, sc);
                    tm_wait_ld();
                } else {
                    if (masked) *masked = __int_as_float(0x7fc00000);
                    ld<E>(sc, myc0);
                }
                if constexpr (!C::kOrtho) {
                    // one ahead of the loop: its load hides behind a rank-one update (12x12: 326 -> 318 us)
                    Rec next = rec[0];
#pragma unroll 1
                    for (int l = 0; l < t; ++l) {
                        const Rec r = next;
                        if (l + 1 < s) next = rec[l + 1];
                        float x[RI], v[RJ];
                        ld<RI>(x, G1s + r.o1() + li * RIP);
                        ld<RJ>(v, G2s + r.o2() + lj * RJP);
                        scale(x, v, r.x);
                        rank1<RI, RJ>(sc, x, v);
                    }
                }
            }
            // the lane's largest |score|, its first column, by column maxima
            float best = 0.f;
            int bc = 0;
#pragma unroll
            for (int c = 0; c < RJ; ++c) {
                float m = 0.f;
#pragma unroll
                for (int r = 0; r < RI; r += 2) m = max3abs(m, sc[c * RI + r], sc[c * RI + r + 1]);
                if (m > best) { best = m; bc = c; }
            }
            // the signal's largest and its smallest (column, row block)
            float M = best;
            int key = (lj * RJ + bc) * LI + li;
#pragma unroll
            for (int o = GL < 32 ? GL / 2 : 16; o > 0; o >>= 1) {
                const float mo = __shfl_xor_sync(kFull, M, o);
                const int ko2 = __shfl_xor_sync(kFull, key, o);
                if (mo > M || (mo == M && ko2 < key)) { M = mo; key = ko2; }
            }
            if constexpr (TW > 1) {   // two slots per parity of t: no barrier before their next use
                float* xs = sb + L.xs + 4 * (t & 1);
                if (lane == 0) *reinterpret_cast<float2*>(xs + 2 * (w % TW)) = make_float2(M, __int_as_float(key));
                sync();
                const float4 v = *reinterpret_cast<const float4*>(xs);
                const int k0 = __float_as_int(v.y), k1 = __float_as_int(v.w);
                const bool first = v.x > v.z || (v.x == v.z && k0 < k1);
                M = first ? v.x : v.z;
                key = first ? k0 : k1;
            }
            const bool pick = live && M != 0.f;
            const int jt = key / LI, lio = key % LI;
            // the owner lane's column, and the first row that holds M
            const int owner = lio + LI * (jt / RJ);
            const bool owner_warp = TW == 1 || w % TW == owner / 32;
            float c8[8];   // tensor memory: the C0 values of that column
            if constexpr (C::kTM) {
                if (owner_warp) {
                    __syncwarp();
                    tm_ld8(tmine + jt % RJ * RI, c8);
                    tm_wait_ld();
                    if (gl == owner)
#pragma unroll
                        for (int r = 0; r < RI; r += 4)
                            *reinterpret_cast<float4*>(col + RI + r) =
                                make_float4(c8[r], c8[r + 1], c8[r + 2], c8[r + 3]);
                }
            }
            if (gl == owner) {
#pragma unroll
                for (int c = 0; c < RJ; ++c)
                    if (bc == c) {
                        float v[RI];
#pragma unroll
                        for (int r = 0; r < RI; ++r) v[r] = sc[c * RI + r];
                        st<RI>(col, v);
                    }
            }
            sync();
            unsigned rows = 0;
#pragma unroll
            for (int r0 = 0; r0 < RI; r0 += GL) {
                constexpr int GW = GL < 32 ? GL : 32;
                const int r = r0 + lane % GW;
                const bool eq = r < RI && fabsf(col[r]) == M;
                const unsigned bal = __ballot_sync(kFull, eq);
                rows |= ((bal >> (GW * grp)) & (unsigned)((1ull << GW) - 1ull)) << r0;
            }
            const int rt = rows ? __ffs(rows) - 1 : 0;
            const int it = lio * RI + rt;
            float* cq = C::kTM ? col + RI + rt : C0s + owner * C::EP + (jt % RJ) * RI + rt;
            const float b = *cq;
            if constexpr (C::kTM) {   // the pick leaves the search: masked in its owner's lane
                if (owner_warp && pick) {
                    __syncwarp();
#pragma unroll
                    for (int r = 0; r < 8; ++r)
                        if (gl == owner && r == rt) c8[r] = __int_as_float(0x7fc00000);
                    tm_st8(tmine + jt % RJ * RI, c8);
                    tm_wait_st();
                }
            }
            const int c1 = lio * RIP + rt, c2 = (jt / RJ) * RJP + jt % RJ;
            const Rec pk{0.f, (unsigned)(it * LD1) | ((unsigned)(jt * LD2) << 16)};
            const float Att = C::kOrtho ? 1.f : G1s[it * LD1 + c1] * G2s[jt * LD2 + c2];
            const bool wr = gl == 0;
            masked = pick && gl == owner ? cq : nullptr;
            bool ok = false;
            if constexpr (C::kOrtho) {
                ok = pick;
                if (ok) {
                    if (wr) rec[t] = Rec{b, pk.o};
                    E2 = fmaf(-b, b, E2);
                }
            } else {
            auto gram = [&](const Rec& r) { return G1s[r.o1() + c1] * G2s[r.o2() + c2]; };
            auto step = [&](auto tc) {
                ok = chol_step<decltype(tc)::value, C::kFast, C::kAsc>(pick, wr, rec, lf, iv, yv, gram, Att, b, pk, E2);
            };
            switch (t) {
                case 0: step(std::integral_constant<int, 0>{}); break;
                case 1: if constexpr (C::SMAX > 1) step(std::integral_constant<int, 1>{}); break;
                case 2: if constexpr (C::SMAX > 2) step(std::integral_constant<int, 2>{}); break;
                case 3: if constexpr (C::SMAX > 3) step(std::integral_constant<int, 3>{}); break;
                case 4: if constexpr (C::SMAX > 4) step(std::integral_constant<int, 4>{}); break;
                case 5: if constexpr (C::SMAX > 5) step(std::integral_constant<int, 5>{}); break;
                case 6: if constexpr (C::SMAX > 6) step(std::integral_constant<int, 6>{}); break;
                case 7: if constexpr (C::SMAX > 7) step(std::integral_constant<int, 7>{}); break;
                case 8:
                    if constexpr (C::SMAX > 8) {
                        step(std::integral_constant<int, 8>{});
                        break;
                    }
                    [[fallthrough]];
                case 9:
                    if constexpr (C::SMAX > 9) {
                        step(std::integral_constant<int, 9>{});
                        break;
                    }
                    [[fallthrough]];
                default:
                    if constexpr (MANY)
                        ok = chol_step_any<(GL < 32 ? GL : 32)>(t, pick, wr, rec, lf, iv, yv, gram, Att, b, pk, E2);
                    break;
            }
            }
            if (ok) cnt = t + 1;
            if (C::kShort && ok) weakest = fminf(weakest, M);
            go = ok;
            sync();   // the step's state is visible
        }

        // ---- the scan after a full shortlist code: the largest correlation of the
        // residual with a pair that was not picked
        float left = 0.f;
        if constexpr (C::kShort) {
            if (any(act && cnt == s)) {
                __syncwarp();
                tm_ld_block<E>(tmine, sc);
                tm_wait_ld();
                unsigned picked[C::MW] = {};
                Rec next = rec[0];
#pragma unroll 1
                for (int l = 0; l < s; ++l) {
                    const Rec r = next;
                    if (l + 1 < s) next = rec[l + 1];
                    float x[RI], v[RJ];
                    ld<RI>(x, G1s + r.o1() + li * RIP);
                    ld<RJ>(v, G2s + r.o2() + lj * RJP);
                    scale(x, v, r.x);
                    rank1<RI, RJ>(sc, x, v);
                    const int i = r.o1() / LD1, j = r.o2() / LD2, e = j % RJ * RI + i % RI;
#pragma unroll
                    for (int m = 0; m < C::MW; ++m)
                        if (i / RI == li && j / RJ == lj && e / 32 == m) picked[m] |= 1u << (e % 32);
                }
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if ((picked[e / 32] >> (e % 32)) & 1u) sc[e] = 0.f;
#pragma unroll
                for (int e = 0; e < E; e += 2) left = max3abs(left, sc[e], sc[e + 1]);
#pragma unroll
                for (int o = GL / 2; o > 0; o >>= 1) left = fmaxf(left, __shfl_xor_sync(kFull, left, o));
            }
        }

        // ---- the code
        if (act) {
            if (a.support)
                for (int l = gl; l < s; l += GL) {
                    const Rec r = rec[l];
                    a.support[(size_t)ko * s + l] = l < cnt ? r.o1() / LD1 + n1 * (r.o2() / LD2) : -1;
                    a.coef[(size_t)ko * s + l] = l < cnt ? r.x : 0.f;
                }
            if (gl == 0) {
                const float e = fmaxf(E2, 0.f);
                if (a.nnz) a.nnz[ko] = cnt;
                if (a.res_energy) a.res_energy[ko] = finite || C::kShort ? e : __int_as_float(0x7fc00000);
                if constexpr (C::kShort) {   // (a flagged signal is coded again)
                    a.flag[ko] = !finite || (cnt == s && left > kCheckMargin * weakest) ? 1 : 0;
                } else {
                    if (finite) ksum(es, ec, e);
                    else record_error(a.err, SDL_ERR_NONFINITE);
                }
            }
        }
        sync();   // records are read before the next unit writes them
        pos = pos_next;
    }

    if constexpr (C::kTmem) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (w == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(C::TCOLS) : "memory");
        }
    }

    // ---- residual energies of this CTA's signals, lanes and warps in a fixed
    // order; the slots past the grid are cleared
    if (a.esum) {
        __syncthreads();
        double* red = reinterpret_cast<double*>(sm);
        double d = (double)es - (double)ec;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(kFull, d, o);
        if (lane == 0) red[w] = d;
        __syncthreads();
        if (threadIdx.x == 0) {
            double tot = 0.0;
            for (int v = 0; v < warps; ++v) tot += red[v];
            for (int slot = blockIdx.x; slot < a.esum_slots; slot += gridDim.x) {
                a.esum[2 * slot] = slot == (int)blockIdx.x ? tot : 0.0;
                a.esum[2 * slot + 1] = 0.0;
            }
        }
    }
}

// Launch on at most max_grid CTAs (0: no limit).  Large signals leave room for
// fewer warps per CTA; SDL_ERR_UNSUPPORTED when not even one fits (the caller
// takes the generic kernel).
template <class C>
int launch(const PassArgs& a, cudaStream_t st, int num_sms, int max_grid) {
    constexpr size_t kSmMax = 227 * 1024, kSmTotal = 228 * 1024;
    int warps = C::WARPS;
    size_t bytes;
    while ((bytes = sizeof(float) * (size_t)layout<C>(a.p1, a.p2, a.s, warps).total) > kSmMax && warps > C::TW)
        warps -= C::TW;
    if (bytes > kSmMax) return SDL_ERR_UNSUPPORTED;
    auto kern = code_group_kernel<C, false>;
    if constexpr (C::S == 0 && !C::kOrtho)
        if (a.s > C::SMAX) kern = code_group_kernel<C, true>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmMax) != cudaSuccess)
        return SDL_ERR_CUDA;
    // the registers allow MINB CTAs per SM (launch bounds); 1 KB per CTA is reserved
    const int bps = std::max(1, std::min<int>(C::MINB, (int)(kSmTotal / (bytes + 1024))));
    const long long units = (a.N + C::SPW - 1) / C::SPW;
    long long grid = std::max<long long>(1, std::min<long long>(units, (long long)num_sms * bps));
    if (max_grid > 0) grid = std::min<long long>(grid, max_grid);
    kern<<<(int)grid, warps * 32, bytes, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? SDL_OK : SDL_ERR_CUDA;
}

}  // namespace group
}  // namespace sdl
