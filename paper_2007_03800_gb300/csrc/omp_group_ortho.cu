// The lane-group coder for orthonormal dictionaries (T_s of D1^T Y D2), and the
// partial sums of a learning pass from its codes in the fused coder's order.
#include "omp_group.cuh"

namespace sdl {
namespace {

// square shapes compiled ahead: ||Y||^2 in the 16 chains of their half-warp coder
template <int P> struct Square;
template <> struct Square<8> { using type = group::Cfg<8, 2, 4, 2, 8, 4, false, false, 8, 8, 8, 8, 0, 16>; };
template <> struct Square<12> { using type = group::Cfg<8, 2, 6, 3, 8, 4, false, false, 12, 12, 12, 12, 0, 16>; };
template <> struct Square<16> { using type = group::Cfg<8, 2, 8, 4, 8, 3, false, false, 16, 16, 16, 16, 0, 16>; };

bool square(const PassArgs& a) {
    return a.p1 == a.p2 && a.s <= 16 && (a.p1 == 8 || a.p1 == 12 || a.p1 == 16);
}

}  // namespace

// a.n1 = a.p1, a.n2 = a.p2 (up to 32), any alignment
int launch_ortho_group(const PassArgs& a, cudaStream_t st, int num_sms, int max_grid) {
    if (square(a)) {
        if (a.p1 == 8) return group::launch<Square<8>::type>(a, st, num_sms, max_grid);
        if (a.p1 == 12) return group::launch<Square<12>::type>(a, st, num_sms, max_grid);
        return group::launch<Square<16>::type>(a, st, num_sms, max_grid);
    }
    if (a.p1 <= 16 && a.p2 <= 16)
        return group::launch<group::Cfg<8, 2, 8, 4, 8, 2, false, false, 0, 0, 0, 0, 0, 32>>(a, st, num_sms, max_grid);
    if (a.p1 <= 32 && a.p2 <= 32)
        return group::launch<group::Cfg<16, 4, 8, 8, 8, 2, false, false, 0, 0, 0, 0, 0, 32>>(a, st, num_sms, max_grid);
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace sdl
