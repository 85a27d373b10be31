// The lane-group coder at the compiled pair shapes (fixed sizes, the compiled
// tilings' arithmetic), with either order of the two contractions.
#include "omp_group.cuh"

namespace sdl {
namespace {

// <lanes per signal, LI, RI, RJ, warps per CTA, CTAs per SM, ...>
template <bool W> using G8x16s4 = group::Cfg<8, 2, 8, 4, 8, 3, true, W, 8, 8, 16, 16, 4>;
template <bool W> using G12x24s6 = group::Cfg<8, 2, 12, 6, 8, 2, true, W, 12, 12, 24, 24, 6>;
template <bool W> using G16x32s8 = group::Cfg<16, 4, 8, 8, 8, 2, true, W, 16, 16, 32, 32, 8>;

template <bool W>
int run(const PassArgs& a, cudaStream_t st, int num_sms, int max_grid) {
    if (a.p1 == 8 && a.p2 == 8 && a.n1 == 16 && a.n2 == 16 && a.s == 4)
        return group::launch<G8x16s4<W>>(a, st, num_sms, max_grid);
    if (a.p1 == 12 && a.p2 == 12 && a.n1 == 24 && a.n2 == 24 && a.s == 6)
        return group::launch<G12x24s6<W>>(a, st, num_sms, max_grid);
    if (a.p1 == 16 && a.p2 == 16 && a.n1 == 32 && a.n2 == 32 && a.s == 8)
        return group::launch<G16x32s8<W>>(a, st, num_sms, max_grid);
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace

int launch_code_group_fixed(const PassArgs& a, bool w_first, cudaStream_t st, int num_sms, int max_grid) {
    return w_first ? run<true>(a, st, num_sms, max_grid) : run<false>(a, st, num_sms, max_grid);
}

}  // namespace sdl
