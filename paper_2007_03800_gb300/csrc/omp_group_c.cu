// The lane-group coder for wide second dictionaries (n2 up to 128): 16 or 32 lanes
// per signal, or a team of two warps, in the arithmetic of the generic kernel's
// four-warp teams.
#include "omp_group.cuh"

namespace sdl {
namespace {

template <int GL, int LI, int RI, int RJ, int W, int M, int P1 = 0, int P2 = 0, int N1 = 0, int N2 = 0>
using Wide = group::Cfg<GL, LI, RI, RJ, W, M, false, false, P1, P2, N1, N2, 0, 0, 128>;

}  // namespace

int launch_code_group_cols(const PassArgs& a, cudaStream_t st, int num_sms) {
    const int n1 = a.n1, n2 = a.n2;
    if (n1 <= 16 && n2 <= 64) return group::launch<Wide<16, 2, 8, 8, 8, 2>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 64) return group::launch<Wide<32, 4, 8, 8, 8, 2>>(a, st, num_sms, 0);
    if (n1 <= 16 && n2 <= 128) return group::launch<Wide<32, 2, 8, 8, 8, 2>>(a, st, num_sms, 0);
    // the hyperspectral-shaped problem with its sizes fixed
    if (a.p1 == 16 && a.p2 == 64 && n1 == 32 && n2 == 128)
        return group::launch<Wide<64, 4, 8, 8, 10, 1, 16, 64, 32, 128>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 128) return group::launch<Wide<64, 4, 8, 8, 10, 1>>(a, st, num_sms, 0);
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace sdl
