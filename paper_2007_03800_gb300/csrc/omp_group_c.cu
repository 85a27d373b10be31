// The lane-group coder for wide second dictionaries (n2 up to 128): 16 or 32 lanes
// per signal, or a team of two warps, in the arithmetic of the generic kernel's
// four-warp teams (whose other warps waited while one did the Cholesky step).
// 50 000 x 16x64, 32x128 pairs, s = 10: 2067 us there (28 300 warp instructions per
// signal); 1721 us with teams of two warps and the C0 blocks in shared memory, which
// then holds 5 signals per SM; 1406 us with them in tensor memory (6 teams of 168
// registers; 8 teams of 128 spill: 1530 us), 52 % of the issue slots and of the
// shared-memory bandwidth in use, the rest fixed-latency dependencies.
#include "omp_group.cuh"

namespace sdl {
namespace {

template <int GL, int LI, int RI, int RJ, int W, int M, int P1 = 0, int P2 = 0, int N1 = 0, int N2 = 0, bool TM = false>
using Wide = group::Cfg<GL, LI, RI, RJ, W, M, false, false, P1, P2, N1, N2, 0, 0, 128, TM>;

}  // namespace

int launch_code_group_cols(const PassArgs& a, cudaStream_t st, int num_sms) {
    const int n1 = a.n1, n2 = a.n2;
    if (n1 <= 16 && n2 <= 64) return group::launch<Wide<16, 2, 8, 8, 8, 2>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 64) return group::launch<Wide<32, 4, 8, 8, 8, 2>>(a, st, num_sms, 0);
    if (n1 <= 16 && n2 <= 128) return group::launch<Wide<32, 2, 8, 8, 8, 2>>(a, st, num_sms, 0);
    // the hyperspectral-shaped problem with its sizes fixed (as in the generic kernel's
    // dispatch): 8000 signals, us fixed | run-time sizes, s = 4 to 32: s = 8 204 | 216, s = 10
    // 251 | 264, s = 16 679 | 694; 64 signals, s = 10 35 | 37
    if (a.p1 == 16 && a.p2 == 64 && n1 == 32 && n2 == 128)
        return group::launch<Wide<64, 4, 8, 8, 12, 1, 16, 64, 32, 128, true>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 128) return group::launch<Wide<64, 4, 8, 8, 12, 1, 0, 0, 0, 0, true>>(a, st, num_sms, 0);
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace sdl
