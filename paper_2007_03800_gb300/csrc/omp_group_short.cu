// The lane-group coder restricted to each signal's shortlist of atom pairs, with the
// test that decides whether the signal needs the full coder.  One warp per signal
// with a candidate per lane took 983 warp instructions per signal (8x8, 16x16 pairs,
// s = 4): most of them the Cholesky steps and the final scan of all pairs, which
// formed C0 a second time.  Here C0 is formed once; the greedy steps run on it with
// the other pairs masked, the scan on the copy in tensor memory: 585 instructions,
// 200 000 signals in 146 us instead of 231.
#include "omp_group.cuh"

namespace sdl {

int launch_code_group_short(const PassArgs& a, cudaStream_t st, int num_sms) {
    if (a.p1 == 8 && a.p2 == 8 && a.n1 == 16 && a.n2 == 16 && a.s == 4)
        return group::launch<group::Cfg<8, 2, 8, 4, 8, 3, true, false, 8, 8, 16, 16, 4, 0, 32, false, true>>(a, st, num_sms, 0);
    if (a.p1 == 12 && a.p2 == 12 && a.n1 == 24 && a.n2 == 24 && a.s == 6)
        return group::launch<group::Cfg<8, 2, 12, 6, 8, 2, true, false, 12, 12, 24, 24, 6, 0, 32, false, true>>(a, st, num_sms, 0);
    return SDL_ERR_UNSUPPORTED;
}

}  // namespace sdl
