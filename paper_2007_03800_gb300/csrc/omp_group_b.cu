// The lane-group coder with run-time sizes: tiles of up to 32 x 32 atom pairs.
#include "omp_group.cuh"

namespace sdl {

int launch_code_group_wide(const PassArgs& a, cudaStream_t st, int num_sms) {
    const int n1 = a.n1, n2 = a.n2;
    if (n1 <= 16 && n2 <= 32) return group::launch<group::Cfg<8, 2, 8, 8, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 16) return group::launch<group::Cfg<8, 2, 16, 4, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 24 && n2 <= 32) return group::launch<group::Cfg<16, 4, 6, 8, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 24) return group::launch<group::Cfg<16, 4, 8, 6, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 32 && n2 <= 32) return group::launch<group::Cfg<16, 4, 8, 8, 8, 2, false, false>>(a, st, num_sms, 0);
    return launch_code_group_cols(a, st, num_sms);
}

}  // namespace sdl
