// The lane-group coder with run-time sizes (the generic kernel's arithmetic):
// tiles of at most 24 x 24 atom pairs.
#include "omp_group.cuh"

namespace sdl {

// The smallest tile that holds n1 x n2 pairs: the scan and the rank-one updates
// run over the whole tile, padding included.
int launch_code_group_any(const PassArgs& a, cudaStream_t st, int num_sms) {
    const int n1 = a.n1, n2 = a.n2;
    if (n1 <= 16 && n2 <= 16) return group::launch<group::Cfg<8, 2, 8, 4, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 16 && n2 <= 24) return group::launch<group::Cfg<8, 2, 8, 6, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 24 && n2 <= 16) return group::launch<group::Cfg<8, 2, 12, 4, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 20 && n2 <= 24) return group::launch<group::Cfg<8, 2, 10, 6, 8, 2, false, false>>(a, st, num_sms, 0);
    if (n1 <= 24 && n2 <= 24) return group::launch<group::Cfg<8, 2, 12, 6, 8, 2, false, false>>(a, st, num_sms, 0);
    return launch_code_group_wide(a, st, num_sms);
}

}  // namespace sdl
