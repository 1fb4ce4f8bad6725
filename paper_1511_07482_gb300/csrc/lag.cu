// FP32 lag kernels (lag.cuh).
#include "lag.cuh"

namespace kdefft {
int lag_table_size(int d, int R, bool dbl) {
    if (R < 0 || R > lag_rmax(d, dbl)) return 0;
    const int Re = (R + 1) & ~1;   // even instantiations
    long long c = 1;
    for (int i = 1; i <= d; ++i) c = c * (Re + i) / i;
    return (int)c;
}

bool lag_single_form(int d, int R, int nv, int nsig) {
    if (d < 1 || d > MAXD || nv < 0 || nv > 2 || nsig < 1 || nsig > MAXSIG) return false;
    if (R == 0) return nv > 0;
    return R == 2 || (R == 4 && nv == 0 && nsig == 1);
}

int lag_covs(int R, int nv, int n) { return n > 2 ? MAXSIG : n < 2 && R == 2 && nv == 0 ? 1 : 2; }

int lag_sums(int d, int R, int nv, bool dbl, int covs) {
    if (nv < 0) return 2;
    int members = R > 0 ? 1 : 0;
    for (int i = 1; i < d && R > 0; ++i) members = members * (R + i) / i;
    if (!dbl) return nv + members;
    return ((nv > 0 ? 1 : 0) + members) * (R > 2 ? 1 : covs);
}

template cudaError_t launch_lag<float>(int, int, int, const LagJob<float>&, cudaStream_t);
}  // namespace kdefft
