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

template cudaError_t launch_lag<float>(int, int, int, const LagJob<float>&, cudaStream_t);
}  // namespace kdefft
