// pa_real_table_plain.cu -- threshold-table sweeps of real couplings without a
// field (the two translation units compile in parallel).
#include "pa_real_table.cuh"

namespace pa {

cudaError_t launch_sweep_real_table_plain(int D, int L, const RealSweepArgs& a, cudaStream_t st, bool* handled)
{
    *handled = true;
#define X(d, l)                                                                                  \
    if constexpr (TabShape<d, l, false>::FITS)                                                   \
        if (D == d && L == l) return launch_real_table<d, l, false>(a, st);
    X(3, 2) X(3, 4) X(3, 6) X(3, 8) X(3, 10) X(3, 12)
    X(2, 2) X(2, 4) X(2, 6) X(2, 8) X(2, 10) X(2, 12) X(2, 16) X(2, 32)
#undef X
    *handled = false;
    return cudaSuccess;
}

}  // namespace pa
