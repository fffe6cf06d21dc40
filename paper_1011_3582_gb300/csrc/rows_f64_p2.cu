// Row kernels of kernels_row.cuh: half rows of 2^p values, fp64.
#include "kernels_row.cuh"

namespace fftlb {

RowSet row_set_f64_p2(int H) {
    switch (H) {
        case 16: return rk::row_set<double, 16>();
        case 32: return rk::row_set<double, 32>();
        case 64: return rk::row_set<double, 64>();
        case 128: return rk::row_set<double, 128>();
        case 256: return rk::row_set<double, 256>();
        case 512: return rk::row_set<double, 512>();
        default: return RowSet();
    }
}

}  // namespace fftlb
