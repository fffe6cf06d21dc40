// Row kernels of kernels_row.cuh: half rows of 3 2^p values, fp64.
#include "kernels_row.cuh"

namespace fftlb {

RowSet row_set_f64_r3(int H) {
    switch (H) {
        case 24: return rk::row_set<double, 24>();
        case 48: return rk::row_set<double, 48>();
        case 96: return rk::row_set<double, 96>();
        case 192: return rk::row_set<double, 192>();
        case 384: return rk::row_set<double, 384>();
        default: return RowSet();
    }
}

}  // namespace fftlb
