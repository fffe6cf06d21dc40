// Row kernels of kernels_row.cuh: half rows of 3 2^p values, fp32.
#include "kernels_row.cuh"

namespace fftlb {

RowSet row_set_f32_r3(int H) {
    switch (H) {
        case 24: return rk::row_set<float, 24>();
        case 48: return rk::row_set<float, 48>();
        case 96: return rk::row_set<float, 96>();
        case 192: return rk::row_set<float, 192>();
        case 384: return rk::row_set<float, 384>();
        case 768: return rk::row_set<float, 768>();
        default: return RowSet();
    }
}

}  // namespace fftlb
