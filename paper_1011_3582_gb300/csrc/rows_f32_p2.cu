// Row kernels of kernels_row.cuh: half rows of 2^p values, fp32.
#include "kernels_row.cuh"

namespace fftlb {

RowSet row_set_f32_p2(int H) {
    switch (H) {
        case 16: return rk::row_set<float, 16>();
        case 32: return rk::row_set<float, 32>();
        case 64: return rk::row_set<float, 64>();
        case 128: return rk::row_set<float, 128>();
        case 256: return rk::row_set<float, 256>();
        case 512: return rk::row_set<float, 512>();
        case 1024: return rk::row_set<float, 1024>();
        default: return RowSet();
    }
}

}  // namespace fftlb
