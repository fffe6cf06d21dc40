// Column kernels of kernels_col.cuh in fp64.
#include "kernels_col.cuh"

namespace fftlb {

ColSet col_set_f64(int NY) {
    switch (NY) {
        case 4: return ck::col_set<double, 4>();
        case 6: return ck::col_set<double, 6>();
        case 8: return ck::col_set<double, 8>();
        case 12: return ck::col_set<double, 12>();
        case 16: return ck::col_set<double, 16>();
        case 24: return ck::col_set<double, 24>();
        case 32: return ck::col_set<double, 32>();
        case 48: return ck::col_set<double, 48>();
        case 64: return ck::col_set<double, 64>();
        case 96: return ck::col_set<double, 96>();
        case 128: return ck::col_set<double, 128>();
        case 192: return ck::col_set<double, 192>();
        case 256: return ck::col_set<double, 256>();
        case 384: return ck::col_set<double, 384>();
        case 512: return ck::col_set<double, 512>();
        case 768: return ck::col_set<double, 768>();
        case 1024: return ck::col_set<double, 1024>();
        default: return ColSet();
    }
}

}  // namespace fftlb
