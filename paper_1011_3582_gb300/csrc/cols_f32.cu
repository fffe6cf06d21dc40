// Column kernels of kernels_col.cuh in fp32.
#include "kernels_col.cuh"

namespace fftlb {

ColSet col_set_f32(int NY) {
    switch (NY) {
        case 4: return ck::col_set<float, 4>();
        case 6: return ck::col_set<float, 6>();
        case 8: return ck::col_set<float, 8>();
        case 12: return ck::col_set<float, 12>();
        case 16: return ck::col_set<float, 16>();
        case 24: return ck::col_set<float, 24>();
        case 32: return ck::col_set<float, 32>();
        case 48: return ck::col_set<float, 48>();
        case 64: return ck::col_set<float, 64>();
        case 96: return ck::col_set<float, 96>();
        case 128: return ck::col_set<float, 128>();
        case 192: return ck::col_set<float, 192>();
        case 256: return ck::col_set<float, 256>();
        case 384: return ck::col_set<float, 384>();
        case 512: return ck::col_set<float, 512>();
        case 768: return ck::col_set<float, 768>();
        case 1024: return ck::col_set<float, 1024>();
        case 1536: return ck::col_set<float, 1536>();
        case 2048: return ck::col_set<float, 2048>();
        default: return ColSet();
    }
}

}  // namespace fftlb
