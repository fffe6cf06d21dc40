// The complex type of each precision.
#pragma once

#include <vector_types.h>

namespace fftlb {

template <typename real> struct cplx_of;
template <> struct cplx_of<double> { using type = double2; };
template <> struct cplx_of<float> { using type = float2; };

}  // namespace fftlb
