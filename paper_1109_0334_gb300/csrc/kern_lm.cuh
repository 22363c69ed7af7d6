// kern_lm.cuh -- the direction count of the sensitivity kernels (kern_lm.cu,
// kern_lm_lanes.cu).
#pragma once
#include <type_traits>

#include "afm_tangent.cuh"

namespace afm {

// f(directions, coefficient directions?): the law's coefficients where the
// free parameters are at least as many, else the parameters (2, or 3 of the
// Kelvin-Voigt law's four coefficients).
template <int FORCE, typename F>
cudaError_t sens_dirs(int D, F&& f) {
    constexpr int NC = aff::CoefDirs<FORCE>::n;
    if (D >= NC) return f(std::integral_constant<int, NC>{}, std::true_type{});
    if constexpr (NC == 4)
        if (D == 3) return f(std::integral_constant<int, 3>{}, std::false_type{});
    return f(std::integral_constant<int, 2>{}, std::false_type{});
}

}  // namespace afm
