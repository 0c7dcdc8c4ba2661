// The instantiated shapes of the sweep kernels: lanes (logical lanes per body, which fix the
// summation order and so the result), threads per body (as many, or half; either gives the same
// result, see sys_sum_lanes) and the extended type of ill-conditioned bodies (FP64 under policy
// 2, with one thread per lane; the compensated single-precision sums otherwise).
#pragma once
#include <type_traits>

#include "sweep_math.cuh"

namespace pabd {

template <class T>
struct TypeOf {
    using type = T;
};

// calls f(lanes, type) with both as compile-time constants
template <class F>
void with_lanes(int lanes, bool f64, F&& f) {
    auto go = [&](auto l) {
        if (f64) f(l, TypeOf<double>{});
        else f(l, TypeOf<ca>{});
    };
    switch (lanes) {
        case 1: go(std::integral_constant<int, 1>{}); break;
        case 2: go(std::integral_constant<int, 2>{}); break;
        case 4: go(std::integral_constant<int, 4>{}); break;
        case 8: go(std::integral_constant<int, 8>{}); break;
        default: go(std::integral_constant<int, 16>{}); break;
    }
}

// calls f(lanes, threads, type); threads is lanes, or half of it
template <class F>
void with_sweep_shape(int lanes, int threads, bool f64, F&& f) {
    with_lanes(lanes, f64, [&](auto l, auto x) {
        constexpr int L = decltype(l)::value;
        if constexpr (L > 1 && !std::is_same<typename decltype(x)::type, double>::value) {
            if (threads < L) return f(l, std::integral_constant<int, L / 2>{}, x);
        }
        f(l, l, x);
    });
}

}  // namespace pabd
