// A loop whose index is a compile-time constant.
#pragma once
#include <type_traits>
#include <utility>

namespace wvl {

// compile-time loop: f(integral_constant<int, 0>) ... f(integral_constant<int, N - 1>),
// so tap indices are constants by construction (no run-time index or test)
template <typename F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

}  // namespace wvl
