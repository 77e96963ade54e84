// ttm_jac.cu -- the Jacobi kernels, instantiated for the rows per lane they are launched with.
//
// A translation unit of its own, so that it compiles beside the rest: the launch code asks for a
// kernel's host function.
#include <cuda_runtime.h>

#include "ttm_jac4.cuh"
#include "ttm_jac_fns.hpp"
#include "ttm_jres.cuh"
#include "ttm_pjac.cuh"

namespace ttm {

void* jacobi_pre_fn(int R) {
  switch (R) {
    case 1: return (void*)jacobi_pre_kernel<1>;
    case 2: return (void*)jacobi_pre_kernel<2>;
    case 4: return (void*)jacobi_pre_kernel<4>;
    case 8: return (void*)jacobi_pre_kernel<8>;
    case 12: return (void*)jacobi_pre_kernel<12>;
    case 16: return (void*)jacobi_pre_kernel<16>;
    case 24: return (void*)jacobi_pre_kernel<24>;
    default: return (void*)jacobi_pre_kernel<32>;
  }
}

template <typename T>
static void* res_fn(int R) {
  switch (R) {
    case 1: return (void*)jacobi_res_kernel<T, kJrB, 1>;
    case 2: return (void*)jacobi_res_kernel<T, kJrB, 2>;
    case 4: return (void*)jacobi_res_kernel<T, kJrB, 4>;
    case 8: return (void*)jacobi_res_kernel<T, kJrB, 8>;
    case 16: return (void*)jacobi_res_kernel<T, kJrB, 16>;
    default: return (void*)jacobi_res_kernel<T, kJrB, 32>;
  }
}
void* jacobi_res_fn(bool f64, int R) { return f64 ? res_fn<double>(R) : res_fn<float>(R); }

void* jacobi4_fn(int R) {
  switch (R) {
    case 1: return (void*)jacobi4_kernel<1>;
    case 2: return (void*)jacobi4_kernel<2>;
    case 4: return (void*)jacobi4_kernel<4>;
    case 8: return (void*)jacobi4_kernel<8>;
    case 16: return (void*)jacobi4_kernel<16>;
    default: return (void*)jacobi4_kernel<32>;
  }
}

}  // namespace ttm
