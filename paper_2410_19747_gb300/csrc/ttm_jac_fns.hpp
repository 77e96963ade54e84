// ttm_jac_fns.hpp -- host functions of the Jacobi kernels by rows per lane (ttm_jac.cu).
#pragma once

namespace ttm {

// 1, 2, 4, 8, 12, 16, 24 or 32 rows per lane
void* jacobi_pre_fn(int R);
inline int jacobi_pre_rows(int rows) {
  return rows <= 2 ? rows : rows <= 16 ? (rows + 3) / 4 * 4 : (rows + 7) / 8 * 8;
}
// 1, 2, 4, 8, 16 or 32
void* jacobi_res_fn(bool f64, int R);
void* jacobi4_fn(int R);

}  // namespace ttm
