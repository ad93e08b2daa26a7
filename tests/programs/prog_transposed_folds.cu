// Generated by `python -m paper_2407_13585_b200.instantiate workloads:transposed_folds:0 workloads:transposed_folds:1 workloads:transposed_folds:2 workloads:transposed_folds:3`.
// Every cluster of every legal clustering of the programs named above, and every node alone.
#include "device/launch.cuh"

namespace acc {

constexpr CProgram make_transposed_folds_0() {
  CProgram p{5, (1ull << 3) | (1ull << 4), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 2, 0, 0, 0);
  p.nodes[1] = pnode(ACC_BACKPERMUTE, ACC_I32, 2, 0, ACC_IDX_TRANSPOSE, 1, 0);  // B
  p.nodes[2] = pnode(ACC_ZIPWITH, ACC_I32, 2, ACC_FN_ADD, 0, 2, 0, 1);  // C
  p.nodes[3] = pnode(ACC_FOLD, ACC_I32, 1, ACC_FN_ADD, 0, 1, 2);  // row_add
  p.nodes[4] = pnode(ACC_FOLD, ACC_I32, 1, ACC_FN_MAX, 0, 1, 2);  // row_max
  return p;
}
inline constexpr CProgram k_transposed_folds_0 = make_transposed_folds_0();
ACC_CLUSTER(k_transposed_folds_0, 0x2, transposed_folds_0__B)
ACC_CLUSTER(k_transposed_folds_0, 0x4, transposed_folds_0__C)
ACC_CLUSTER(k_transposed_folds_0, 0x8, transposed_folds_0__row_add)
ACC_CLUSTER(k_transposed_folds_0, 0x10, transposed_folds_0__row_max)
ACC_CLUSTER(k_transposed_folds_0, 0x6, transposed_folds_0__B_C)
ACC_CLUSTER(k_transposed_folds_0, 0xC, transposed_folds_0__C_row_add)
ACC_CLUSTER(k_transposed_folds_0, 0x14, transposed_folds_0__C_row_max)
ACC_CLUSTER(k_transposed_folds_0, 0x18, transposed_folds_0__row_add_row_max)
ACC_CLUSTER(k_transposed_folds_0, 0xE, transposed_folds_0__B_C_row_add)
ACC_CLUSTER(k_transposed_folds_0, 0x16, transposed_folds_0__B_C_row_max)
ACC_CLUSTER(k_transposed_folds_0, 0x1C, transposed_folds_0__C_row_add_row_max)
ACC_CLUSTER(k_transposed_folds_0, 0x1E, transposed_folds_0__B_C_row_add_row_max)

constexpr CProgram make_transposed_folds_1() {
  CProgram p{5, (1ull << 3) | (1ull << 4), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 2, 0, 0, 0);
  p.nodes[1] = pnode(ACC_BACKPERMUTE, ACC_F32, 2, 0, ACC_IDX_TRANSPOSE, 1, 0);  // B
  p.nodes[2] = pnode(ACC_ZIPWITH, ACC_F32, 2, ACC_FN_ADD, 0, 2, 0, 1);  // C
  p.nodes[3] = pnode(ACC_FOLD, ACC_F32, 1, ACC_FN_MAX, 0, 1, 2);  // row_max
  p.nodes[4] = pnode(ACC_FOLD, ACC_F32, 1, ACC_FN_MIN, 0, 1, 2);  // row_min
  return p;
}
inline constexpr CProgram k_transposed_folds_1 = make_transposed_folds_1();
ACC_CLUSTER(k_transposed_folds_1, 0x2, transposed_folds_1__B)
ACC_CLUSTER(k_transposed_folds_1, 0x4, transposed_folds_1__C)
ACC_CLUSTER(k_transposed_folds_1, 0x8, transposed_folds_1__row_max)
ACC_CLUSTER(k_transposed_folds_1, 0x10, transposed_folds_1__row_min)
ACC_CLUSTER(k_transposed_folds_1, 0x6, transposed_folds_1__B_C)
ACC_CLUSTER(k_transposed_folds_1, 0xC, transposed_folds_1__C_row_max)
ACC_CLUSTER(k_transposed_folds_1, 0x14, transposed_folds_1__C_row_min)
ACC_CLUSTER(k_transposed_folds_1, 0x18, transposed_folds_1__row_max_row_min)
ACC_CLUSTER(k_transposed_folds_1, 0xE, transposed_folds_1__B_C_row_max)
ACC_CLUSTER(k_transposed_folds_1, 0x16, transposed_folds_1__B_C_row_min)
ACC_CLUSTER(k_transposed_folds_1, 0x1C, transposed_folds_1__C_row_max_row_min)
ACC_CLUSTER(k_transposed_folds_1, 0x1E, transposed_folds_1__B_C_row_max_row_min)

constexpr CProgram make_transposed_folds_2() {
  CProgram p{4, (1ull << 3), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_U32, 2, 0, 0, 0);
  p.nodes[1] = pnode(ACC_BACKPERMUTE, ACC_U32, 2, 0, ACC_IDX_TRANSPOSE, 1, 0);  // B
  p.nodes[2] = pnode(ACC_ZIPWITH, ACC_U32, 2, ACC_FN_ADD, 0, 2, 0, 1);  // C
  p.nodes[3] = pnode(ACC_FOLD, ACC_U32, 1, ACC_FN_MIN, 0, 1, 2);  // row_min
  return p;
}
inline constexpr CProgram k_transposed_folds_2 = make_transposed_folds_2();
ACC_CLUSTER(k_transposed_folds_2, 0x2, transposed_folds_2__B)
ACC_CLUSTER(k_transposed_folds_2, 0x4, transposed_folds_2__C)
ACC_CLUSTER(k_transposed_folds_2, 0x8, transposed_folds_2__row_min)
ACC_CLUSTER(k_transposed_folds_2, 0x6, transposed_folds_2__B_C)
ACC_CLUSTER(k_transposed_folds_2, 0xC, transposed_folds_2__C_row_min)
ACC_CLUSTER(k_transposed_folds_2, 0xE, transposed_folds_2__B_C_row_min)

constexpr CProgram make_transposed_folds_3() {
  CProgram p{4, (1ull << 3), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 2, 0, 0, 0);
  p.nodes[1] = pnode(ACC_BACKPERMUTE, ACC_F32, 2, 0, ACC_IDX_TRANSPOSE, 1, 0);  // B
  p.nodes[2] = pnode(ACC_ZIPWITH, ACC_F32, 2, ACC_FN_ADD, 0, 2, 0, 1);  // C
  p.nodes[3] = pnode(ACC_FOLD, ACC_F32, 1, ACC_FN_ADD, 0, 1, 2);  // row_add
  return p;
}
inline constexpr CProgram k_transposed_folds_3 = make_transposed_folds_3();
ACC_CLUSTER(k_transposed_folds_3, 0x2, transposed_folds_3__B)
ACC_CLUSTER(k_transposed_folds_3, 0x4, transposed_folds_3__C)
ACC_CLUSTER(k_transposed_folds_3, 0x8, transposed_folds_3__row_add)
ACC_CLUSTER(k_transposed_folds_3, 0x6, transposed_folds_3__B_C)
ACC_CLUSTER(k_transposed_folds_3, 0xC, transposed_folds_3__C_row_add)
ACC_CLUSTER(k_transposed_folds_3, 0xE, transposed_folds_3__B_C_row_add)

}  // namespace acc
