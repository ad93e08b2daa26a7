// Clusters of workloads:sum_of_two_gathers and workloads:scan_of_reversed, as `python -m paper_2407_13585_b200.instantiate` prints
// them, of each program only the one of all its nodes (its nodes alone are among those of csrc/programs).
#include "device/launch.cuh"

namespace acc {

constexpr CProgram make_sum_of_two_gathers() {
  CProgram p{7, (1ull << 6), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[3] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 1, 0);  // g
  p.nodes[4] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 2, 0);  // h
  p.nodes[5] = pnode(ACC_ZIPWITH, ACC_I32, 1, ACC_FN_ADD, 0, 2, 3, 4);  // u
  p.nodes[6] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 5);  // s
  return p;
}
inline constexpr CProgram k_sum_of_two_gathers = make_sum_of_two_gathers();
ACC_CLUSTER(k_sum_of_two_gathers, 0x78, sum_of_two_gathers__g_h_u_s)

constexpr CProgram make_scan_of_reversed() {
  CProgram p{3, (1ull << 2), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_BACKPERMUTE, ACC_F32, 1, 0, ACC_IDX_REVERSE, 1, 0);  // y
  p.nodes[2] = pnode(ACC_SCANL, ACC_F32, 1, ACC_FN_ADD, 0, 1, 1);  // s
  return p;
}
inline constexpr CProgram k_scan_of_reversed = make_scan_of_reversed();
ACC_CLUSTER(k_scan_of_reversed, 0x6, scan_of_reversed__y_s)

}  // namespace acc
