// Clusters of workloads:gathered_scans for the roots that the tests ask for, as `python -m paper_2407_13585_b200.instantiate`
// prints them, of each program only the one of all its nodes (its nodes alone are among those of csrc/programs).
#include "device/launch.cuh"

namespace acc {

constexpr CProgram make_gathered_scans_3() {
  CProgram p{6, (1ull << 4) | (1ull << 5), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_MAP, ACC_I32, 1, ACC_FN_AND_MASK, 0, 1, 1);  // k
  p.nodes[3] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 2, 0);  // h
  p.nodes[4] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 3);  // s
  p.nodes[5] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_MAX, 0, 1, 3);  // m
  return p;
}
inline constexpr CProgram k_gathered_scans_3 = make_gathered_scans_3();
ACC_CLUSTER(k_gathered_scans_3, 0x3C, gathered_scans_3__k_h_s_m)

constexpr CProgram make_gathered_scans_5() {
  CProgram p{6, (1ull << 4) | (1ull << 5), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_MAP, ACC_I32, 1, ACC_FN_AND_MASK, 0, 1, 1);  // k
  p.nodes[3] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 2, 0);  // h
  p.nodes[4] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 3);  // s
  p.nodes[5] = fixed(pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 3), 1, kRunTime);  // e
  return p;
}
inline constexpr CProgram k_gathered_scans_5 = make_gathered_scans_5();
ACC_CLUSTER(k_gathered_scans_5, 0x3C, gathered_scans_5__k_h_s_e)

constexpr CProgram make_gathered_scans_9() {
  CProgram p{6, (1ull << 4) | (1ull << 5), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_MAP, ACC_I32, 1, ACC_FN_AND_MASK, 0, 1, 1);  // k
  p.nodes[3] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 2, 0);  // h
  p.nodes[4] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 3);  // s
  p.nodes[5] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 2);  // t
  return p;
}
inline constexpr CProgram k_gathered_scans_9 = make_gathered_scans_9();
ACC_CLUSTER(k_gathered_scans_9, 0x3C, gathered_scans_9__k_h_s_t)

constexpr CProgram make_gathered_scans_27() {
  CProgram p{8, (1ull << 4) | (1ull << 5) | (1ull << 6) | (1ull << 7), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_MAP, ACC_I32, 1, ACC_FN_AND_MASK, 0, 1, 1);  // k
  p.nodes[3] = pnode(ACC_GATHER, ACC_I32, 1, 0, 0, 2, 2, 0);  // h
  p.nodes[4] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 3);  // s
  p.nodes[5] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_MAX, 0, 1, 3);  // m
  p.nodes[6] = pnode(ACC_SCANL, ACC_I32, 1, ACC_FN_ADD, 0, 1, 2);  // t
  p.nodes[7] = pnode(ACC_FOLD, ACC_I32, 0, ACC_FN_ADD, 0, 1, 2);  // total
  return p;
}
inline constexpr CProgram k_gathered_scans_27 = make_gathered_scans_27();
ACC_CLUSTER(k_gathered_scans_27, 0xFC, gathered_scans_27__k_h_s_m_t_total)

}  // namespace acc
