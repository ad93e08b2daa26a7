// Generated by `python -m paper_2407_13585_b200.instantiate workloads:segmented_products workloads:segmented_reversed workloads:segmented_weights`.
// Every cluster of every legal clustering of the programs named above, and every node alone.
#include "device/launch.cuh"

namespace acc {

constexpr CProgram make_segmented_products() {
  CProgram p{6, (1ull << 4) | (1ull << 5), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_F32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[3] = pnode(ACC_ZIPWITH, ACC_F32, 1, ACC_FN_MUL, 0, 2, 0, 1);  // w
  p.nodes[4] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_ADD, 0, 1, 3, 2);  // sums
  p.nodes[5] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_MAX, 0, 1, 3, 2);  // maxes
  return p;
}
inline constexpr CProgram k_segmented_products = make_segmented_products();
ACC_CLUSTER(k_segmented_products, 0x8, segmented_products__w)
ACC_CLUSTER(k_segmented_products, 0x10, segmented_products__sums)
ACC_CLUSTER(k_segmented_products, 0x20, segmented_products__maxes)
ACC_CLUSTER(k_segmented_products, 0x30, segmented_products__sums_maxes)
ACC_CLUSTER(k_segmented_products, 0x38, segmented_products__w_sums_maxes)
// not instantiated (outside the skeletons): w_sums, w_maxes

constexpr CProgram make_segmented_reversed() {
  CProgram p{5, (1ull << 3) | (1ull << 4), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_BACKPERMUTE, ACC_F32, 1, 0, ACC_IDX_REVERSE, 1, 0);  // r
  p.nodes[3] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_ADD, 0, 1, 2, 1);  // sums
  p.nodes[4] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_MIN, 0, 1, 2, 1);  // mins
  return p;
}
inline constexpr CProgram k_segmented_reversed = make_segmented_reversed();
ACC_CLUSTER(k_segmented_reversed, 0x4, segmented_reversed__r)
ACC_CLUSTER(k_segmented_reversed, 0x8, segmented_reversed__sums)
ACC_CLUSTER(k_segmented_reversed, 0x10, segmented_reversed__mins)
ACC_CLUSTER(k_segmented_reversed, 0x18, segmented_reversed__sums_mins)
ACC_CLUSTER(k_segmented_reversed, 0x1C, segmented_reversed__r_sums_mins)
// not instantiated (outside the skeletons): r_sums, r_mins

constexpr CProgram make_segmented_weights() {
  CProgram p{6, (1ull << 4) | (1ull << 5), {}};
  p.nodes[0] = pnode(ACC_INPUT, ACC_F32, 1, 0, 0, 0);
  p.nodes[1] = pnode(ACC_INPUT, ACC_I32, 1, 0, 0, 0);
  p.nodes[2] = pnode(ACC_GENERATE, ACC_F32, 1, ACC_FN_IMOD_TO_F32, 0, 0);  // g
  p.nodes[3] = pnode(ACC_ZIPWITH, ACC_F32, 1, ACC_FN_MUL, 0, 2, 0, 2);  // w
  p.nodes[4] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_ADD, 0, 1, 3, 1);  // sums
  p.nodes[5] = pnode(ACC_FOLDSEG, ACC_F32, 1, ACC_FN_MAX, 0, 1, 0, 1);  // maxes
  return p;
}
inline constexpr CProgram k_segmented_weights = make_segmented_weights();
ACC_CLUSTER(k_segmented_weights, 0x4, segmented_weights__g)
ACC_CLUSTER(k_segmented_weights, 0x8, segmented_weights__w)
ACC_CLUSTER(k_segmented_weights, 0x10, segmented_weights__sums)
ACC_CLUSTER(k_segmented_weights, 0x20, segmented_weights__maxes)
ACC_CLUSTER(k_segmented_weights, 0xC, segmented_weights__g_w)
ACC_CLUSTER(k_segmented_weights, 0x18, segmented_weights__w_sums)
ACC_CLUSTER(k_segmented_weights, 0x1C, segmented_weights__g_w_sums)
ACC_CLUSTER(k_segmented_weights, 0x38, segmented_weights__w_sums_maxes)
ACC_CLUSTER(k_segmented_weights, 0x3C, segmented_weights__g_w_sums_maxes)
// not instantiated (outside the skeletons): w_maxes, g_w_maxes

}  // namespace acc
