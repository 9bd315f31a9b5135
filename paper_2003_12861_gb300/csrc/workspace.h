// Sizes of a dataset's evaluation buffers.  A dataset keeps one set of them
// for every model that is evaluated on it, in any order, so each call asks
// for what its own model's kernels index.
#pragma once

#include <algorithm>
#include <cstddef>

#include "nll_kernels.cuh"

namespace rf {

struct WorkspaceBytes {
  size_t consts, theta, out, flags, tree, node_words;  // node_words: tree_bad and tickets, each
  size_t ffc, part_m, part_fb, part_info;              // of the model's kernel, 0 = not used
};

// n_nodes, n_chunks: tree nodes and chunks of all sets together; ff_floats: a
// set's float-float constants (kFFConst).
inline WorkspaceBytes workspace_bytes(const Program& P, int shape, size_t n_sets, int64_t n_nodes, int64_t n_chunks,
                                      size_t ff_floats) {
  const size_t nodes = (size_t)std::max<int64_t>(1, n_nodes), Q = 1 + (size_t)P.n_slots;
  WorkspaceBytes b{};
  b.consts = sizeof(double) * n_sets * (size_t)std::max(1, P.n_const);
  b.theta = sizeof(double) * n_sets * (size_t)std::max(1, P.n_free);
  b.out = sizeof(double) * n_sets * (size_t)(1 + P.n_free);
  b.flags = sizeof(int32_t) * n_sets;
  b.tree = sizeof(double) * nodes * 2 * Q;
  b.node_words = sizeof(int32_t) * nodes;
  const size_t parts = (size_t)parts_for(n_chunks, shape);
  if (shape != SHAPE_GENERIC) {
    b.ffc = sizeof(float) * n_sets * ff_floats;
    b.part_m = sizeof(float) * nodes * parts * kPartFloats;
    b.part_fb = sizeof(double) * nodes * parts * Q;
    b.part_info = sizeof(int32_t) * nodes * parts;
  } else if (parts > 1) {  // (sum, compensation) per quantity
    b.part_fb = sizeof(double) * nodes * parts * 2 * Q;
    b.part_info = sizeof(int32_t) * nodes * parts;
  }
  return b;
}

}  // namespace rf
