// The evaluation buffers' sizes (workspace.h) against what the event kernels
// index, for models of different sizes taken in turn on one dataset: a buffer
// holds the largest size asked for so far (DevBuf::ensure).  Prints, per
// dataset, the number of part records or tree rows that would not fit.
#include <cstdio>

#include "workspace.h"

using namespace rf;

struct Step { int shape, n_slots, n_const, n_free; };
// exponential on the interpreter; decay float-float, interpreter; Gauss + line
// float-float; product model float-float and interpreter; the largest model
static const Step kSteps[] = {{SHAPE_GENERIC, 1, 4, 1},  {SHAPE_SUM_GAUSSEXP_CHEB2, 6, 17, 6},
                              {SHAPE_GENERIC, 6, 17, 6}, {SHAPE_SUM_GAUSS_POLY1, 4, 10, 4},
                              {SHAPE_SUM_GAUSSEXP_CHEB2, 6, 17, 6}, {SHAPE_GENERIC, 4, 10, 4},
                              {SHAPE_PROD3, 12, 40, 12}, {SHAPE_GENERIC, 12, 40, 12},
                              {SHAPE_GENERIC, kMaxSlots, kMaxConst, kMaxFree}, {SHAPE_PROD3, 12, 40, 12}};

int main() {
  const long long chunk_counts[] = {0, 1, 3, 33, 34, 66, 133, 245, 266, 531, 532, 760, 1063, 1064, 5000};
  for (long long chunks : chunk_counts) {
    const size_t nodes = chunks ? (size_t)chunks + (size_t)(chunks + 31) / 32 + 2 : 0, sets = 3;
    int lost = 0;
    for (int first = 0; first < 10; ++first) {  // every order of a rotation
      WorkspaceBytes have{};
      for (int i = 0; i < 10; ++i) {
        const Step& t = kSteps[(first + i) % 10];
        Program P{};
        P.n_slots = t.n_slots;
        P.n_const = t.n_const;
        P.n_free = t.n_free;
        const WorkspaceBytes b = workspace_bytes(P, t.shape, sets, (int64_t)nodes, chunks, 512);
        have.tree = std::max(have.tree, b.tree);
        have.ffc = std::max(have.ffc, b.ffc);
        have.part_m = std::max(have.part_m, b.part_m);
        have.part_fb = std::max(have.part_fb, b.part_fb);
        have.part_info = std::max(have.part_info, b.part_info);
        // one past the last double or word that a unit of the last node writes
        const size_t Q = 1 + (size_t)t.n_slots, parts = (size_t)parts_for(chunks, t.shape), recs = nodes * parts;
        lost += nodes * 2 * Q * sizeof(double) > have.tree;
        if (t.shape == SHAPE_GENERIC) {
          if (parts == 1) continue;
          lost += recs * 2 * Q * sizeof(double) > have.part_fb;
        } else {
          lost += recs * Q * sizeof(double) > have.part_fb;
          lost += recs * kPartFloats * sizeof(float) > have.part_m;
          lost += sets * 512 * sizeof(float) > have.ffc;
        }
        lost += recs * sizeof(int32_t) > have.part_info;
      }
    }
    std::printf("%lld %d\n", chunks, lost);
  }
  return 0;
}
