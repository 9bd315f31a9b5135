// Prints, per slot of launch_pass (-1: none), whether its pass counts as one
// that runs beside another.
#include <cstdio>

#include "api_internal.h"

int main() {
  for (int slot = -1; slot < rf::kPassSlots; ++slot) std::printf("%d %d\n", slot, rf::slot_beside(slot) ? 1 : 0);
  return 0;
}
