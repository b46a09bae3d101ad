// Prints "thread slot row col source" for every slot of the capacitance
// kernel's solving block (host side of csrc/emu_capslots.h).
#include <cstdio>

#include "emu_capslots.h"

int main() {
  for (int s = 0; s < emu::kCapOwn; ++s)
    for (int t = 0; t < emu::kCapThreads; ++t) {
      int row, col;
      emu::cap_slot(t, s, &row, &col);
      printf("%d %d %d %d %d\n", t, s, row, col, emu::cap_source(row, col));
    }
  return 0;
}
