// Checks of short strips (csrc/strips.cuh, two and four rows): on the GPU as strips_check.cu does for
// longer ones, on small and ragged levels; on the host that the rule for the rows never makes more
// blocks than the mesh has 32 x 8 tiles, the room of the partial sums.  Prints "ok".
#define main strips_check_main
#include "strips_check.cu"
#undef main

static bool room() {
  for (int n = 4; n <= 400; n += 2)
    for (int m = 4; m <= 400; m += 2)
      for (int cols : {1, 2, 3, 10, 40, 96, 2560}) {
        const int rows = strip_rows(n, m, cols);
        const long tiles = (long)((n + 31) / 32) * ((m + 7) / 8);
        if (rows < 2 || strip_blocks<30>(n, m, rows) > tiles || strip_blocks<31>(n, m, rows) > tiles) {
          std::printf("%d x %d, %d columns: %d rows, more blocks than tiles\n", n, m, cols, rows);
          return false;
        }
      }
  return true;
}

int main() {
  bool ok = room();
  const int sizes[][2] = {{4, 4}, {8, 6}, {30, 10}, {32, 14}, {62, 18}, {96, 34}};
  for (auto& s : sizes)
    for (int rows : {2, 4})
      for (bool smooth : {false, true}) ok = run(s[0], s[1], rows, smooth) && ok;
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
