// The tile shape that a plan takes for each requested one: rows cols threads form on stdin; prints the
// status, the shape and whether the library plans the tiles.
#include "../paper_1810_09784_gb300/csrc/gfh_host.cpp"

#include <cstdio>

int main() {
  gfh_tile_config c;
  while (std::scanf("%d %d %d %d", &c.rows, &c.cols, &c.threads, &c.form) == 4) {
    gfh_tile_config t{};
    const int rc = tile_config(&c, &t);
    std::printf("%d %d %d %d %d %d\n", rc, t.rows, t.cols, t.threads, t.form, (int)same_shape(t, kDefaultShape));
  }
  return 0;
}
