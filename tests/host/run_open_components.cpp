// Test infrastructure: the components next to the middle row that the host
// counts once per triangulation (open_components) are as many under every sign
// vector.  Usage: run_open_components <d> <edges file> <sign vectors>; prints
// their number and what the block sweep's middle phase holds; exit 0 when all
// agree.
#define main run_table_sweep_main
#include "run_table_sweep.cpp"
#undef main

int main(int argc, char **argv) {
  const int d = atoi(argv[1]);
  std::vector<int32_t> e;
  std::ifstream f(argv[2]);
  for (int a; f >> a;) e.push_back(a);
  std::vector<std::array<Pt, 3>> tris;
  ts_tri t;
  if (argc < 4 || !triangles_of(d, e.data(), (int)e.size() / 4, tris) || !build_diamond(d, tris, t.dia) ||
      !pack_tables(t.dia, &t))
    return 2;
  for (int i = 0; i < atoi(argv[3]); ++i)
    if (open_components(t.dia, mix64(i) >> (64 - (d + 1) * (d + 2) / 2)) != t.open) return 1;
  printf("%d %d\n", t.open, tc_block_nodes(d));
  return 0;
}
