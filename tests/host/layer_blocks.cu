// Host check of how the CPML layer's launch splits into clusters, compiled
// from the library's own source: reads "nx ny nz npml" lines, prints "ok" or
// what is wrong.
#include <cstdio>
#include <map>
#include <tuple>
#include <vector>

#include "../../paper_2404_04441_gb300/csrc/cpml.cuh"

using namespace gbw;

struct Visit {
  int block, phase, axis;
};

static const char *check(int nx, int ny, int nz, int npml) {
  CpmlGeom g{};
  g.nx = nx;
  g.ny = ny;
  g.nz = nz;
  g.npml = npml;
  g.w = npml + 4;
  const int n[3] = {nx, ny, nz}, w = g.w;
  std::map<std::tuple<int, int, int, int>, int> lines;  // (axis, side, p, q) -> count
  std::vector<std::vector<Visit>> at((size_t)nx * ny * nz);
  const char *bad = nullptr;
  {
    const CpmlTiles t = cpml_tiles(nx, ny, nz, w, -1);
    for (int blk = 0; blk < t.start[7]; ++blk)
      for (int tid = 0; tid < kCpmlLines; ++tid) {
        int phase = 0;
        cpml_block(
            g, t, blk, tid,
            [&](int ax, int side, int p, int q) {
              const int np = ax == 0 ? ny : nx, nq = ax == 2 ? ny : nz;
              if (p < 0 || p >= np || q < 0 || q >= nq) {
                bad = "line outside the grid";
                return;
              }
              lines[{ax, side, p, q}]++;
              for (int j = 0; j < w; ++j) {
                const int i = side ? n[ax] - 1 - j : j;
                const int x = ax == 0 ? i : p, y = ax == 1 ? i : ax == 0 ? p : q,
                          z = ax == 2 ? i : q;
                at[((size_t)z * ny + y) * nx + x].push_back({blk, phase, ax});
              }
            },
            [&] { ++phase; });
      }
  }
  if (bad) return bad;
  size_t want = 0;
  for (int ax = 0; ax < 3; ++ax) want += 2 * (size_t)nx * ny * nz / n[ax];
  if (lines.size() != want) return "a line is missing";
  for (auto &l : lines)
    if (l.second != 1) return "a line is taken twice";
  // a point's terms come in axis order, all in one cluster, each after the
  // one before it by a barrier
  for (auto &v : at)
    for (size_t i = 0; i < v.size(); ++i)
      for (size_t j = 0; j < v.size(); ++j)
        if (v[i].axis < v[j].axis &&
            !(v[i].block == v[j].block && v[i].phase < v[j].phase))
          return "two axes meet without an order";
  return "ok";
}

int main() {
  int nx, ny, nz, npml;
  while (std::scanf("%d %d %d %d", &nx, &ny, &nz, &npml) == 4)
    std::printf("%s\n", check(nx, ny, nz, npml));
  return 0;
}
