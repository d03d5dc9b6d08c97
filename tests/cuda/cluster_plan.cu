// Host check (no GPU): the coarse levels of every FP32 hierarchy find a cluster
// that holds them, however long the lattice.  Prints the lattices that do not.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "hca_internal.cuh"

namespace hca {
int cluster_plan(const MGLevel* lv, int nl, int from, int cs, long long smem, MGCluster* R);
}

int main() {
  const long long M = 1000000;
  std::vector<std::vector<long long>> dims = {
      {600, 1, 1},       {16, 16, 16},     {512, 512, 512},  {1600, 1100, 1200}, {46000, 46000, 1}, {1, 46000, 46000},
      {20000 * 100, 1, 1}, {1, 20 * M, 1}, {1, 1, 20 * M},   {1, 1, 160 * M},    {1, 700 * M, 1},   {2, 2, 120 * M},
      {700 * M, 1, 1},   {2147483647, 1, 1}, {3, 3, 80 * M}, {5, 1, 400 * M},    {65536, 3, 4000},  {7, 9000, 9000}};
  int bad = 0;
  for (auto& d : dims) {
    long long nx = d[0], ny = d[1], nz = d[2], n = nx * ny * nz;
    std::vector<hca::MGLevel> lv(hca::MG_MAXLEV);
    int nl = 1;
    while (n > hca::MG_MIN_SITES && std::max(nx, std::max(ny, nz)) > 1 && nl < hca::MG_MAXLEV) {
      nx = (nx + 1) / 2;
      ny = (ny + 1) / 2;
      nz = (nz + 1) / 2;
      n = nx * ny * nz;
      hca::MGLevel& L = lv[nl++];
      L = hca::MGLevel{};
      L.nx = (int)nx;
      L.ny = (int)ny;
      L.nz = (int)nz;
      L.pitch = (int)((nx + 3) / 4 * 4);
      L.n = n;
    }
    for (int cs = 1; cs <= 16; cs *= 2) {
      int from = 1;
      while (from < nl - 1 && lv[from].n > hca::kClusterSites * cs) ++from;
      hca::MGCluster R;
      const int lc = hca::cluster_plan(lv.data(), nl, from, cs, hca::kClusterSmem, &R);
      if (lc < 1 || lc >= nl || R.smem > hca::kClusterSmem || lv[nl - 1].n > hca::MG_MIN_SITES) {
        ++bad;
        std::printf("%lld x %lld x %lld, %d blocks: first level %d of %d, coarsest level %lld sites\n", d[0], d[1], d[2], cs,
                    lc, nl, lv[nl - 1].n);
      }
    }
  }
  return bad != 0;
}
