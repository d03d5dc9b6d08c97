// Host check (no GPU): the marching kernels' plans use the chip on tall lattices
// of few tiles.  A pass over such a lattice takes as long as its thickest slab,
// so a plan with fewer blocks than half the multiprocessors must consist of the
// thinnest slabs there are (two planes).  Prints the plans that do not.
#include <cstdio>
#include <vector>

#include "march.cuh"

namespace hca {
void march_tile(MGLevel& L, int halo_rows);
void march_blocks(std::vector<MGLevel*>& lv, const std::vector<int>& reps, int sm_count, int extra, std::vector<int4>& out);
}  // namespace hca

int main() {
  const int sms = 152;
  int bad = 0;
  for (int nx : {8, 16, 25, 40, 43, 64, 100})
    for (int ny : {8, 16, 27, 41, 64})
      for (int nz = 1; nz <= 2000; nz = nz < 400 ? nz + 1 : nz + 37)
        for (int halo : {1, 2}) {
          hca::MGLevel L{};
          L.nx = nx;
          L.ny = ny;
          L.nz = nz;
          L.pitch = (nx + 3) / 4 * 4;
          hca::march_tile(L, halo);
          std::vector<hca::MGLevel*> set{&L};
          std::vector<int4> blocks;
          hca::march_blocks(set, {0}, sms, halo == 1 ? 4 : 6, blocks);
          int thickest = 0;
          for (const int4& b : blocks) thickest = thickest > b.w - b.z ? thickest : b.w - b.z;
          if ((int)blocks.size() < sms / 2 && thickest > 2 && ++bad <= 20)
            std::printf("%d x %d x %d, halo %d: %d blocks, slabs of %d planes\n", nx, ny, nz, halo, (int)blocks.size(),
                        thickest);
        }
  return bad != 0;
}
