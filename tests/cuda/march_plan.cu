// Host check of the plane-marching kernels' plans (no GPU): every block's
// segment sums fit the slots its shared memory has for them, and the blocks of
// a replicate cover its planes once.  Prints one line per plan that does not.
#include <cstdio>
#include <vector>

#include "march.cuh"

namespace hca {
void march_tile(MGLevel& L, int halo_rows);
void march_blocks(std::vector<MGLevel*>& lv, const std::vector<int>& reps, int sm_count, int extra, std::vector<int4>& out);
}  // namespace hca

int main() {
  // (nx, ny, replicates): one tile to thousands, rows and columns of them
  const int shapes[][3] = {{16, 16, 1},  {100, 100, 1}, {100, 100, 32}, {300, 200, 1},  {496, 496, 1},   {640, 512, 1},
                           {592, 592, 1}, {640, 640, 1}, {1000, 1000, 1}, {4000, 20, 1}, {7, 4000, 1}, {2000, 2000, 1}};
  int plans = 0, bad = 0;
  for (int sms : {152, 148, 64})
    for (auto& sh : shapes)
      for (int nz = 1; nz <= 300; ++nz)
        for (int halo : {1, 2}) {
          const int extra = halo == 1 ? 4 : 6;   // pass A and the residual; the V-cycle's sweeps
          std::vector<hca::MGLevel> lv(sh[2]);
          std::vector<hca::MGLevel*> set;
          std::vector<int> ids;
          for (int r = 0; r < sh[2]; ++r) {
            lv[r] = hca::MGLevel{};
            lv[r].nx = sh[0];
            lv[r].ny = sh[1];
            lv[r].nz = nz;
            lv[r].pitch = (sh[0] + 3) / 4 * 4;
            hca::march_tile(lv[r], halo);
            set.push_back(&lv[r]);
            ids.push_back(r);
          }
          std::vector<int4> blocks;
          hca::march_blocks(set, ids, sms, extra, blocks);
          ++plans;
          int most = 0;
          long long planes = 0;
          bool ok = true;
          for (const int4& b : blocks) {
            const hca::MGLevel& L = lv[b.x];
            const int n = (b.w - b.z + L.seg - 1) / L.seg;
            most = most > n ? most : n;
            planes += b.w - b.z;
            ok = ok && b.z % L.seg == 0 && b.z < b.w && b.w <= nz && b.z / L.seg + n <= L.nseg;
          }
          ok = ok && planes == (long long)nz * lv[0].tx * lv[0].ty * sh[2];
          if (most > hca::kMaxSeg || !ok) {
            if (++bad <= 20)
              std::printf("bad: %d x %d x %d, %d replicates, halo %d, %d multiprocessors: %d segments\n", sh[0], sh[1], nz,
                          sh[2], halo, sms, most);
          }
        }
  std::printf("plans %d bad %d\n", plans, bad);
  return bad != 0;
}
