// complex64 instantiations of the 3-D GMRES step kernels (hh_gmres3d.cuh), and
// the split of the work.
#include "hh_gmres3d.cuh"

namespace hh {

HH_GM3D_INST(float)

// Planes per run: about eight blocks per SM over the batch for the vector kernels
// (latency), two for the Gram kernel (every block of the update adds its sums).
Gm3dPlan gm3d_plan(int N, int batch, int sms) {
  Gm3dPlan p;
  const int tiles = ((N + kBX - 1) / kBX) * ((N + kBY - 1) / kBY);
  auto split = [&](int per, int *planes, int *blocks) {
    const int runs = std::max(1, per * sms / (tiles * batch));
    *planes = (N + runs - 1) / runs;
    *blocks = tiles * ((N + *planes - 1) / *planes);
  };
  split(8, &p.vplanes, &p.vblocks);
  split(2, &p.planes, &p.blocks);
  const int pts = (N * N * (N + 1) + 255) / 256;
  p.ublocks = std::min(pts, std::max(1, 4 * sms / batch));
  return p;
}

}  // namespace hh
