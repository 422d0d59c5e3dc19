// complex64 instantiations of the 3-D GMRES step kernels (hh_gmres3d.cuh), and
// the split of the work.
#include "hh_gmres3d.cuh"

namespace hh {

HH_GM3D_INST(float)

// Planes per run: about eight blocks per SM over the batch for the vector kernels
// (latency), two for the Gram kernel (every block of the update adds its sums).  In
// complex128, where the FP64 pipe of the busy SMs is the bound, the Gram kernel has 64
// blocks per right-hand side if runs of four planes give them: with 16 at 63^3 a solve
// of 16 whose other twelve had stopped took 2949 us a cycle.
Gm3dPlan gm3d_plan(int N, int batch, int sms, bool fp64) {
  Gm3dPlan p;
  const int tiles = ((N + kBX - 1) / kBX) * ((N + kBY - 1) / kBY);
  auto split = [&](int per, int least, int *planes, int *blocks) {
    const int runs = std::max(least, per * sms / (tiles * batch));
    *planes = (N + runs - 1) / runs;
    *blocks = tiles * ((N + *planes - 1) / *planes);
  };
  split(8, 1, &p.vplanes, &p.vblocks);
  split(2, fp64 ? std::max(1, std::min(64 / tiles, N / 4)) : 1, &p.planes, &p.blocks);
  const int pts = (N * N * (N + 1) + 255) / 256;
  p.ublocks = std::min(pts, std::max(1, 4 * sms / batch));
  return p;
}

}  // namespace hh
