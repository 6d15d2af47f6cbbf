// Instantiations of the 3-D pencil kernels (FP32, windows of up to 16 taps).
#include "points_pencil.cuh"

namespace gbnfft {

PencilLaunch pencil_launch_f32(int taps, bool spread) {
  PencilLaunch l{};
#define GBNFFT_PENCIL(W, NR)                                                                               \
  if (taps == W) {                                                                                         \
    l.fn = spread ? reinterpret_cast<const void*>(&k_spread_pencil<W, NR>)                                 \
                  : reinterpret_cast<const void*>(&k_interp_pencil<W, NR>);                                \
    l.threads = spread ? PencilShape<W, NR>::THREADS : SlabShape<W, NR>::THREADS;                          \
    l.smem = spread ? pencil_smem_bytes<W, NR>() : SlabShape<W, NR>::smem_bytes();                         \
    l.slab_points = slab_points(W);                                                                        \
    l.edge = 8 * NR + 1 - W;                                                                               \
  }
  GBNFFT_PENCIL_CASES(GBNFFT_PENCIL)
#undef GBNFFT_PENCIL
  return l;
}

}  // namespace gbnfft
