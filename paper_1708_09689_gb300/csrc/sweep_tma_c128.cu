// Instantiations of the TMA-staged sweep (sweep_tma.cuh) for complex128 TI
// vectors, the choice of untuned complex128 TI sweeps of large blocks.  A
// complex128 site of R vectors has the byte layout of a complex64 site of 2R
// vectors, so the tiles, rings and swizzle of layout 2R serve it (R = 16, 32,
// 64: slices of 8 vectors on the tiles of layout 16); each thread updates one
// vector of one site, sixteen warps on the large tile.  Sixteen warps leave 128
// registers a thread, and every instantiation spills some of the eight aligned
// sums and the tile offsets (the R = 8 KPM sweep 164 bytes of stores and 208 of
// loads); eight warps on the same tile took 995 us where these take 898.  This
// unit's kernels report copy-wait timeouts in its own error word.
#include "sweep_tma.cuh"

namespace pvsc {

template <int R2>
static void tiles_of(const Geometry& g, int64_t* n, double* full) {
  using L = TmaLayout<R2, false, 16>;
  const int64_t tx = (g.L[0] + L::TX - 1) / L::TX, ty = (g.L[1] + L::TY - 1) / L::TY;
  *n = tx * ty;
  *full = (double)(g.L[0] * g.L[1]) / (double)(tx * L::TX * ty * L::TY);
}

// An untuned complex128 sweep runs the tiles with 2^20 site-vectors and tiles three quarters full:
// sixteen warps and no wait on HBM against the eight of the register march, for a longer launch and
// a second read of the neighbours from shared memory.  KPM sweeps, march -> tiles, us: 128x128x64
// R = 8: 1031 -> 895, R = 1: 149 -> 142; 64x64x64 R = 8: 275 -> 241, R = 2: 77 -> 80; 128x128x8 R = 8:
// 143 -> 142; 32x32x32 R = 16: 77 -> 78; 101x87x53 R = 1 (tiles 0.71 full): 70 -> 92, R = 8: 489 -> 425.
bool tma_c128_default(const pvsc_lattice* lat, int R) {
  const Geometry& g = lat->g;
  if (g.model != PVSC_TI || g.zhalo || g.n_sites * R < (1 << 20) || g.L[0] >= 65536 || g.L[1] >= 65536 ||
      g.L[2] >= 65536)
    return false;
  int64_t n;
  double full;
  if (R == 1) tiles_of<2>(g, &n, &full);
  else if (R == 2) tiles_of<4>(g, &n, &full);
  else if (R == 4) tiles_of<8>(g, &n, &full);
  else tiles_of<16>(g, &n, &full);
  const int64_t SL = R > 8 ? R / 8 : 1;
  return full >= 0.75 && n <= (int64_t)kTmaUnitsPerSm * (lat->sm_count / SL);
}

int launch_sweep_tma_c128(const pvsc_lattice* lat, int feat, Sweep& p, cudaStream_t st) {
  const LaunchShape sh;
  constexpr int F = kModelTIC128;
  switch (p.R) {
    case 1: return launch_tma_r<2, false, 16, F>(lat, feat, p, sh, st);
    case 2: return launch_tma_r<4, false, 16, F>(lat, feat, p, sh, st);
    case 4: return launch_tma_r<8, false, 16, F>(lat, feat, p, sh, st);
    case 8: return launch_tma_r<16, false, 16, F>(lat, feat, p, sh, st);
    case 16: return launch_tma_r<16, false, 16, F, 2>(lat, feat, p, sh, st);
    case 32: return launch_tma_r<16, false, 16, F, 4>(lat, feat, p, sh, st);
    default: return launch_tma_r<16, false, 16, F, 8>(lat, feat, p, sh, st);
  }
}

int tma_error_c128(int clear, int* flag) {
  int h = 0;
  PVSC_CUDA_TRY(cudaMemcpyFromSymbol(&h, g_tma_sweep_error, sizeof(int)));
  if (clear) {
    const int z = 0;
    PVSC_CUDA_TRY(cudaMemcpyToSymbol(g_tma_sweep_error, &z, sizeof(int)));
  }
  *flag = h;
  return PVSC_OK;
}

}  // namespace pvsc
