// Plan of the float-float pass over FP32 X.
#include <algorithm>

#include "launch.cuh"
#include "xff.cuh"

namespace relax {

// Strips x row groups: the choice with the least work of the busiest CTA, a
// block's six axpy warps taking as long as a dot warp with six vectors per lane.
cudaError_t xff_plan(XSPlan& pl, int NB, int64_t n, int64_t p) {
  pl = XSPlan{};
  pl.xk = XK_F32;
  pl.cert = true;
  pl.NF = 1;
  pl.NB = NB;
  pl.words = 2;
  if (NB < 1 || NB > 2 || n < 1 || p < 1 || n > INT32_MAX || p > INT32_MAX) return cudaErrorNotSupported;
  pl.kernel = NB == 1 ? reinterpret_cast<const void*>(&xff_kernel<1>) : reinterpret_cast<const void*>(&xff_kernel<2>);
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t nvec = (p + 3) / 4, cap = 32 * XF_TV;
  pl.B = XF_B;
  pl.nblk = (int)((n + XF_B - 1) / XF_B);
  int64_t best = INT64_MAX;
  for (int64_t gc = (nvec + cap - 1) / cap; gc <= std::min<int64_t>({(int64_t)nsm, nvec, (int64_t)255}); ++gc) {
    const int64_t v = (nvec + gc - 1) / gc;
    const int64_t nbox = (v * 4 + 255) / 256, vpb = (v + nbox - 1) / nbox;
    const int64_t gcc = (nvec + nbox * vpb - 1) / (nbox * vpb);
    if (nbox * vpb > cap || gcc > nsm) continue;
    const int64_t gr = std::max<int64_t>(1, std::min<int64_t>(nsm / gcc, (pl.nblk + 1) / 2));
    const int64_t cost = (pl.nblk + gr - 1) / gr * (XF_TV + (nbox * vpb + 31) / 32);
    if (cost >= best) continue;   // fewer strips where the cost is the same
    best = cost;
    pl.nbox = (int)nbox;
    pl.inner = (int)(vpb * 4);
    pl.sw = nbox * pl.inner;
    pl.Gc = (int)gcc;
    pl.Gr = (int)gr;
  }
  if (best == INT64_MAX) return cudaErrorNotSupported;   // p wider than nsm strips
  pl.boxb = XF_B * pl.inner * 4;
  pl.boxb = (pl.boxb + 127) / 128 * 128;
  pl.SA = XF_SA;
  pl.SB = XF_SB;
  pl.grid = pl.Gc * pl.Gr;
  pl.threads = XF_T;
  const size_t stage = (size_t)pl.nbox * pl.boxb;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaFuncGetAttributes(&fa, pl.kernel);
  if (e != cudaSuccess) return e;
  pl.RA = (int)std::min<size_t>(XF_MAXR, ((size_t)optin - fa.sharedSizeBytes - 128) / stage);
  pl.RB = 0;
  if (pl.RA < 2) return cudaErrorNotSupported;
  pl.smem = (size_t)pl.RA * stage + 128;
  if (fa.maxDynamicSharedSizeBytes < (int)pl.smem) {
    e = cudaFuncSetAttribute(pl.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem);
    if (e != cudaSuccess) return e;
  }
  int per = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pl.kernel, pl.threads, pl.smem);
  if (e != cudaSuccess) return e;
  return per >= 1 && per * nsm >= pl.grid ? cudaSuccess : cudaErrorNotSupported;
}

}  // namespace relax
