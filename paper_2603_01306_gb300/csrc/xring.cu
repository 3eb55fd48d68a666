// Plan of the passes over FP32 and FP64 X with one product z.
#include <algorithm>
#include <cmath>

#include "launch.cuh"
#include "xring.cuh"

namespace relax {

// Strips (at most 192 vectors: one per lane of the six axpy warps, six per lane
// of a dot warp) x row groups (at least two blocks of 16 rows each).  The
// float-float pass is bound by its sums: the choice with the least work of the
// busiest CTA, a block's axpy taking as long as dot products with six vectors
// per lane.  The FP32 pass is bound by X: the choice that keeps the most SMs
// busy, strips under 2 KB counted as streaming less efficiently.
template <typename TX, bool FF, int ROWS>
static const void* ring_ptr(int NB) {
  return NB == 1 ? reinterpret_cast<const void*>(&xring_kernel<TX, 1, FF, ROWS>)
                 : reinterpret_cast<const void*>(&xring_kernel<TX, 2, FF, ROWS>);
}

cudaError_t xring_plan(XSPlan& pl, int xk, bool f64acc, int NB, int64_t n, int64_t p) {
  const bool dbl = xk == XK_F64, ff = f64acc && !dbl;
  const int es = xkind_esize(xk), vec = xkind_vec(xk);
  pl = XSPlan{};
  pl.xk = xk;
  pl.cert = f64acc;
  pl.NF = 1;
  pl.NB = NB;
  pl.words = 2;
  pl.keep = x_fits_l2(xk, n, p);
  if (NB < 1 || NB > 2 || n < 1 || p < 1 || n > INT32_MAX || p > INT32_MAX) return cudaErrorNotSupported;
  pl.B = dbl || ff || pl.keep ? 16 : 8;   // (both sides: xring.cuh)
  pl.kernel = dbl           ? ring_ptr<double, false, 16>(NB)
              : ff          ? ring_ptr<float, true, 16>(NB)
              : pl.B == 16 ? ring_ptr<float, false, 16>(NB)
                            : ring_ptr<float, false, 8>(NB);
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t nvec = (p + vec - 1) / vec, cap = 32 * XF_TV;
  pl.nblk = (int)((n + pl.B - 1) / pl.B);
  const int64_t most = std::max<int64_t>(1, ((n + 15) / 16 + 1) / 2);
  double best = 0.0;
  for (int64_t gc = (nvec + cap - 1) / cap; gc <= std::min<int64_t>({(int64_t)nsm, nvec, (int64_t)255}); ++gc) {
    const int64_t v = (nvec + gc - 1) / gc;
    const int64_t nbox = (v * vec + 255) / 256, vpb = (v + nbox - 1) / nbox;
    const int64_t gcc = (nvec + nbox * vpb - 1) / (nbox * vpb);
    if (nbox * vpb > cap || gcc > nsm) continue;
    const int64_t gr = std::max<int64_t>(1, std::min<int64_t>(nsm / gcc, most));
    const double score = ff ? 1.0 / ((double)((pl.nblk + gr - 1) / gr) * (double)(XF_TV + (nbox * vpb + 31) / 32))
                            : (double)(gcc * gr) * std::sqrt(std::min(1.0, (double)(v * 16) / 2048.0));
    if (score <= best * 1.0001) continue;   // fewer strips where the score is the same
    best = score;
    pl.nbox = (int)nbox;
    pl.inner = (int)(vpb * vec);
    pl.sw = nbox * pl.inner;
    pl.Gc = (int)gcc;
    pl.Gr = (int)gr;
  }
  if (best == 0.0) return cudaErrorNotSupported;   // p wider than nsm strips
  pl.boxb = (pl.B * pl.inner * es + 127) / 128 * 128;
  pl.SA = ff ? XF<float, true, 16>::SA : dbl ? XF<double, false, 16>::SA : XF<float, false, 8>::SA;
  pl.SB = XF_TV;
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
  if ((e = raise_smem(pl.kernel, pl.smem)) != cudaSuccess) return e;
  int per = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pl.kernel, pl.threads, pl.smem);
  if (e != cudaSuccess) return e;
  return per >= 1 && per * nsm >= pl.grid ? cudaSuccess : cudaErrorNotSupported;
}

}  // namespace relax
