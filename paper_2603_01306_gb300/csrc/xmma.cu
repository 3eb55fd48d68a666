// Instantiations, plan and launch of the tensor-core pass over BF16 / FP8
// storage of X.
#include <algorithm>
#include <cmath>

#include "launch.cuh"
#include "xmma.cuh"

namespace relax {

static const void* xmma_ptr(int xk, int NB) {
  if (xk == XK_BF16)
    return NB == 1 ? reinterpret_cast<const void*>(&xmma_kernel<__nv_bfloat16, 1>)
                   : reinterpret_cast<const void*>(&xmma_kernel<__nv_bfloat16, 2>);
  return NB == 1 ? reinterpret_cast<const void*>(&xmma_kernel<__nv_fp8_e4m3, 1>)
                 : reinterpret_cast<const void*>(&xmma_kernel<__nv_fp8_e4m3, 2>);
}

// boxes and steps of a strip of `vps` 16-byte vectors: box rows of an odd
// number of vectors, at most 256 elements wide
static void xmma_shape(int64_t vps, int vec, int64_t& nbox, int64_t& vpb, int64_t& steps) {
  const int64_t most = 256 / vec - 1;   // odd
  nbox = (vps + most - 1) / most;
  vpb = (vps + nbox - 1) / nbox;
  vpb += 1 - vpb % 2;
  steps = nbox * ((vpb + 1) / 2);
}

// The strips and row groups are chosen as xstrip_plan does; blocks have 16
// rows (the MMA's M or K), a strip at most the steps whose fragments the dot
// warps hold in registers.
cudaError_t xmma_plan(XSPlan& pl, int xk, int NB, int64_t n, int64_t p) {
  pl = XSPlan{};
  pl.xk = xk;
  pl.NF = 1;
  pl.NB = NB;
  pl.words = 2;
  pl.mma = true;
  pl.keep = x_fits_l2(xk, n, p);
  if ((xk != XK_BF16 && xk != XK_FP8) || NB < 1 || NB > 2 || n < 1 || p < 1 || n > INT32_MAX || p > INT32_MAX)
    return cudaErrorNotSupported;
  pl.kernel = xmma_ptr(xk, NB);
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int vec = xkind_vec(xk);
  const int64_t most = xk == XK_BF16 ? XMShape<__nv_bfloat16>::STEPS : XMShape<__nv_fp8_e4m3>::STEPS;
  const int64_t nvec = (p + vec - 1) / vec;
  int64_t vps = 0, nbox, vpb, steps;
  double best = -1.0;
  for (int64_t gr = 1; gr <= nsm; ++gr) {
    int64_t gc = std::min<int64_t>({(int64_t)nsm / gr, nvec, (int64_t)255});   // a row's arrivals are counted in eight bits
    if (gc < 1) break;
    const int64_t v = (nvec + gc - 1) / gc;
    xmma_shape(v, vec, nbox, vpb, steps);
    if (steps > most) continue;
    gc = (nvec + nbox * vpb - 1) / (nbox * vpb);
    if (gr > 1 && n < gr * 16) break;   // too few rows to keep the groups busy
    const double score = (double)(gc * gr) * std::sqrt(std::min(1.0, (double)(v * 16) / 1024.0));
    if (score > best * 1.0001) { best = score; vps = v; }
  }
  if (vps <= 0) return cudaErrorNotSupported;
  xmma_shape(vps, vec, nbox, vpb, steps);
  pl.nbox = (int)nbox;
  pl.vpb = (int)vpb;
  pl.spb = (int)((vpb + 1) / 2);
  pl.steps = (int)steps;
  pl.inner = (int)(vpb * vec);
  pl.sw = nbox * pl.inner;
  pl.Gc = (int)((p + pl.sw - 1) / pl.sw);
  pl.B = 16;
  pl.boxb = (int)((16 * vpb * 16 + 16 + 127) / 128 * 128);   // a zeroed tail: a row's last step reads 16 bytes on
  pl.nblk = (int)((n + 15) / 16);
  pl.Gr = (int)std::max<int64_t>(1, std::min<int64_t>(nsm / pl.Gc, (pl.nblk + 1) / 2));
  pl.SA = XM_SA;
  pl.SB = XM_SB;
  pl.grid = pl.Gc * pl.Gr;
  pl.threads = XM_T;
  // the ring: every stage that shared memory holds (the blocks in flight
  // between HBM and the end of their agreement)
  const size_t stage = (size_t)nbox * pl.boxb, extra = (size_t)most * 256 * (xk == XK_BF16 ? 1 : 2) + 128, fixed = 8192;
  pl.RA = std::min<int>(XM_MAXR, (int)(((size_t)optin - fixed - extra) / stage));
  pl.RB = 0;
  if (pl.RA < 2) return cudaErrorNotSupported;
  pl.smem = (size_t)pl.RA * stage + extra;
  cudaError_t e = raise_smem(pl.kernel, pl.smem);
  if (e != cudaSuccess) return e;
  int per = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pl.kernel, pl.threads, pl.smem);
  if (e != cudaSuccess) return e;
  return per >= 1 && per * nsm >= pl.grid ? cudaSuccess : cudaErrorNotSupported;
}

cudaError_t xmma_launch(const XSPlan& pl, const XSArgs& a, cudaStream_t st) {
  XMArgs xa;
  xa.a = a;
  xa.vpb = pl.vpb;
  xa.spb = pl.spb;
  xa.steps = pl.steps;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(pl.grid, 1, 1);
  cfg.blockDim = dim3(pl.threads, 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[1] = {(void*)&xa};
  return cudaLaunchKernelExC(&cfg, pl.kernel, args);
}

}  // namespace relax
