// Instantiations, plan and launch of the strip-stationary fused pass.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "launch.cuh"

namespace relax {

template <typename TX, typename TA, int NF, int NB, bool FF = false>
static const void* kptr() {
  return reinterpret_cast<const void*>(&xstrip_kernel<TX, TA, NF, NB, FF>);
}

// the certificate of two different vectors; FP32 X in float-float arithmetic
static const void* xstrip_ptr(int xk, bool f64acc, int NF, int NB) {
  if (NF != 2 || NB != 1) return nullptr;
  if (xk == XK_F64) return kptr<double, double, 2, 1>();
  if (xk == XK_F32 && f64acc) return kptr<float, float, 2, 1, true>();
  return nullptr;
}

static int xs_tv(int vec) { return vec == 2 ? XSShape<2>::TV : XSShape<4>::TV; }

// Shape of the pass for an n x p design.
//  * strips of a row of at most 32*TV vectors (the registers of one lane
//    row), chosen to keep the most SMs busy (Gc strips x Gr row groups), at
//    least 2 KB wide where possible;
//  * a strip is nbox tensor boxes of `inner` <= 256 columns;
//  * blocks of B <= 16 rows so that a stage is about 40 KB; 3 + 3 warps and
//    as many stages per warp as shared memory holds (ring A first);
//  * phase A may lead phase B by `lag` blocks: about 64 MB of X in L2 (at
//    least 20 blocks with four or more row groups).
// Lags and row groups were measured on the loop's passes while this kernel ran
// them; the certificate of two different vectors kept the choices.
cudaError_t xstrip_plan(XSPlan& pl, int xk, bool f64acc, int NF, int NB, int64_t n, int64_t p) {
  if ((xk == XK_BF16 || xk == XK_FP8) && !f64acc && NF == 1) return xmma_plan(pl, xk, NB, n, p);
  if ((xk == XK_F32 || xk == XK_F64) && NF == 1) return xring_plan(pl, xk, f64acc, NB, n, p);
  pl = XSPlan{};
  pl.xk = xk;
  pl.cert = f64acc;
  pl.NF = pl.words = NF;
  pl.NB = NB;
  pl.kernel = xstrip_ptr(xk, f64acc, NF, NB);
  if (!pl.kernel || n < 1 || p < 1 || n > INT32_MAX || p > INT32_MAX) return cudaErrorNotSupported;
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int es = xkind_esize(xk);
  const int vec = xkind_vec(xk);
  // strips: over the number of row groups Gr, the strip width (at most `cap`
  // vectors) that keeps the most SMs busy, strips under 2 KB counted as
  // streaming less efficiently
  const int64_t nvec = (p + vec - 1) / vec;
  const int64_t cap = (int64_t)32 * xs_tv(vec);
  int64_t vps = 0;
  double best = -1.0;
  for (int64_t gr = 1; gr <= nsm; ++gr) {
    int64_t gc = std::min<int64_t>(nsm / gr, nvec);
    if (gc < 1) break;
    const int64_t v = (nvec + gc - 1) / gc;
    if (v > cap) continue;
    gc = (nvec + v - 1) / v;
    if (gr > 1 && n < gr * 16) break;   // too few rows to keep the groups busy
    const double score = (double)(gc * gr) * std::sqrt(std::min(1.0, (double)(v * 16) / 2048.0));
    if (score > best * 1.0001) { best = score; vps = v; }
  }
  if (vps <= 0 || vps > cap) return cudaErrorNotSupported;   // p wider than nsm strips of one lane row
  const int64_t cols = vps * vec;
  const int64_t nbox = (cols + 255) / 256;
  const int64_t inner = ((cols + nbox - 1) / nbox + vec - 1) / vec * vec;
  pl.inner = (int)inner;
  pl.nbox = (int)nbox;
  pl.sw = nbox * inner;
  if (pl.sw / vec > cap) return cudaErrorNotSupported;
  const int64_t Gc = (p + pl.sw - 1) / pl.sw;
  pl.Gc = (int)Gc;
  // blocks
  int64_t B = std::max<int64_t>(1, std::min<int64_t>(XS_MAXB, 40960 / (pl.sw * es)));
  B = std::min<int64_t>(B, n);
  auto boxb = [&](int64_t b) { return (b * inner * es + 127) / 128 * 128; };
  const size_t fixed = 2048 + 128;   // static shared memory, alignment slack
  auto fits = [&](int64_t b, int sa, int sb) {
    return (size_t)(sa + sb) * (size_t)(nbox * boxb(b)) + fixed <= (size_t)optin;
  };
  while (B > 1 && !fits(B, 3, 3)) --B;
  const int SA = 3, SB = 3;   // 2 + SA + SB warps <= 8
  static_assert(2 + 3 + 3 <= XS_MAXT / 32);
  if (!fits(B, SA, SB)) return cudaErrorNotSupported;
  // ring depths: stages per warp.  A stage is held from its TMA issue until
  // its warp has read the block, so small blocks (narrow element types) need
  // more of them to keep enough of X in flight; ring A (HBM) first, then
  // ring B (L2), while shared memory allows
  int mA = 1, mB = 1;
  while ((mA + 1) * SA <= XS_MAXR && fits(B, (mA + 1) * SA, mB * SB)) ++mA;
  if (mA > 1 && (mB + 1) * SB <= XS_MAXR && fits(B, mA * SA, (mB + 1) * SB)) ++mB;
  if (mA * SA > XS_MAXR || mB * SB > XS_MAXR || !fits(B, mA * SA, mB * SB)) return cudaErrorNotSupported;
  pl.RA = mA * SA;
  pl.RB = mB * SB;
  pl.B = (int)B;
  pl.boxb = (int)boxb(B);
  pl.nblk = (int)((n + B - 1) / B);
  pl.SA = SA;
  pl.SB = SB;
  pl.Gr = (int)std::max<int64_t>(1, std::min<int64_t>(nsm / Gc, pl.nblk));
  // at least two blocks per CTA: a row group costs the p-phase one partial of
  // X'r per column, and the pass little (loop passes, 1000 x 1000 FP32, 63 -> 32
  // groups: pass 21.7 -> 20.8 us, p-phase 31.6 -> 29.2; 500 x 1000 FP64, 30 ->
  // 16: 30.9 -> 30.6, 33.7 -> 29.7; fewer still and the pass loses more)
  pl.Gr = std::max(1, std::min(pl.Gr, (pl.nblk + 1) / 2));
  const double row_bytes = (double)p * es;
  pl.lag = (int)std::max(4.0, std::min(64.0, 64.0e6 / (B * row_bytes * pl.Gr)));
  // tall designs (four or more row groups): a deeper lead measured faster
  // (100000 x 20000 logistic loop pass: lag 12 -> 20, 0.28 -> 0.43 of the copy
  // bandwidth) although it holds more of X than L2 does
  if (pl.Gr >= 4) pl.lag = std::max(pl.lag, 20);
  pl.grid = pl.Gc * pl.Gr;
  pl.threads = 32 * (2 + SA + SB);   // two producers, SA dot, SB axpy
  // the combine of the axpy warps' strip sums reuses the rings
  const size_t ring = (size_t)(pl.RA + pl.RB) * nbox * pl.boxb;
  const size_t comb = (size_t)SB * NB * pl.sw * 8;
  pl.smem = std::max(ring, comb) + 128;
  if (pl.smem + 2048 > (size_t)optin) return cudaErrorNotSupported;
  cudaError_t e = raise_smem(pl.kernel, pl.smem);
  if (e != cudaSuccess) return e;
  int per = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pl.kernel, pl.threads, pl.smem);
  if (e != cudaSuccess) return e;
  if (per < 1 || per * nsm < pl.grid) return cudaErrorNotSupported;
  return cudaSuccess;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

cudaError_t xstrip_bind(XSPlan& pl, const void* X, int64_t ldx, int64_t n, int64_t p) {
  const int es = xkind_esize(pl.xk);
  if ((reinterpret_cast<uintptr_t>(X) & 15u) != 0 || ((size_t)ldx * es) % 16 != 0 || ldx < p)
    return cudaErrorInvalidValue;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const CUtensorMapDataType dt = pl.xk == XK_F64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                                 : pl.xk == XK_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : pl.xk == XK_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                    : CU_TENSOR_MAP_DATA_TYPE_UINT8;
  const cuuint64_t dims[2] = {(cuuint64_t)p, (cuuint64_t)n};
  const cuuint64_t strides[1] = {(cuuint64_t)ldx * es};
  const cuuint32_t box[2] = {(cuuint32_t)pl.inner, (cuuint32_t)pl.B};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(&pl.tm, dt, 2, const_cast<void*>(X), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The per-pass area zeroed before every launch:
//   cnt[nblk] | zcnt | zmax[2] | zfix[words of a row x n]
static size_t zero_off_zcnt(const XSPlan& pl) { return ((size_t)pl.nblk * sizeof(unsigned) + 15) / 16 * 16; }
size_t xstrip_zero_bytes(const XSPlan& pl, int64_t n) {
  return (zero_off_zcnt(pl) + 32 + (size_t)pl.words * n * sizeof(unsigned long long) + 15) / 16 * 16;
}
void xstrip_zero_layout(const XSPlan& pl, void* base, XSArgs& a) {
  unsigned char* b = static_cast<unsigned char*>(base);
  const size_t oz = zero_off_zcnt(pl);
  a.cnt = reinterpret_cast<unsigned*>(b);
  a.zcnt = reinterpret_cast<unsigned*>(b + oz);
  a.zmax = reinterpret_cast<unsigned long long*>(b + oz + 16);
  a.zfix = reinterpret_cast<unsigned long long*>(b + oz + 32);
}

// Three quarters of L2: an X below that is found there by the next pass (4000 x
// 4000 FP32 29.2 -> 29.0 us, certificates at 2000 x 5000 28.8 -> 27.5), a larger
// one only pushes out the vectors that are (20000 x 50000: p-phase 57 -> 71 us).
bool x_fits_l2(int xk, int64_t n, int64_t p) {
  int dev = 0, l2 = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
  return (double)n * (double)p * xkind_esize(xk) <= 0.75 * (double)l2;
}

cudaError_t xstrip_launch(const XSPlan& pl, const XSArgs& a, bool clear, cudaStream_t st) {
  if (clear) {
    const cudaError_t e = cudaMemsetAsync(a.cnt, 0, xstrip_zero_bytes(pl, a.n), st);
    if (e != cudaSuccess) return e;
  }
  if (pl.mma) return xmma_launch(pl, a, st);
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
  void* args[1] = {(void*)&a};
  return cudaLaunchKernelExC(&cfg, pl.kernel, args);
}

}  // namespace relax
