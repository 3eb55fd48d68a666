// Fused pass over a BF16 or FP8 copy of X (the loop's storage of the
// low-precision configurations): z = X beta, r = link(z), g = X' r, with X read
// from HBM once, both products on the tensor cores.
//
// Strips x row groups as in xstrip.cuh, z in fixed point; what differs:
//  * A tile stays in shared memory from its dot products until its axpy: the
//    ring holds the blocks of one agreement's round trip, X crosses from L2
//    to the SMs once (the second crossing of xstrip.cuh was what its narrow
//    instantiations came to be bound by next to issue).
//  * A row's z takes two words, 54 bits and 44 further ones, that carry their
//    own arrival counts in the low eight bits: a block is agreed on by polling
//    its rows' words, no release, no counter, one round trip through L2.  The
//    unit follows from the largest row and the largest |beta_j|, so a row far
//    below that bound needs the second word (with one, a row 10^6 times lighter
//    than the heaviest was off by 9e-5 of itself, by 5e-3 at 10^8).
//  * On the CUDA cores a narrow element costs a conversion and up to three
//    FMAs (BF16 0.37, FP8 0.22 of the copy bandwidth, DRAM 31% busy).  Here a
//    tile of 16 rows x 16 columns costs one ldmatrix and one mma.sync m16n8k16
//    per product.  (tcgen05 would want the small operand in shared memory and
//    M = 128; with one or two right-hand sides the tiles are memory-bound
//    either way, and fragments in registers need no round trip through TMEM.)
//  * The small operand (beta, a block's row weights) is split into four
//    planes, one per column of the MMA's N = 8, so that products are exact and
//    sums FP32.  On a common scale (the largest in [2^4, 2^5)) the first two
//    planes of a value from 1 on are integers of at most six bits, whose sums
//    over the MMA's K come out exactly: the tensor cores truncate, a bias that
//    no later sum removes (with three planes of 8 bits g of 30000 rows was off
//    by 3e-8).  A smaller value takes the last three planes with all their
//    bits: the four hold every FP32 value exactly, FP16 planes (scaled up one
//    by one) down to 2^-34 of the largest.  The sums of one or two MMAs are
//    folded into compensated FP32 pairs.
//  * The link has warps of its own, two blocks each at a time, which leave the
//    weights' fragments in shared memory; an axpy warp owns every SB-th step
//    of the strip.
// FP8: the e4m3 bytes become FP16 values times 2^-8 by shifts (exact, subnormals
// included; a NaN in X makes every z NaN through the bound on the rows), the
// columns taken in whatever order the fragments have them, the same for both
// operands.  A box's rows are an odd number of 16-byte vectors apart, so that
// ldmatrix meets no bank conflict.
#pragma once
#include <cuda_fp16.h>

#include "xstrip.cuh"

namespace relax {

constexpr int XM_SA = 4, XM_NL = 3, XM_SB = 8;               // dot, link and axpy warps
constexpr int XM_T = 32 * (1 + XM_SA + XM_NL + XM_SB);
constexpr int XM_MAXR = 16;                                  // ring stages at most
constexpr int XM_RW = 4 * XM_NL;                             // blocks of weights in shared memory
template <typename TX> struct XMShape {   // 32-byte steps of a strip's row at most
  static constexpr int STEPS = sizeof(TX) == 2 ? 52 : 32;
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
template <bool BF>
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  if constexpr (BF)
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
        "%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
        "%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// bytes 0 and 2 (ev), 1 and 3 (od) of four e4m3 values, as FP16 times 2^-8
__device__ __forceinline__ uint32_t e4m3_ev(uint32_t w) { return ((w << 8) & 0x80008000u) | ((w << 7) & 0x3f803f80u); }
__device__ __forceinline__ uint32_t e4m3_od(uint32_t w) { return (w & 0x80008000u) | ((w >> 1) & 0x3f803f80u); }
// Plane q holds its part times 2^plane_exp (FP16 has five bits of exponent; the
// parts are at most 2^5, 1, 2^-6 and 2^-18, or 0, 1, 2^-12 and 2^-24 of an |x| < 1)
template <bool BF>
__device__ __forceinline__ constexpr int plane_exp(int q) {
  return BF || q == 0 ? 0 : q == 1 ? 15 : q == 2 ? 21 : 33;
}
template <bool BF>
__device__ __forceinline__ float plane_inv(int q) {   // 2^-plane_exp
  return BF ? 1.f : q == 0 ? 1.f : q == 1 ? 0x1p-15f : q == 2 ? 0x1p-21f : 0x1p-33f;
}
// the four planes of x (on the common scale, |x| < 2^5) as the MMA's 16-bit operand
template <bool BF>
__device__ __forceinline__ void planes16(float x, uint16_t (&u)[4]) {
  const bool whole = fabsf(x) >= 1.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float v = q == 0 ? (whole ? rintf(x) : 0.f) : q == 1 && whole ? rintf(x * 32.f) * 0.03125f : x;
    if constexpr (BF) {
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      u[q] = __bfloat16_as_ushort(h);
      x -= __bfloat162float(h);   // exact
    } else {
      const __half h = __float2half_rn(v * (float)(1ull << plane_exp<BF>(q)));
      u[q] = __half_as_ushort(h);
      x -= __half2float(h) * plane_inv<BF>(q);
    }
  }
}
// exponent e with max * 2^e in [2^4, 2^5); 0 for a zero, Inf or NaN max
__device__ __forceinline__ int plane_scale(float mx) {
  if (!(mx > 0.f) || !(mx < INFINITY)) return 0;
  int e;
  frexpf(mx, &e);   // mx < 2^e
  return min(126, 5 - e);
}

constexpr int Z_LO = 44;   // bits of z's second word below the first one's unit

// m 2^sh as hi + lo 2^-Z_LO, in two's complement (|m 2^sh| < 2^54)
__device__ __forceinline__ void fixed_words(float m, int sh, long long& hi, long long& lo) {
  const uint32_t b = __float_as_uint(m);
  const int ex = (int)((b >> 23) & 255u);
  const unsigned long long mant = ex ? (b & 0x7fffffu) | 0x800000u : b & 0x7fffffu;
  const int k = min((ex ? ex : 1) - 150 + sh, 38);   // |m| 2^sh = mant 2^k
  long long h = 0, l = 0;
  if (k >= 0) {
    h = (long long)(mant << k);
  } else {
    const unsigned long long rem = k > -24 ? mant & ((1ull << -k) - 1ull) : mant;
    if (k > -24) h = (long long)(mant >> -k);
    const int s = k + Z_LO;
    l = s >= 0 ? (long long)(rem << s) : s > -32 ? (long long)((rem + (1ull << (-s - 1))) >> -s) : 0ll;
  }
  const bool neg = (b >> 31) != 0u;
  hi += neg ? -h : h;
  lo += neg ? -l : l;
}

// bounded wait until the low eight bits of both words of a row count `want` arrivals
__device__ __forceinline__ bool wait_row(const unsigned long long* p, unsigned want, unsigned long long& h, unsigned long long& l,
                                          uint64_t limit_ns, int* status) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(h), "=l"(l) : "l"(p) : "memory");
    if ((unsigned)(h & 255ull) == want && (unsigned)(l & 255ull) == want) return true;
    if ((it & 15u) == 0u) {
      const uint64_t t = globaltimer_ns();
      if (it == 0) t0 = t;
      else if (t - t0 > limit_ns) {
        atomicCAS(status, ST_OK, ST_TIMEOUT);
        return false;
      }
    }
  }
}

struct XMArgs {
  XSArgs a;
  int vpb;     // 16-byte vectors per box row (odd)
  int spb;     // 32-byte steps per box
  int steps;   // nbox * spb
};

template <typename TX, int NB>
__global__ void __launch_bounds__(XM_T, 1) xmma_kernel(const __grid_constant__ XMArgs xa) {
  constexpr bool BF = sizeof(TX) == 2;
  constexpr int VEC = 16 / (int)sizeof(TX);
  constexpr int STEPS = XMShape<TX>::STEPS;
  constexpr int MM = BF ? 1 : 2;                      // MMAs per step
  const XSArgs& a = xa.a;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[XM_MAXR], empty[XM_MAXR], wfull[XM_RW], wempty[XM_RW];
  __shared__ __align__(16) uint16_t wfrag[XM_RW][8][16];   // [slot][N column][block row]
  __shared__ float wscale[XM_RW];
  __shared__ volatile int tmo;
  __shared__ int skip;
  __shared__ float smax[XM_T / 32];
  __shared__ __align__(16) uint32_t toff[STEPS];   // a step's byte offset in a tile, and its column in the strip
  __shared__ int tcol[STEPS];        // (the second vector of a box's last step does not exist: bit 30)
  __shared__ double lcomb[XM_NL][3];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    tmo = 0;
    skip = a.ps->done;
    for (int s = 0; s < a.RA; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], XM_SB); }
    for (int s = 0; s < XM_RW; ++s) { mbar_init(&wfull[s], 1); mbar_init(&wempty[s], XM_SB); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < STEPS; i += XM_T) {
    const int box = i / xa.spb, st = i - box * xa.spb;
    const bool on = i < xa.steps;
    toff[i] = on ? (uint32_t)box * a.boxb + (uint32_t)st * 32u : 0u;
    tcol[i] = on ? (box * a.inner + 2 * st * VEC) | (2 * st + 1 < xa.vpb ? 0 : 1 << 30) : 0;
  }
  unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  {
    // the boxes' tails, which no copy writes
    const int data = 16 * xa.vpb * 16, tail = (a.boxb - data) / 16, boxes = a.RA * a.nbox;
    for (int i = tid; i < boxes * tail; i += XM_T)
      *reinterpret_cast<int4*>(smem + (size_t)(i / tail) * a.boxb + data + (i % tail) * 16) = make_int4(0, 0, 0, 0);
  }
  __syncthreads();
  if (skip) return;   // uniform (same flag everywhere)

  const int cc = blockIdx.x % a.Gc, cr = blockIdx.x / a.Gc;
  const int64_t n = a.n, p = a.p;
  const int64_t s0 = (int64_t)cc * a.sw;
  const uint32_t pitch = (uint32_t)xa.vpb * 16;
  const uint32_t tilebytes = (uint32_t)a.nbox * 16 * pitch;   // whole boxes, out-of-range parts zero-filled
  const int kloc = (cr < a.nblk) ? (a.nblk - cr + a.Gr - 1) / a.Gr : 0;
  const size_t stage = (size_t)a.nbox * a.boxb;
  // the strip of beta as the MMA's B fragments [step][lane][2 MM]
  uint32_t* frag = reinterpret_cast<uint32_t*>(smem + (size_t)a.RA * stage);

  if (warp == 0) {
    // ------------------------------------------------ producer: HBM -> ring
    if (lane == 0) {
      const uint64_t pol = a.keep ? policy_evict_normal() : policy_evict_first();
      int issued = 0;
      for (int k = 0; k < kloc; ++k) {
        const int s = k % a.RA;
        if (tmo) break;
        if (k >= a.RA && !mbar_wait(&empty[s], ((k / a.RA) - 1) & 1, a.limit_ns, a.status)) { tmo = 1; break; }
        const int y0 = (cr + k * a.Gr) * 16;
        mbar_arrive_expect_tx(&full[s], tilebytes);
        for (int i = 0; i < a.nbox; ++i)
          tma_load_2d(smem + s * stage + (size_t)i * a.boxb, &a.tm, (int)s0 + i * a.inner, y0, &full[s], pol);
        issued = k + 1;
      }
      // let every copy in flight land before the CTA may exit
      for (int k = (issued > a.RA ? issued - a.RA : 0); k < issued; ++k)
        mbar_wait(&full[k % a.RA], (k / a.RA) & 1, a.limit_ns, a.status);
    }
    __syncwarp();
  } else if (warp < 1 + XM_SA) {
    // ------------------------------------------------ phase A: strip dot products
    const int st = warp - 1;
    constexpr int DT = 32 * XM_SA;
    // beta of this thread's columns, at most DC of them
    constexpr int DC = (STEPS * 2 * VEC + DT - 1) / DT;
    float bv[DC];
    float mx = 0.f;
    bool nan = false;
#pragma unroll
    for (int i = 0; i < DC; ++i) {
      const int c = tid - 32 + i * DT;
      const int64_t col = s0 + c;
      bv[i] = 0.f;
      if (c < (int)a.sw && col < p) {
        const double bd = static_cast<const double*>(a.ps->beta)[col];
        bv[i] = a.colscale ? (float)(bd * (double)a.colscale[col]) : (float)bd;
      }
      nan |= bv[i] != bv[i];
      mx = fmaxf(mx, fabsf(bv[i]));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (__any_sync(0xffffffffu, nan)) mx = __int_as_float(0x7fc00000);
    if (lane == 0) smax[warp] = mx;
    for (int i = tid - 32; i < STEPS * 32 * 2 * MM; i += DT) frag[i] = 0u;
    named_sync(1, DT);
    mx = 0.f;
    for (int w = 1; w < 1 + XM_SA; ++w) mx = smax[w] != smax[w] || mx != mx ? __int_as_float(0x7fc00000) : fmaxf(mx, smax[w]);
    if (st == 0 && lane == 0) {
      // this CTA's max |beta_j| (NaN dominates: its bits compare above +Inf)
      atomicMax(&a.zmax[0], (unsigned long long)__double_as_longlong(fabs((double)mx)));
      __threadfence();
      atomicAdd(a.zcnt, 1u);
    }
    const int be = plane_scale(mx);
    const float bsc = ldexpf(1.f, be);
    // Column n of B holds plane n / 2 if n is even (the others stay zero), so
    // that a lane's sums are all of one plane.  BF16: register i = vector
    // v0 + i, columns 2t, 2t + 1; FP8: MMA i / 2 = vector v0 + i / 2, columns
    // 4t + (i & 1), + 2.
#pragma unroll
    for (int i = 0; i < DC; ++i) {
      const int c = tid - 32 + i * DT;
      if (c < (int)a.sw) {
        const int box = c / a.inner, cb = c - box * a.inner, v = cb / VEC, el = cb - v * VEC;
        const int st2 = box * xa.spb + (v >> 1);
        const int reg = BF ? v & 1 : 2 * (v & 1) + (el & 1), t = BF ? el >> 1 : el >> 2, half = BF ? el & 1 : (el >> 1) & 1;
        uint16_t u[4];
        planes16<BF>(bv[i] * bsc, u);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          reinterpret_cast<uint16_t*>(frag + ((st2 * 32 + 8 * q + t) * 2 * MM + reg))[half] = u[q];
      }
    }
    named_sync(1, DT);
    const uint32_t* fl = frag + lane * 2 * MM;
    int zs = 0;
    bool have_scale = false;
    // this lane's row of the four matrices: rows 0-7, 8-15 of vector v0, then of v0 + 1
    const uint32_t rowoff = (uint32_t)(lane & 15) * pitch + (uint32_t)(lane >> 4) * 16;
    for (int k = st; k < kloc; k += XM_SA) {
      if (tmo) break;
      const int sa = k % a.RA;
      if (!__all_sync(0xffffffffu, mbar_wait(&full[sa], (k / a.RA) & 1, a.limit_ns, a.status))) {
        tmo = 1;
        break;
      }
      const int b = cr + k * a.Gr;
      const int64_t r0 = (int64_t)b * 16;
      const int rows = (int)((n - r0) < 16 ? (n - r0) : 16);
      // a step's lanes of the second vector may read past a box's row (the next
      // row, or the box's zeroed tail), against zeros
      const uint32_t base = smem_u32(smem + sa * stage) + rowoff;
      // four MMAs at a time, two chained per sum: rows g, g + 8 of the lane's
      // plane in the pairs (hi, lo).  A rolled loop: unrolled, with the
      // fragments in registers, the FP8 kernel waited for instructions a third
      // of its time (25000 x 20000: 924 us, BF16 305; rolled 277 and 246).
      float2 hi0 = make_float2(0.f, 0.f), lo0 = hi0, hi1 = hi0, lo1 = hi0;
      constexpr int GS = BF ? 4 : 2;   // steps per group
#pragma unroll 2
      for (int s = 0; s < xa.steps; s += GS) {   // (steps past the last read the first tile's start, against zeros)
        uint32_t r[GS][4], f[GS][2 * MM], to[GS];
        if constexpr (BF) *reinterpret_cast<uint4*>(to) = *reinterpret_cast<const uint4*>(toff + s);
        else *reinterpret_cast<uint2*>(to) = *reinterpret_cast<const uint2*>(toff + s);
#pragma unroll
        for (int u = 0; u < GS; ++u) {
          ldsm4(r[u], base + to[u]);
          if constexpr (BF) *reinterpret_cast<uint2*>(f[u]) = *reinterpret_cast<const uint2*>(fl + (s + u) * 64);
          else *reinterpret_cast<uint4*>(f[u]) = *reinterpret_cast<const uint4*>(fl + (s + u) * 128);
        }
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (BF) {
          mma16816<BF>(d0, r[0][0], r[0][1], r[0][2], r[0][3], f[0][0], f[0][1]);
          mma16816<BF>(d1, r[1][0], r[1][1], r[1][2], r[1][3], f[1][0], f[1][1]);
          mma16816<BF>(d0, r[GS - 2][0], r[GS - 2][1], r[GS - 2][2], r[GS - 2][3], f[GS - 2][0], f[GS - 2][1]);
          mma16816<BF>(d1, r[GS - 1][0], r[GS - 1][1], r[GS - 1][2], r[GS - 1][3], f[GS - 1][0], f[GS - 1][1]);
        } else {
          mma16816<BF>(d0, e4m3_ev(r[0][0]), e4m3_ev(r[0][1]), e4m3_od(r[0][0]), e4m3_od(r[0][1]), f[0][0], f[0][1]);
          mma16816<BF>(d1, e4m3_ev(r[1][0]), e4m3_ev(r[1][1]), e4m3_od(r[1][0]), e4m3_od(r[1][1]), f[1][0], f[1][1]);
          mma16816<BF>(d0, e4m3_ev(r[0][2]), e4m3_ev(r[0][3]), e4m3_od(r[0][2]), e4m3_od(r[0][3]), f[0][2 * MM - 2], f[0][2 * MM - 1]);
          mma16816<BF>(d1, e4m3_ev(r[1][2]), e4m3_ev(r[1][3]), e4m3_od(r[1][2]), e4m3_od(r[1][3]), f[1][2 * MM - 2], f[1][2 * MM - 1]);
        }
        two_sum_acc2(hi0, lo0, make_float2(d0[0], d0[2]));   // (the odd columns are zero)
        two_sum_acc2(hi1, lo1, make_float2(d1[0], d1[2]));
      }
      two_sum_acc2(hi0, lo0, hi1);
      lo0 = add2(lo0, lo1);
      // the planes (lanes t = 0 .. 3) together
      const float ps = plane_inv<BF>(lane & 3);
      ffs zr = ff_add(ffs{hi0.x * ps, lo0.x * ps}, ffs{0.f, 0.f}), yr = ff_add(ffs{hi0.y * ps, lo0.y * ps}, ffs{0.f, 0.f});
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        zr = ff_add(zr, ffs{__shfl_xor_sync(0xffffffffu, zr.hi, o), __shfl_xor_sync(0xffffffffu, zr.lo, o)});
        yr = ff_add(yr, ffs{__shfl_xor_sync(0xffffffffu, yr.hi, o), __shfl_xor_sync(0xffffffffu, yr.lo, o)});
      }
      // row g on lanes t = 0, 1, row g + 8 on lanes t = 2, 3, its first word on
      // the even lane, the second on the odd one
      const int row = (lane >> 2) + ((lane & 2) ? 8 : 0), word = lane & 1;
      const float zh = (lane & 2) ? yr.hi : zr.hi, zl = (lane & 2) ? yr.lo : zr.lo;
      if (!have_scale) {
        if (!__all_sync(0xffffffffu, wait_count(a.zcnt, gridDim.x, a.limit_ns, a.status))) {
          tmo = 1;
          break;
        }
        zs = fixed_scale(a.rowl1 * __longlong_as_double((long long)__ldcg(&a.zmax[0])));
        have_scale = true;
      }
      if (row < rows) {
        long long qh = 0, ql = 0;
        if (zs != INT_MIN) {
          const int sh = zs - be - (BF ? 8 : 0);   // eight bits for the count (FP8: X is times 2^-8)
          fixed_words(zh, sh, qh, ql);
          fixed_words(zl, sh, qh, ql);
        }
        atomicAdd(&a.zfix[2 * (r0 + row) + word], ((unsigned long long)(word ? ql : qh) << 8) + 1ull);
      }
    }
  } else if (warp < 1 + XM_SA + XM_NL) {
    // ------------------------------------------------ the link of the rows
    const int st = warp - 1 - XM_SA;
    const bool need_zp = a.link == LINK_LOGISTIC && NB > 1;
    const double* zprev = static_cast<const double*>(a.ps->zprev);
    double* zout = static_cast<double*>(a.ps->zout);
    const double mom = a.ps->mom;
    const int jl = lane & 15, hb = lane >> 4;
    double uh = 0.0, ul = 0.0;   // values of the words' units
    bool have_scale = false;
    double lsum[3] = {0.0, 0.0, 0.0};
    // two blocks at a time, one per half warp
    for (int k0 = 2 * st; k0 < kloc; k0 += 2 * XM_NL) {
      if (tmo) break;
      const int k = k0 + hb;
      const bool on = k < kloc;
      const int b = cr + (on ? k : k0) * a.Gr;
      const int64_t r0 = (int64_t)b * 16;
      const int rows = (int)((n - r0) < 16 ? (n - r0) : 16);
      const int64_t rowj = r0 + (jl < rows ? jl : rows - 1);
      const double yd = a.y[rowj];
      const double zp = need_zp ? zprev[rowj] : 0.0;
      const int ws = k % XM_RW;
      bool ok = !on || k < XM_RW || mbar_wait(&wempty[ws], ((k / XM_RW) - 1) & 1, a.limit_ns, a.status);
      // the row's words, complete once their low bits count every strip
      unsigned long long wh = 0ull, wl = 0ull;
      ok = ok && wait_row(&a.zfix[2 * rowj], (unsigned)a.Gc, wh, wl, a.limit_ns, a.status);
      if (!__all_sync(0xffffffffu, ok)) {
        tmo = 1;
        break;
      }
      if (!have_scale) {
        if (!__all_sync(0xffffffffu, wait_count(a.zcnt, gridDim.x, a.limit_ns, a.status))) {
          tmo = 1;
          break;
        }
        const int zs = fixed_scale(a.rowl1 * __longlong_as_double((long long)__ldcg(&a.zmax[0])));
        uh = zs == INT_MIN ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, 8 - zs);
        ul = ldexp(uh, -Z_LO);
        have_scale = true;
      }
      double z[1];
      z[0] = fma((double)((long long)wl >> 8), ul, (double)((long long)wh >> 8) * uh);
      double rv[NB];
      link_of<1, NB, true>(a.link, z, yd, zp, mom, rv);
      float w[NB];
      float mx = 0.f;
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        w[q] = jl < rows ? (float)rv[q] : 0.f;   // rows past the end carry weight 0
        mx = fmaxf(mx, fabsf(w[q]));
      }
      // the block's scale
      for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const int e = plane_scale(mx);
      const float sc = ldexpf(1.f, e);
      if (jl == 0 && on) wscale[ws] = ldexpf(1.f, (BF ? 0 : 8) - e);   // (FP8: X is times 2^-8)
      // four planes per weight: N columns 2 plane + q (one right-hand side: plane)
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        uint16_t u[4];
        planes16<BF>(w[q] * sc, u);
        if (on)
#pragma unroll
          for (int pl = 0; pl < 4; ++pl) wfrag[ws][NB == 2 ? 2 * pl + q : pl][jl] = u[pl];
      }
      if (NB == 1 && on)
#pragma unroll
        for (int q = 4; q < 8; ++q) wfrag[ws][q][jl] = 0;
      __syncwarp();
      if (jl == 0 && on) mbar_arrive(&wfull[ws]);
      if (on && cc == k % a.Gc && jl < rows) {   // this CTA records the block
        if (zout) zout[r0 + jl] = z[0];
        if (a.lsum) loss_of<1, true>(a.link, z, yd, zp, lsum);
      }
    }
    if (a.lsum) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double v = warp_sum(lsum[i]);
        if (lane == 0) lcomb[st][i] = v;
      }
    }
  } else {
    // ------------------------------------------------ phase B: X' r over the strip
    const int e = warp - 1 - XM_SA - XM_NL;
    constexpr int MS = (STEPS + XM_SB - 1) / XM_SB;   // this warp's steps: e, e + SB, ...
    float2 hi[MS][2 * MM], lo[MS][2 * MM];            // sums of (columns n, n + 1) at rows m = g, g + 8 per MMA
#pragma unroll
    for (int i = 0; i < MS; ++i)
#pragma unroll
      for (int q = 0; q < 2 * MM; ++q) { hi[i][q] = make_float2(0.f, 0.f); lo[i][q] = make_float2(0.f, 0.f); }
    // this lane's row of the four matrices (transposed): rows 0-7 of vectors
    // v0, v0 + 1, then rows 8-15
    const uint32_t rowoff = (uint32_t)((lane & 7) + ((lane >> 4) << 3)) * pitch;
    const int vsel = (lane >> 3) & 1;
    const int bn = lane >> 2, bt = lane & 3;
    const float2 pinv = NB == 2 ? make_float2(plane_inv<BF>(bt), plane_inv<BF>(bt))
                                : make_float2(plane_inv<BF>((2 * bt) & 3), plane_inv<BF>((2 * bt + 1) & 3));
    uint32_t off[MS];
#pragma unroll
    for (int i = 0; i < MS; ++i) off[i] = rowoff + (uint32_t)vsel * 16 + (e + XM_SB * i < STEPS ? toff[e + XM_SB * i] : 0u);
    for (int k = 0; k < kloc; ++k) {
      if (tmo) break;
      // (the block's tile is there: its own dot products are part of the agreed z)
      const int ws = k % XM_RW, sb = k % a.RA;
      const bool ok = mbar_wait(&full[sb], (k / a.RA) & 1, a.limit_ns, a.status) &&
                      mbar_wait(&wfull[ws], (k / XM_RW) & 1, a.limit_ns, a.status);
      if (!__all_sync(0xffffffffu, ok)) {
        tmo = 1;
        break;
      }
      const uint32_t* wf = reinterpret_cast<const uint32_t*>(&wfrag[ws][bn][0]);
      const uint32_t b0 = wf[bt], b1 = wf[bt + 4];
      // (two right-hand sides: this lane's columns are of plane bt; one: of planes 2 bt, 2 bt + 1)
      const float wsc = wscale[ws];
      const float2 sc = make_float2(wsc * pinv.x, wsc * pinv.y);
      const uint32_t base = smem_u32(smem + sb * stage);
      constexpr int GS = BF ? 4 : 2;   // steps in flight
#pragma unroll
      for (int i0 = 0; i0 < MS; i0 += GS) {
        if (e + XM_SB * i0 < xa.steps) {
          uint32_t r[GS][4];
#pragma unroll
          for (int u = 0; u < GS; ++u)
            if (i0 + u < MS) ldsm4t(r[u], base + off[i0 + u]);   // (steps past the last read the first again, unused)
#pragma unroll
          for (int u = 0; u < GS; ++u) {
            const int i = i0 + u;
            if (i < MS) {
              if constexpr (BF) {
                float d[4] = {0.f, 0.f, 0.f, 0.f};
                mma16816<BF>(d, r[u][0], r[u][1], r[u][2], r[u][3], b0, b1);
                two_sum_acc2(hi[i][0], lo[i][0], mul2(make_float2(d[0], d[1]), sc));
                two_sum_acc2(hi[i][1], lo[i][1], mul2(make_float2(d[2], d[3]), sc));
              } else {
                uint32_t ev[4], od[4];   // the even and the odd columns of the pairs
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  ev[q] = e4m3_ev(r[u][q]);
                  od[q] = e4m3_od(r[u][q]);
                }
                float d[4] = {0.f, 0.f, 0.f, 0.f}, f[4] = {0.f, 0.f, 0.f, 0.f};
                mma16816<BF>(d, ev[0], ev[1], ev[2], ev[3], b0, b1);
                mma16816<BF>(f, od[0], od[1], od[2], od[3], b0, b1);
                two_sum_acc2(hi[i][0], lo[i][0], mul2(make_float2(d[0], d[1]), sc));
                two_sum_acc2(hi[i][1], lo[i][1], mul2(make_float2(d[2], d[3]), sc));
                two_sum_acc2(hi[i][2 * MM - 2], lo[i][2 * MM - 2], mul2(make_float2(f[0], f[1]), sc));
                two_sum_acc2(hi[i][2 * MM - 1], lo[i][2 * MM - 1], mul2(make_float2(f[2], f[3]), sc));
              }
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&empty[sb]);
        mbar_arrive(&wempty[ws]);
      }
    }
    // the planes' columns together (lanes t = 0 .. 3), then g[cr][q][column]
    float2* g = static_cast<float2*>(a.g);
#pragma unroll
    for (int i = 0; i < MS; ++i) {
      const int s = e + XM_SB * i;
      if (s < xa.steps) {
        const int tc = tcol[s];
#pragma unroll
        for (int q = 0; q < 2 * MM; ++q) {
          ffs x = ff_add(ffs{hi[i][q].x, lo[i][q].x}, ffs{0.f, 0.f}), y = ff_add(ffs{hi[i][q].y, lo[i][q].y}, ffs{0.f, 0.f});
          const ffs x1{__shfl_down_sync(0xffffffffu, x.hi, 1), __shfl_down_sync(0xffffffffu, x.lo, 1)};
          const ffs y1{__shfl_down_sync(0xffffffffu, y.hi, 1), __shfl_down_sync(0xffffffffu, y.lo, 1)};
          x = ff_add(x, x1);   // lanes t = 0: planes 0, 1; t = 2: planes 2, 3 (one right-hand side: columns 0, 2 and 1, 3)
          y = ff_add(y, y1);
          const ffs x2{__shfl_down_sync(0xffffffffu, x.hi, 2), __shfl_down_sync(0xffffffffu, x.lo, 2)};
          const ffs y2{__shfl_down_sync(0xffffffffu, y.hi, 2), __shfl_down_sync(0xffffffffu, y.lo, 2)};
          const int v = q & 1;                                     // rows m = g: the first vector; g + 8: the second
          const int c = BF ? bn : 2 * bn + (q >> 1);
          const int64_t col = s0 + (tc & 0xffff) + v * VEC + c;
          if (bt == 0 && (v == 0 || !(tc >> 30)) && col < p) {
            ffs r0 = NB == 2 ? ff_add(x, x2) : ff_add(x, y), r1 = ff_add(y, y2);
            if (a.colscale) {   // FP8: times the column's scale, the product's error kept
              const float cs = a.colscale[col];
              float h = r0.hi * cs;
              r0 = ff_add(ffs{h, fmaf(r0.hi, cs, -h)}, ffs{r0.lo * cs, 0.f});
              h = r1.hi * cs;
              r1 = ff_add(ffs{h, fmaf(r1.hi, cs, -h)}, ffs{r1.lo * cs, 0.f});
            }
            g[((size_t)cr * NB) * p + col] = make_float2(r0.hi, r0.lo);
            if (NB == 2) g[((size_t)cr * NB + 1) * p + col] = make_float2(r1.hi, r1.lo);
          }
        }
      }
    }
  }
  __syncthreads();
  if (a.lsum && tid < 4) {
    double v = 0.0;
    if (tid < 3)
      for (int w = 0; w < XM_NL; ++w) v += lcomb[w][tid];
    a.lsum[4 * (size_t)blockIdx.x + tid] = v;
  }
}

}  // namespace relax
