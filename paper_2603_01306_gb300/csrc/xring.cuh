// Fused passes over FP32 or FP64 X with one product z: z = X beta, r = link(z),
// g = X' r, X read from HBM once.  FP64 X: FP64 throughout.  FP32 X, FF = false:
// the loop's pass, FP32 sums in compensated pairs.  FF = true: float-float arithmetic (the certificates, the
// power iteration, the last digits of FP32 solves).
//
// Strips x row groups, tiles kept in a ring from their dot products until
// their axpy, the rows' words of z with their own arrival counts, link warps of
// their own: as in xmma.cuh.  The twelve or so warps of sums:
//  * a dot warp holds the strip of beta and takes R rows of a block at a time;
//  * an axpy warp owns 32 vectors of the strip and takes all rows, the weights
//    read as ready operand pairs from shared memory.
// z in two words of fixed point (xmma.cuh), converted by shifts: FP64
// conversions of two lanes per row pair would take as long as the sums.  A
// block's words go out in one instruction: 40 iterations of 20000 x 50000 FP32
// took 33.4 ms with one word, 35.6 with two in two instructions, 33.3 so.
//
// FP32: bound by how much of X the rings hold (32 MB) against the round trip
// from HBM to the end of a block's agreement.  20000 x 50000: 852 us on
// xstrip.cuh's kernel, which sent X through L2 twice, 718 to 723 now (5.55 TB/s).
// Eight rows per dot warp: its butterfly takes 9 exchanges of pairs instead of 12
// for two times four (776 us; two rows 1204).  5 + 4 dot and link warps; 6 + 3
// 725, 5 + 3 722, 6 + 4 740, 7 + 2 740, and with four rows 4 + 5 776, 6 + 5 741,
// 4 + 9 788.  Blocks of 8 rows, of 16 where X stays in L2 (ROWS): 20000 x 50000
// 718 and 764, 4000 x 4000 logistic 28.9 and 25.0 (42.5 before), 1000 x 1000 14.3
// and 14.2 (24.5).  Prefetching the blocks after the ring into L2 lost: 920.
//
// FP64: latency in small designs (500 x 1000: 30.4 -> 16.4 us; a dependent FP64
// operation takes 64 cycles), the FP64 pipe in large ones (16 cycles per warp
// instruction and SM).  Blocks of 16 rows, since every block costs the link warps
// the same.
//
// FF: each product x b, b = bh + bl, is formed exactly as the FMA pair plus
// x bl and summed by TwoSum in packed pairs (dot_ff2: eleven instructions for
// two terms, about 48 significant bits).  The sums are what bounds it: 22 us of
// the FP32 pipes per product of 5000 x 10000 at two cycles each, against 30 us
// for X from HBM.  Hence six warps per product, three of the twelve on each
// scheduler.  96 certificates at 2000 x 5000: 45 us each on xstrip.cuh's kernel
// (six summing warps, two per scheduler at most), 27.0 here; 5000 x 10000, two
// right-hand sides: 171 and 96 us.  Four rows per dot warp (two: 2.68 ms for the
// 96, 45.9 for 256 nodes of 5000 x 10000; four 2.60, 45.0; eight 2.46, 45.9).  What is left is the depth of the ring (four
// blocks of 46 KB) and, in small problems, filling it.  Blocks of 8 rows: 3%
// slower.
#pragma once
#include "xmma.cuh"

namespace relax {

template <typename TX, bool FF, int ROWS> struct XF {
  static constexpr bool LOOP = !FF && sizeof(TX) == 4;
  static constexpr int SA = FF ? 6 : LOOP ? 5 : 4, SB = 6, NL = FF ? 3 : LOOP ? 4 : 5;   // dot, axpy and link warps
  static constexpr int B = ROWS;            // rows of a block
  static constexpr int R = LOOP ? 8 : 4;   // rows a dot warp takes at a time
  static constexpr int RW = 4 * NL;         // blocks of weights in shared memory
  static constexpr int WF = FF ? 8 : 2;     // words of 32 bits of a weight there
};
constexpr int XF_T = 512;
static_assert(1 + XF<float, true, 16>::SA + XF<float, true, 16>::SB + XF<float, true, 16>::NL == XF_T / 32 &&
              1 + XF<float, false, 8>::SA + XF<float, false, 8>::SB + XF<float, false, 8>::NL == XF_T / 32 &&
              1 + XF<double, false, 16>::SA + XF<double, false, 16>::SB + XF<double, false, 16>::NL == XF_T / 32);
constexpr int XF_TV = 6;                    // vectors of the strip per lane of a dot warp = axpy warps
constexpr int XF_MAXR = 16;                 // ring stages at most

template <typename TX, int NB, bool FF, int ROWS>
__global__ void __launch_bounds__(XF_T, 1) xring_kernel(const __grid_constant__ XSArgs a) {
  using K = XF<TX, FF, ROWS>;
  constexpr int XF_SA = K::SA, XF_SB = K::SB, XF_NL = K::NL, XF_B = K::B, XF_RW = K::RW, R = K::R;
  constexpr bool D = sizeof(TX) == 8;            // FP64 throughout
  constexpr int VEC = 16 / (int)sizeof(TX);
  static_assert(!(FF && D), "float-float: FP32 X");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[XF_MAXR], empty[XF_MAXR], wfull[XF_RW], wempty[XF_RW];
  __shared__ __align__(16) float wts[XF_RW][XF_B][NB][K::WF];   // w w (FP64: w), or wh wh -wh -wh wl wl
  __shared__ volatile int tmo;
  __shared__ int skip;
  __shared__ double lcomb[XF_NL][3];
  __shared__ __align__(16) float bsh[FF ? 2 : 1][D ? 4 : 32 * XF_TV * 4];   // the strip of beta, hi and lo
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    tmo = 0;
    skip = a.ps->done;
    for (int s = 0; s < a.RA; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], XF_SB); }
    for (int s = 0; s < XF_RW; ++s) { mbar_init(&wfull[s], 1); mbar_init(&wempty[s], XF_SB); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (skip) return;   // uniform (same flag everywhere)

  unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int cc = blockIdx.x % a.Gc, cr = blockIdx.x / a.Gc;
  const int64_t n = a.n, p = a.p;
  const int64_t s0 = (int64_t)cc * a.sw;
  const int nvs = (int)((min(s0 + a.sw, p) - s0 + VEC - 1) / VEC);   // vectors of the strip
  const uint32_t rowpitch = (uint32_t)a.inner * (uint32_t)sizeof(TX);
  const uint32_t tilebytes = (uint32_t)a.nbox * XF_B * rowpitch;   // whole boxes, out-of-range parts zero-filled
  const int kloc = (cr < a.nblk) ? (a.nblk - cr + a.Gr - 1) / a.Gr : 0;
  const size_t stage = (size_t)a.nbox * a.boxb;
  const int vpb = a.inner / VEC;
  // byte offset of a vector in row 0 of a tile (vectors past the strip read its
  // last one: their beta is zero and their sums are never written)
  auto voffset = [&](int v) {
    v = min(v, nvs - 1);
    return (uint32_t)((v / vpb) * a.boxb + (v % vpb) * 16);
  };

  if (warp == 0) {
    // ------------------------------------------------ producer: HBM -> ring
    if (lane == 0) {
      const uint64_t pol = a.keep ? policy_evict_normal() : policy_evict_first();
      int issued = 0;
      for (int k = 0; k < kloc; ++k) {
        const int s = k % a.RA;
        if (tmo) break;
        if (k >= a.RA && !mbar_wait(&empty[s], ((k / a.RA) - 1) & 1, a.limit_ns, a.status)) { tmo = 1; break; }
        const int y0 = (cr + k * a.Gr) * XF_B;
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
  } else if (warp < 1 + XF_SA) {
    // ------------------------------------------------ phase A: strip dot products
    const int st = warp - 1;
    // the strip of beta as pairs, split once for all dot warps
    unsigned long long mb = 0ull;
    for (int c = tid - 32; c < 32 * XF_TV * VEC; c += 32 * XF_SA) {
      const int64_t col = s0 + c;
      const double bd = c < (int)a.sw && col < p ? static_cast<const double*>(a.ps->beta)[col] : 0.0;
      unsigned long long bits = (unsigned long long)__double_as_longlong(bd) & ~(1ull << 63);
      if constexpr (!D) {
        const float h = (float)bd;
        bsh[0][c] = h;
        if constexpr (FF) bsh[1][c] = (float)(bd - (double)h);
        if (!(fabsf(h) < INFINITY) && bits < 0x7ff0000000000000ull) bits = 0x7ff0000000000000ull;   // beyond FP32
      }
      mb = bits > mb ? bits : mb;
    }
    // this CTA's max |beta_j| (NaN dominates: its bits compare above +Inf)
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ob = __shfl_xor_sync(0xffffffffu, mb, o);
      mb = ob > mb ? ob : mb;
    }
    if (lane == 0 && mb) atomicMax(&a.zmax[0], mb);
    if (lane == 0) __threadfence();
    named_sync(1, 32 * XF_SA);
    if (st == 0 && lane == 0) {
      __threadfence();
      atomicAdd(a.zcnt, 1u);
    }
    double bd[D ? XF_TV : 1][2];
    float2 bh[XF_TV][2], nb[FF ? XF_TV : 1][2], bl[FF ? XF_TV : 1][2];
    uint32_t voff[XF_TV];
#pragma unroll
    for (int t = 0; t < XF_TV; ++t) {
      const int v = lane + 32 * t;
      voff[t] = voffset(v);
      if constexpr (D) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int64_t col = s0 + (int64_t)v * 2 + c;
          bd[t][c] = v < nvs && col < p ? static_cast<const double*>(a.ps->beta)[col] : 0.0;
        }
        continue;
      }
      const float4 h = *reinterpret_cast<const float4*>(&bsh[0][D ? 0 : 4 * v]);
      bh[t][0] = make_float2(h.x, h.y);
      bh[t][1] = make_float2(h.z, h.w);
      if constexpr (FF) {
        const float4 l = *reinterpret_cast<const float4*>(&bsh[1][4 * v]);
        nb[t][0] = make_float2(-h.x, -h.y);
        nb[t][1] = make_float2(-h.z, -h.w);
        bl[t][0] = make_float2(l.x, l.y);
        bl[t][1] = make_float2(l.z, l.w);
      }
    }
    int zs = 0;
    double zf = 0.0;   // FP64: 2^(zs - 8)
    bool have_scale = false;
    constexpr int UB = XF_B / R;
    const int units = kloc * UB;
#pragma unroll 1
    for (int i = st; i < units; i += XF_SA) {
      if (tmo) break;
      const int k = i / UB, pr = i % UB;
      const int sa = k % a.RA;
      if (!__all_sync(0xffffffffu, mbar_wait(&full[sa], (k / a.RA) & 1, a.limit_ns, a.status))) {
        tmo = 1;
        break;
      }
      const int64_t r0 = (int64_t)(cr + k * a.Gr) * XF_B + R * pr;
      const unsigned char* row0 = smem + sa * stage + (size_t)(R * pr) * rowpitch;
      double zd[R];
      if constexpr (D) {
#pragma unroll
        for (int u = 0; u < R; ++u) zd[u] = 0.0;
#pragma unroll
        for (int t = 0; t < XF_TV; ++t) {
          if (32 * t < nvs) {   // uniform
#pragma unroll
            for (int u = 0; u < R; ++u) {
              const double2 x = *reinterpret_cast<const double2*>(row0 + u * rowpitch + voff[t]);
              zd[u] = fma(x.x, bd[t][0], zd[u]);
              zd[u] = fma(x.y, bd[t][1], zd[u]);
            }
          }
        }
        int o = 16;
#pragma unroll
        for (int half = R / 2; half >= 1; half >>= 1, o >>= 1) {
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int u = 0; u < half; ++u) {
            const double s = up ? zd[u] : zd[u + half];
            zd[u] = (up ? zd[u + half] : zd[u]) + __shfl_xor_sync(0xffffffffu, s, o);
          }
        }
#pragma unroll
        for (o = 16 / R; o > 0; o >>= 1) zd[0] += __shfl_xor_sync(0xffffffffu, zd[0], o);
      }
      float h[R], l[R];
      if constexpr (!D) {
      float2 hh[R], ll[FF ? R : 1];
#pragma unroll
      for (int u = 0; u < R; ++u) hh[u] = make_float2(0.f, 0.f);
      if constexpr (FF)
#pragma unroll
        for (int u = 0; u < R; ++u) ll[u] = make_float2(0.f, 0.f);
#pragma unroll
      for (int t = 0; t < XF_TV; ++t) {
        if (32 * t < nvs) {   // uniform
          float4 x[R];
#pragma unroll
          for (int u = 0; u < R; ++u) x[u] = *reinterpret_cast<const float4*>(row0 + u * rowpitch + voff[t]);
#pragma unroll
          for (int u = 0; u < R; ++u) {
            const float2 xa = make_float2(x[u].x, x[u].y), xb = make_float2(x[u].z, x[u].w);
            if constexpr (FF) {
              dot_ff2(hh[u], ll[u], xa, bh[t][0], nb[t][0], bl[t][0]);
              dot_ff2(hh[u], ll[u], xb, bh[t][1], nb[t][1], bl[t][1]);
            } else {
              hh[u] = fma2(xa, bh[t][0], hh[u]);
              hh[u] = fma2(xb, bh[t][1], hh[u]);
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < R; ++u) {
        h[u] = hh[u].x;
        l[u] = FF ? ll[FF ? u : 0].x + ll[FF ? u : 0].y : 0.f;
        two_sum_acc(h[u], l[u], hh[u].y);
      }
      // the lanes' sums, half of the rows to each half warp (and quarter), then
      // row lane / (32 / R) over its 32 / R lanes
      int o = 16;
#pragma unroll
      for (int half = R / 2; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int u = 0; u < half; ++u) {
          const float sh = up ? h[u] : h[u + half], sl = up ? l[u] : l[u + half];
          h[u] = up ? h[u + half] : h[u];
          l[u] = up ? l[u + half] : l[u];
          pair_add(h[u], l[u], __shfl_xor_sync(0xffffffffu, sh, o), __shfl_xor_sync(0xffffffffu, sl, o));
        }
      }
#pragma unroll
      for (o = 16 / R; o > 0; o >>= 1)
        pair_add(h[0], l[0], __shfl_xor_sync(0xffffffffu, h[0], o), __shfl_xor_sync(0xffffffffu, l[0], o));
      }
      if (!have_scale) {
        if (!__all_sync(0xffffffffu, wait_count(a.zcnt, gridDim.x, a.limit_ns, a.status))) {
          tmo = 1;
          break;
        }
        zs = fixed_scale(a.rowl1 * __longlong_as_double((long long)__ldcg(&a.zmax[0])));
        zf = zs == INT_MIN ? 0.0 : ldexp(1.0, zs - 8);
        have_scale = true;
      }
      // (a row's lanes hold the same sum: the first adds its first word, the
      // second its second one, the block's words in one instruction)
      const int64_t row = r0 + lane / (32 / R);
      const int word = lane % (32 / R);
      if (word < 2 && row < n) {
        long long qh = 0, ql = 0;
        if (zs != INT_MIN) {
          if constexpr (D) {
            const double v = zd[0] * zf, vi = rint(v);
            qh = (long long)vi;
            ql = __double2ll_rn((v - vi) * (double)(1ll << Z_LO));
          } else {
            fixed_words(h[0], zs - 8, qh, ql);
            fixed_words(l[0], zs - 8, qh, ql);
          }
        }
        atomicAdd(&a.zfix[2 * row + word], ((unsigned long long)(word ? ql : qh) << 8) + 1ull);
      }
    }
  } else if (warp < 1 + XF_SA + XF_SB) {
    // ------------------------------------------------ phase B: X' r over the strip
    const int e = warp - 1 - XF_SA;
    const int v = 32 * e + lane;
    const bool on = 32 * e < nvs;   // uniform
    const uint32_t voff = voffset(v);
    double ad[NB][2];
    float2 hi[NB][2], lo[NB][2];
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int u = 0; u < 2; ++u) { hi[q][u] = make_float2(0.f, 0.f); lo[q][u] = make_float2(0.f, 0.f); ad[q][u] = 0.0; }
    for (int k = 0; k < kloc; ++k) {
      if (tmo) break;
      const int ws = k % XF_RW, sb = k % a.RA;
      const bool ok = mbar_wait(&full[sb], (k / a.RA) & 1, a.limit_ns, a.status) &&
                      mbar_wait(&wfull[ws], (k / XF_RW) & 1, a.limit_ns, a.status);
      if (!__all_sync(0xffffffffu, ok)) {
        tmo = 1;
        break;
      }
      if (on) {
        const unsigned char* col = smem + sb * stage + voff;
        if constexpr (D) {
#pragma unroll
          for (int j = 0; j < XF_B; ++j) {
            const double2 x = *reinterpret_cast<const double2*>(col + (size_t)j * rowpitch);
#pragma unroll
            for (int q = 0; q < NB; ++q) {
              const double w = *reinterpret_cast<const double*>(&wts[ws][j][q][0]);
              ad[q][0] = fma(x.x, w, ad[q][0]);
              ad[q][1] = fma(x.y, w, ad[q][1]);
            }
          }
        } else if constexpr (FF) {
#pragma unroll 4
          for (int j = 0; j < XF_B; ++j) {
            const float4 x = *reinterpret_cast<const float4*>(col + (size_t)j * rowpitch);
#pragma unroll
            for (int q = 0; q < NB; ++q) {
              const float4 w = *reinterpret_cast<const float4*>(&wts[ws][j][q][0]);
              const float2 wl = *reinterpret_cast<const float2*>(&wts[ws][j][q][K::WF / 2]);
              dot_ff2(hi[q][0], lo[q][0], make_float2(x.x, x.y), make_float2(w.x, w.y), make_float2(w.z, w.w), wl);
              dot_ff2(hi[q][1], lo[q][1], make_float2(x.z, x.w), make_float2(w.x, w.y), make_float2(w.z, w.w), wl);
            }
          }
          // the low parts folded back, so that their own rounding stays small
#pragma unroll
          for (int q = 0; q < NB; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const float2 s = add2(hi[q][u], lo[q][u]);
              lo[q][u] = sub2(lo[q][u], sub2(s, hi[q][u]));
              hi[q][u] = s;
            }
        } else {
          // plain FP32 over the block's rows, the blocks' sums in pairs
          float2 acc[NB][2];
#pragma unroll
          for (int q = 0; q < NB; ++q) acc[q][0] = acc[q][1] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < XF_B; ++j) {
            const float4 x = *reinterpret_cast<const float4*>(col + (size_t)j * rowpitch);
#pragma unroll
            for (int q = 0; q < NB; ++q) {
              const float2 w = *reinterpret_cast<const float2*>(&wts[ws][j][q][0]);
              acc[q][0] = fma2(make_float2(x.x, x.y), w, acc[q][0]);
              acc[q][1] = fma2(make_float2(x.z, x.w), w, acc[q][1]);
            }
          }
#pragma unroll
          for (int q = 0; q < NB; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) two_sum_acc2(hi[q][u], lo[q][u], acc[q][u]);
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&empty[sb]);
        mbar_arrive(&wempty[ws]);
      }
    }
    // g[cr][q][column], FP32 data as normalised pairs
    if constexpr (D) {
      if (v < nvs)
#pragma unroll
        for (int q = 0; q < NB; ++q)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int64_t colj = s0 + (int64_t)v * 2 + c;
            if (colj < p) static_cast<double*>(a.g)[((size_t)cr * NB + q) * p + colj] = ad[q][c];
          }
    } else if (v < nvs)
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int64_t colj = s0 + (int64_t)v * 4 + c;
          const float2 h2 = hi[q][c >> 1], l2 = lo[q][c >> 1];
          const ffs s = ff_add((c & 1) ? ffs{h2.y, l2.y} : ffs{h2.x, l2.x}, ffs{0.f, 0.f});
          if (colj < p) static_cast<float2*>(a.g)[((size_t)cr * NB + q) * p + colj] = make_float2(s.hi, s.lo);
        }
  } else {
    // ------------------------------------------------ the link of the rows
    const int st = warp - 1 - XF_SA - XF_SB;
    const bool need_zp = a.link == LINK_CERT2_LS || a.link == LINK_CERT2_LOGI || (a.link == LINK_LOGISTIC && NB > 1);
    const double* zprev = static_cast<const double*>(a.ps->zprev);
    double* zout = static_cast<double*>(a.ps->zout);
    const double mom = a.ps->mom;
    double uh = 0.0, ul = 0.0;   // values of the words' units
    bool have_scale = false;
    double lsum[3] = {0.0, 0.0, 0.0};
    const int jl = lane % XF_B;
    for (int k = st; k < kloc; k += XF_NL) {
      if (tmo) break;
      const bool on = lane < XF_B;
      const int64_t r0 = (int64_t)(cr + k * a.Gr) * XF_B;
      const int rows = (int)((n - r0) < XF_B ? (n - r0) : XF_B);
      const int64_t rowj = r0 + (jl < rows ? jl : rows - 1);
      const double yd = a.y[rowj];
      const double zp = need_zp ? zprev[rowj] : 0.0;
      const int ws = k % XF_RW;
      unsigned long long wh = 0ull, wl = 0ull;
      bool ok = k < XF_RW || mbar_wait(&wempty[ws], ((k / XF_RW) - 1) & 1, a.limit_ns, a.status);
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
      link_of<1, NB, !FF && !D>(a.link, z, yd, zp, mom, rv);
      if (on) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          const double r = jl < rows ? rv[q] : 0.0;   // rows past the end carry weight 0
          const float h = (float)r;
          if constexpr (D) {
            *reinterpret_cast<double*>(&wts[ws][jl][q][0]) = r;
          } else if constexpr (FF) {
            const float l = (float)(r - (double)h);
            *reinterpret_cast<float4*>(&wts[ws][jl][q][0]) = make_float4(h, h, -h, -h);
            *reinterpret_cast<float2*>(&wts[ws][jl][q][K::WF / 2]) = make_float2(l, l);
          } else {
            *reinterpret_cast<float2*>(&wts[ws][jl][q][0]) = make_float2(h, h);
          }
        }
      }
      __syncwarp();
      if (jl == 0 && on) mbar_arrive(&wfull[ws]);
      if (on && cc == k % a.Gc && jl < rows) {   // this CTA records the block
        if (zout) zout[r0 + jl] = z[0];
        if (a.lsum) {
          if (a.loss64) loss_of<1, false>(a.link, z, yd, zp, lsum);
          else loss_of<1, !FF && !D>(a.link, z, yd, zp, lsum);
        }
      }
    }
    if (a.lsum) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double v = warp_sum(lsum[i]);
        if (lane == 0) lcomb[st][i] = v;
      }
    }
  }
  __syncthreads();
  if (a.lsum && tid < 4) {
    double v = 0.0;
    if (tid < 3)
      for (int w = 0; w < XF_NL; ++w) v += lcomb[w][tid];
    a.lsum[4 * (size_t)blockIdx.x + tid] = v;
  }
}

}  // namespace relax
