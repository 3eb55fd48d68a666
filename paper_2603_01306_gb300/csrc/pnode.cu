// The node p-phase (pnode.cuh): kernel, plan and launch.
#include <algorithm>
#include <cfloat>

#include "launch.cuh"

namespace relax {

namespace {

// What the stages share, at the start of the dynamic shared memory
struct PnSh {
  NArgs a;
  IterState st;
  // the problem: this CTA's coordinates are cb .. cb + cnt - 1
  const double* bcur;
  const double* bprev;
  const int8_t* fix;
  const void* part;
  const void* Gprev;
  void* Gcur;
  int64_t cb;
  int cnt, kb, pb, rank, prob, item, q0;
  // shared memory regions
  unsigned long long *xbuf, *red, *seg1, *seg3, *loc1, *loc3, *flat1, *flat3, *srt1, *srt3;
  float f3[PN_CAP];    // srt3 in FP32
  double* vw;          // v of the wide coordinates, by list place
  uint32_t* ka;        // FP32 key of |a_j| on Jf, else 0
  float* mv;           // |v_j| (FP32) on Jf, else 0
  uint16_t* wl;        // wide coordinates, a list per warp
  uint8_t* fl;         // bit 0 v < 0, 1 wide, 2 free, 3 fixed in
  int nw[PN_MAXW];     // wide coordinates per warp
  // brackets and decisions
  uint32_t lo1, hi1, lo3, hi3;
  unsigned c1lo, c1hi, cmlo, cmhi, ctlo, cthi;
  float z3lo, z3hi;
  int more1, more3, n1, n3, miss1, miss3, go, flags, done;
  unsigned bad, nnz, dom, nab, nzv, cnt0, cnt1;
  double loss[2], tot[XS_NSUM], red_[2], c, top, t1, g, w, mu, tau, mom, phi;
  float Tl, Th, ccd;
  uint8_t nsl[2][PN_TILES];
};

// dynamic shared memory: PnSh, exchange buffers, per-warp words, bracket
// lists, then 19 bytes per coordinate (whole warps' worth)
__host__ __device__ inline size_t pn_smem(int cl, int warps, int wch, int lc) {
  const size_t cp = (size_t)(warps - 1) * wch;
  return (sizeof(PnSh) + 15) / 16 * 16 + (size_t)2 * cl * XW_WORDS * 8 + (size_t)warps * XW_WORDS * 8 +
         (size_t)2 * cl * lc * 8 + (size_t)2 * lc * 8 + (size_t)4 * PN_CAP * 8 + cp * (8 + 4 + 4 + 2 + 1) + 16;
}

extern __shared__ __align__(16) unsigned char pn_raw[];
__device__ __forceinline__ PnSh& pn() { return *reinterpret_cast<PnSh*>(pn_raw); }

// a sum in the data's working precision: float-float, or FP64
template <bool S64> struct Acc;
template <> struct Acc<false> {
  ffs s;
  __device__ Acc() : s{0.f, 0.f} {}
  __device__ explicit Acc(unsigned long long w) { s = ffs{__uint_as_float((unsigned)w), __uint_as_float((unsigned)(w >> 32))}; }
  __device__ void add(double x) { ff_acc(s, x); }
  __device__ void add(float x) { ff_acc(s, x); }
  __device__ void merge(const Acc& o) { s = ff_add(s, o.s); }
  __device__ unsigned long long word() const { return ((unsigned long long)__float_as_uint(s.lo) << 32) | __float_as_uint(s.hi); }
  __device__ double val() const { return (double)s.hi + (double)s.lo; }
};
template <> struct Acc<true> {
  double s;
  __device__ Acc() : s(0.0) {}
  __device__ explicit Acc(unsigned long long w) { s = __longlong_as_double((long long)w); }
  __device__ void add(double x) { s += x; }
  __device__ void add(float x) { s += (double)x; }
  __device__ void merge(const Acc& o) { s += o.s; }
  __device__ unsigned long long word() const { return (unsigned long long)__double_as_longlong(s); }
  __device__ double val() const { return s; }
};
template <bool S64>
__device__ __forceinline__ void warp_merge(Acc<S64>& a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a.merge(Acc<S64>(__shfl_xor_sync(0xffffffffu, a.word(), o)));
}
__device__ __forceinline__ unsigned long long pack2(unsigned lo, unsigned hi) { return ((unsigned long long)hi << 32) | lo; }
__device__ __forceinline__ void st_cluster_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Candidates of a warm round: the predicted key kc, and around it kc -+ 2^(e-i),
// geometrically finer towards it, so that the bracket is about as wide as the
// prediction is off; clamped into (lo, hi).  e follows the last deviation.
__device__ __forceinline__ uint32_t pn_warm(uint32_t kc, int e, uint32_t lo, uint32_t hi, int q) {
  const int i = q < 15 ? q : 31 - q;   // 15 steps below, 15 above, one far above
  const int sh = max(0, q == 31 ? e + 2 : q < 15 ? e - i : e + 1 - i);
  const long long off = q == 15 ? 0ll : q < 15 ? -(1ll << sh) : (1ll << sh);
  long long x = (long long)kc + off;
  if (x <= (long long)lo) x = (long long)lo + 1;
  if (x >= (long long)hi) x = (long long)hi - 1;
  return (uint32_t)x;
}

constexpr uint32_t kInfKey = KeyOf<float>::kInf;

// ---------------------------------------------------------------- exchanges
// (nx counts them; the buffers alternate)
__device__ __forceinline__ unsigned long long* pn_slot(int nx, int r, int w) {
  PnSh& s = pn();
  return s.xbuf + ((nx & 1) * s.a.cl + r) * XW_WORDS + w;
}
__device__ __forceinline__ uint32_t pn_remote(uint32_t loc, int r) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(loc), "r"(r));
  return ra;
}
__device__ __forceinline__ unsigned long long xcnt(int nx, int w) {
  const int S = pn().a.cl;
  const unsigned long long* src = pn_slot(nx, 0, w);
  unsigned long long v = 0;
#pragma unroll 4
  for (int r = 0; r < S; ++r) v += src[r * XW_WORDS];
  return v;
}
template <typename A>
__device__ __forceinline__ A xacc(int nx, int w) {   // over the CTAs in rank order
  const int S = pn().a.cl;
  const unsigned long long* src = pn_slot(nx, 0, w);
  A v(src[0]);
#pragma unroll 4
  for (int r = 1; r < S; ++r) v.merge(A(src[r * XW_WORDS]));
  return v;
}
// Every warp's words of `red` are in place: sum them over the warps, push the
// sums into every CTA's shared memory, and wait until every CTA has pushed.
// Words below na0 are float-float, below na1 A sums, the others counts.
template <int K>
__device__ __noinline__ void pn_exchange(int nx, int na0, int na1, int words) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  __syncthreads();
  const int W = blockDim.x >> 5, S = s.a.cl;
  const int t = threadIdx.x;
  if (t < words) {   // words <= 105 < blockDim.x
    const unsigned long long* src = s.red + t;
    unsigned long long w = src[0];
    if (t < na0) {
      Acc<false> v(w);
#pragma unroll 8
      for (int i = 1; i < W; ++i) v.merge(Acc<false>(src[i * XW_WORDS]));
      w = v.word();
    } else if (t < na1) {
      A v(w);
#pragma unroll 4
      for (int i = 1; i < W; ++i) v.merge(A(src[i * XW_WORDS]));
      w = v.word();
    } else {
#pragma unroll 8
      for (int i = 1; i < W; ++i) w += src[i * XW_WORDS];
    }
    const uint32_t loc = smem_u32(pn_slot(nx, s.rank, t));
#pragma unroll 4
    for (int r = 0; r < S; ++r) st_cluster_u64(pn_remote(loc, r), w);
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
}
// A small cluster-wide sum of two A sums and two counts per lane -> red_,
// cnt0, cnt1; returns the next exchange's number
template <int K>
__device__ __noinline__ int pn_small_sum(int nx, unsigned long long w0, unsigned long long w1, unsigned c0, unsigned c1) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  A v0(w0), v1(w1);
  warp_merge<(K != PK_PAIR)>(v0);
  warp_merge<(K != PK_PAIR)>(v1);
  c0 = __reduce_add_sync(0xffffffffu, c0);
  c1 = __reduce_add_sync(0xffffffffu, c1);
  if (lane == 0) {
    unsigned long long* rw = s.red + warp * XW_WORDS;
    rw[0] = v0.word();
    rw[1] = v1.word();
    rw[2] = pack2(c0, c1);
  }
  pn_exchange<K>(nx, 0, 2, 3);
  if (warp == 0) {
    if (lane < 2) s.red_[lane] = xacc<A>(nx, lane).val();
    else if (lane == 2) {
      const unsigned long long c = xcnt(nx, 2);
      s.cnt0 = (unsigned)c;
      s.cnt1 = (unsigned)(c >> 32);
    }
  }
  __syncthreads();
  return nx + 1;
}

// ------------------------------------------------------------- the gradient
// right-hand side q of coordinate j from the products' output, as a pair; all
// of a coordinate's loads go out before the first is used
__device__ __forceinline__ ffs pn_gpair(int64_t j, int q) {
  const PnSh& s = pn();
  const NArgs& a = s.a;
  if (a.tiles) {
    const float* src = a.tiles + (size_t)(q * a.m + s.prob) * a.p + j;
    const int ns = s.nsl[q][(int)(j / BG_BM) - (int)(s.cb / BG_BM)];
    const size_t chunk = (size_t)a.NB * a.m * a.p;
    ffs v{0.f, 0.f};
#pragma unroll 1
    for (int c = 0; c < ns; c += 4) {
      float y[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) y[i] = c + i < ns ? __ldcg(src + (c + i) * chunk) : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) ff_acc(v, y[i]);
    }
    return ff_add(v, ffs{0.f, 0.f});
  }
  const float2* src = static_cast<const float2*>(s.part) + (size_t)q * a.p + j;
  const size_t stride = (size_t)a.NB * a.p;
  ffs v{0.f, 0.f}, u{0.f, 0.f};
#pragma unroll 1
  for (int c = 0; c < a.ncl; c += 8) {   // two chains
    float2 y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = c + i < a.ncl ? __ldcg(src + (size_t)(c + i) * stride) : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      v = ff_add(v, ffs{y[i].x, y[i].y});
      u = ff_add(u, ffs{y[i + 1].x, y[i + 1].y});
    }
  }
  return ff_add(v, u);
}
// the same in FP64 (sums of pairs too, but in the loop on FP32 data).  Inlined:
// lanes call it on their own, and as a function of its own with an unrolled
// loop it came out wrong (by whole partials) for lanes that a branch had split
// from their warp.
template <int K>
__device__ __forceinline__ double pn_gdbl(int64_t j, int q) {
  const PnSh& s = pn();
  if (K == PK_PAIR) {
    const ffs v = pn_gpair(j, q);
    return (double)v.hi + (double)v.lo;
  }
  const size_t stride = (size_t)s.a.NB * s.a.p;
  double v = 0.0;
  if (K == PK_PAIR64 || s.a.gpair) {
    const float2* src = static_cast<const float2*>(s.part) + (size_t)q * s.a.p + j;
#pragma unroll 4
    for (int c = 0; c < s.a.ncl; ++c) {
      const float2 y = __ldcg(src + c * stride);
      v += (double)y.x + (double)y.y;
    }
    return v;
  }
  const double* src = static_cast<const double*>(s.part) + (size_t)q * s.a.p + j;
#pragma unroll 4
  for (int c = 0; c < s.a.ncl; ++c) v += __ldcg(src + c * stride);
  return v;
}
// FP64 G^t_j, as stage 1 stored it
template <int K>
__device__ __forceinline__ double pn_G64(int64_t j) {
  if (K == PK_F64) return static_cast<const double*>(pn().Gcur)[j];
  const float2 v = static_cast<const float2*>(pn().Gcur)[j];
  return (double)v.x + (double)v.y;
}
template <int K>
__device__ __forceinline__ double pn_vin(int64_t j) {   // the standalone operations' input
  const void* v = pn().a.vin;
  return K == PK_F64 ? static_cast<const double*>(v)[j] : (double)static_cast<const float*>(v)[j];
}
template <int K>
__device__ __forceinline__ double pn_a64(int64_t j) {
  if (K != PK_PAIR && pn().a.mode == PM_GSTAR) return fabs(pn_vin<K>(j));
  if (K == PK_PAIR64) return fabs(pn_gdbl<K>(j, 0)) * pn().a.kc.inv2l;   // (the stored pair only ranks the coordinates)
  return fabs(pn_G64<K>(j)) * pn().a.kc.inv2l;
}

// v_j of a wide coordinate, FP64 (on FP32 data the gradient at y, whose terms
// are FP32 pairs, in float-float)
template <int K>
__device__ __forceinline__ double pn_v_wide(int64_t j, double b, double mu) {
  const PnSh& s = pn();
  const double bp = s.bprev[j];
  double gy;
  if (is_zero_bits(mu)) {
    gy = pn_G64<K>(j);
  } else if (s.a.loss == 0) {
    if (K == PK_F64) {
      gy = (1.0 + mu) * pn_G64<K>(j) - mu * static_cast<const double*>(s.Gprev)[j];
    } else {
      const float2 g = static_cast<const float2*>(s.Gcur)[j], gp = static_cast<const float2*>(s.Gprev)[j];
      // G + mu (G - Gprev)
      const ffs d = ff_add(ffs{g.x, g.y}, ffs{-gp.x, -gp.y});
      const float mh = s.st.mu32, ml = s.st.mu_lo, h = mh * d.hi;
      const ffs m{h, fmaf(mh, d.hi, -h) + fmaf(mh, d.lo, ml * d.hi)};
      const ffs r = ff_add(ffs{g.x, g.y}, m);
      gy = (double)r.hi + (double)r.lo;
    }
  } else {
    gy = pn_gdbl<K>(j, 1);
  }
  return (b + mu * (b - bp)) - s.a.step * gy;
}

// T^{-1}(m): where a coordinate of magnitude m reaches z = 1, in FP32
__device__ __forceinline__ float pn_tinv(float m, const PConst& kc) { return m <= kc.M1r_f ? m * kc.rr_f : m - kc.M; }

// ------------------------------------------------------------------ rounds
// One round of candidates: this warp's counts for S1 (do1) and counts and sums
// for S3 (do3), into its words of `red`
__device__ __noinline__ void pn_count(bool do1, bool do3, uint32_t x1, uint32_t x3) {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const PConst& kc = s.a.kc;
  unsigned n1 = 0, n3 = 0, nt = 0, above1 = 0, above3 = 0;
  ffs s3{0.f, 0.f}, sa{0.f, 0.f};
  const uint32_t x1min = __shfl_sync(0xffffffffu, x1, 0), x1max = __shfl_sync(0xffffffffu, x1, 31);
  const float cq = __uint_as_float(x3);
  const float cmin = __shfl_sync(0xffffffffu, cq, 0), cmax = __shfl_sync(0xffffffffu, cq, 31);
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0;
#pragma unroll 1
  for (int i0 = w0; i0 < w1; i0 += 32) {
    const int i = i0 + lane;
    if (do1) {
      const uint32_t key = i < w1 ? s.ka[i] : 0u;
      above1 += key >= x1max ? 1u : 0u;
      unsigned act = __ballot_sync(0xffffffffu, key >= x1min && key < x1max);
#pragma unroll 1
      while (act) {
        const int src = __ffs(act) - 1;
        act &= act - 1u;
        n1 += __shfl_sync(0xffffffffu, key, src) >= x1 ? 1u : 0u;
      }
    }
    if (do3) {
      const float m = i < w1 ? s.mv[i] : 0.f;
      const float ti = pn_tinv(m, kc);
      const bool abv = m > cmax && !(ti > cmin);
      above3 += abv ? 1u : 0u;
      ff_acc(sa, abv ? m : 0.f);
      unsigned act = __ballot_sync(0xffffffffu, m > cmin && !abv);
#pragma unroll 1
      while (act) {
        const int src = __ffs(act) - 1;
        act &= act - 1u;
        const float mm = __shfl_sync(0xffffffffu, m, src);
        const float tt = __shfl_sync(0xffffffffu, ti, src);
        const bool top = tt > cq, mid = mm > cq && !top;
        nt += top ? 1u : 0u;
        n3 += mid ? 1u : 0u;
        ff_acc(s3, mid ? mm : 0.f);
      }
    }
  }
  n1 += __reduce_add_sync(0xffffffffu, above1);
  above3 = __reduce_add_sync(0xffffffffu, above3);
  Acc<false> s3a;
  s3a.s = s3;
  if (above3) {
    Acc<false> v;
    v.s = sa;
    warp_merge<false>(v);
    s3a.merge(v);
  }
  unsigned long long* rw = s.red + warp * XW_WORDS;
  rw[XW_S3 + lane] = s3a.word();
  rw[XW_N3 + lane] = pack2(n3 + above3, nt);
  rw[XW_N1 + lane] = n1;
}
// the round's decisions from the exchanged words: warp 0 S3's, warp 1 S1's
__device__ __noinline__ void pn_decide(int nx, bool do1, bool do3, uint32_t x1, uint32_t x3) {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cap = min(PN_CAP / 2, s.a.lc);
  int qlo, qhi;
  if (warp == 0 && do3) {
    const ffs S3 = xacc<Acc<false>>(nx, XW_S3 + lane).s;
    const unsigned long long nn = xcnt(nx, XW_N3 + lane);
    const unsigned n = (unsigned)nn, ntop = (unsigned)(nn >> 32);
    // sum z >= kbar at c: (S - c n) - (kbar - ntop) w >= 0, w = min(c / rho, M), in float-float
    const PConst& kc = s.a.kc;
    const float c = __uint_as_float(x3), nf = (float)n, kr = (float)(s.kb - (int)ntop);
    const float h1 = c * nf, l1 = fmaf(c, nf, -h1);
    ffs w{kc.M, kc.M_lo};
    if (x3 < kc.krho) {
      w.hi = c * kc.inv_rho_f;
      w.lo = fmaf(c, kc.inv_rho_f, -w.hi) + c * kc.inv_rho_lo;
    }
    const float h2 = kr * w.hi, l2 = fmaf(kr, w.hi, -h2) + kr * w.lo;
    ffs z = ff_add(ff_add(S3, ffs{-h1, -l1}), ffs{-h2, -l2});
    if (!(fabsf(w.hi) < 3e38f)) z = ffs{-1.f, 0.f};   // no box: c beyond every magnitude
    uint32_t lo = s.lo3, hi = s.hi3;
    bracket_step<uint32_t>(x3, z.hi >= 0.f, lo, hi, qlo, qhi);
    const float zw = z.hi / w.hi;   // Z - kbar: the secant's ends
    const unsigned cm = n + ntop;
    const int sl = qlo >= 0 ? qlo : 0, shh = qhi < 32 ? qhi : 0;
    const float zlo = __shfl_sync(0xffffffffu, zw, sl), zhi = __shfl_sync(0xffffffffu, zw, shh);
    const unsigned a0 = __shfl_sync(0xffffffffu, cm, sl), b0 = __shfl_sync(0xffffffffu, ntop, sl);
    const unsigned a1 = __shfl_sync(0xffffffffu, cm, shh), b1 = __shfl_sync(0xffffffffu, ntop, shh);
    if (lane == 0) {
      if (qlo >= 0) { s.cmlo = a0; s.ctlo = b0; s.z3lo = zlo; }
      if (qhi < 32) { s.cmhi = a1; s.cthi = b1; s.z3hi = zhi; }
      s.lo3 = lo;
      s.hi3 = hi;
      s.more3 = (int)((s.cmlo - s.cmhi) + (s.ctlo - s.cthi)) > cap && hi - lo > 1;
    }
  }
  if (warp == 1 && do1) {
    const unsigned n = (unsigned)xcnt(nx, XW_N1 + lane);
    uint32_t lo = s.lo1, hi = s.hi1;
    bracket_step<uint32_t>(x1, n >= (unsigned)s.kb, lo, hi, qlo, qhi);
    const unsigned c0 = __shfl_sync(0xffffffffu, n, qlo >= 0 ? qlo : 0), c1 = __shfl_sync(0xffffffffu, n, qhi < 32 ? qhi : 0);
    if (lane == 0) {
      if (qlo >= 0) s.c1lo = c0;
      if (qhi < 32) s.c1hi = c1;
      s.lo1 = lo;
      s.hi1 = hi;
      s.more1 = (int)(s.c1lo - s.c1hi) > cap && hi - lo > 1;
    }
  }
}
// further rounds while a bracket holds too many entries (no prediction yet, or
// one that was far off)
template <int K>
__device__ __noinline__ int pn_more_rounds(int nx) {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31;
  while (s.more1 || s.more3) {
    const bool d1 = s.more1 != 0, d3 = s.more3 != 0;
    const uint32_t x1 = d1 ? cand<uint32_t>(s.lo1, s.hi1, lane) : 0u;
    const uint32_t x3 = d3 ? cand<uint32_t>(s.lo3, s.hi3, lane) : 0u;
    pn_count(d1, d3, x1, x3);
    if (lane < XS_NSUM) s.red[(threadIdx.x >> 5) * XW_WORDS + XW_SUM + lane] = Acc<(K != PK_PAIR)>().word();
    pn_exchange<K>(nx, XW_SUM, XW_SUM + XS_NSUM, XW_INT);
    pn_decide(nx, d1, d3, x1, x3);
    __syncthreads();
    ++nx;
  }
  return nx;
}

// --------------------------------------------------------- finishing of S3
// One classification step of S3 at cc (counts of the coordinates at z = 1 and
// in between, the sum of the latter): the closed form on the piece, the
// bracket [cl, ch] tightened by the sign at cc; true when it stands
struct C3 {
  double cc, cl, ch;
  int n;
};
// A root at the end of a flat stretch of the sum is moved onto it: all `nm`
// coordinates in between at z = 1 (kr of them wanted), or all at z = 0.  Any
// point of the stretch is a root; on it n_top and n_nz count as Algorithm 2's block does.
__device__ __forceinline__ double pn_flat(double c, double kr, double nm, double sm) {
  if (nm == 0.0) return c;
  if (kr == nm) return c - fmin(0x1p-50 * (sm / nm), 0x1p-10 * c);
  return kr == 0.0 ? c * (1.0 + 0x1p-50) : c;
}
__device__ __noinline__ bool pn_step3(C3& z, double Nt, double Nm, double Sm) {
  const PnSh& s = pn();
  const double rho = s.a.rho, rhoM = s.a.kc.rhoM, M = s.a.M;
  const double kr = (double)s.kb - Nt;
  const bool low = z.cc <= rhoM;
  const double f = low ? rho * (Sm - z.cc * Nm) - kr * z.cc : (Sm - z.cc * Nm) - kr * M;
  if (f >= 0.0) z.cl = fmax(z.cl, z.cc);
  else z.ch = fmin(z.ch, z.cc);
  const double num = low ? rho * Sm : Sm - M * kr, den = low ? kr + rho * Nm : Nm;
  // a flat piece (no coordinate in between): any c on it is a root when
  // Ntop == kbar, none when not
  const bool none = Nm == 0.0 && kr != 0.0;
  double cn = none ? -1.0 : Nm == 0.0 ? z.cc : num / den;
  // a root that reproduces the point it was formed at lies on its piece
  if (fabs(cn - z.cc) <= 0x1p-50 * z.cc) {
    z.cc = pn_flat(cn, kr, Nm, Sm);
    return true;
  }
  // else on to it, where it narrows the bracket (the sum bends both ways, and the
  // roots of two pieces can name each other: the end of the bracket is no
  // progress, and every fourth step bisects)
  if (!(cn > z.cl && cn < z.ch) || (z.n & 3) == 3) {
    cn = z.cl > 0.0 ? sqrt(z.cl) * sqrt(z.ch) : z.ch * 0x1p-20;
    if (!(cn > z.cl && cn < z.ch)) return true;   // the bracket is one value
  }
  ++z.n;
  z.cc = cn;
  return false;
}
__device__ __forceinline__ double pn_T(double c) {
  const NArgs& a = pn().a;
  return c <= a.kc.rhoM ? c * a.kc.kTc : c + a.M;
}
// S3 on the sorted list of the bracket's entries (warp 1).  The classification
// is searched in FP32 arithmetic (sums float-float), then the closed form
// taken once in FP64 and the classification checked against the exact values;
// where it does not stand the search goes on in FP64.
template <int K>
__device__ __noinline__ void pn_finish3(int nx, int n3) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31;
  const PConst& kc = s.a.kc;
  const unsigned long long nn = xcnt(nx, 3);
  const unsigned nt0 = (unsigned)nn, nm0 = (unsigned)(nn >> 32);
  const A sm0 = xacc<A>(nx, 1);
  const uint32_t lok = s.lo3 > 2 ? s.lo3 - 2 : 0u, hik = min(s.hi3 + 2, kInfKey - 1);
  const float lo = __uint_as_float(s.lo3), hi = __uint_as_float(min(s.hi3, kInfKey - 1));
  const float d = s.z3lo - s.z3hi;
  float c = d > 0.f && s.z3lo >= 0.f && s.z3hi < 0.f && lo > 0.f ? lo + (hi - lo) * __fdividef(s.z3lo, d) : hi;
  if (!(c > 0.f && c <= hi)) c = hi;
  // nothing beyond the bracket: c lies below the list's largest entry
  if (nt0 + nm0 == 0 && n3 > 0) c = fminf(c, s.f3[0] * 0.9999f);
  const double smd = sm0.val();
  const ffs sm0f = K != PK_PAIR ? ff_of(smd) : ffs{__uint_as_float((unsigned)sm0.word()), __uint_as_float((unsigned)(sm0.word() >> 32))};
  unsigned pt = ~0u, pm = ~0u, nt = 0, nm = 0;
  bool settled = false;
  ffs Sm = sm0f;
#pragma unroll 1
  for (int it = 0; it < 32; ++it) {
    const bool low = key_of(c) < kc.krho;
    const float T = low ? c * kc.kTc_f : c + kc.M;
    nt = nm = 0;
    Acc<false> v;
#pragma unroll 2
    for (int i = lane; i < n3; i += 32) {
      const float x = s.f3[i];
      const bool top = x >= T, mid = x > c && !top;
      nt += top;
      nm += mid;
      v.add(mid ? x : 0.f);
    }
    nt = nt0 + __reduce_add_sync(0xffffffffu, nt);
    nm = nm0 + __reduce_add_sync(0xffffffffu, nm);
    if (nt == pt && nm == pm && (nm > 0 || nt == (unsigned)s.kb)) {   // (c is the one that these counts belong to)
      settled = true;
      break;
    }
    pt = nt;
    pm = nm;
    warp_merge<false>(v);
    Sm = ff_add(sm0f, v.s);
    const float kr = (float)(s.kb - (int)nt), nmf = (float)nm;
    float cn;
    if (nm == 0) cn = nt == (unsigned)s.kb ? c : 0.5f * (c + (nt < (unsigned)s.kb ? lo : hi));
    else if (low) cn = __fdividef(kc.rho_f * Sm.hi, kr + kc.rho_f * nmf);
    else {
      const float h = kr * kc.M, l = fmaf(kr, kc.M, -h) + kr * kc.M_lo;
      cn = __fdividef(ff_add(Sm, ffs{-h, -l}).hi, nmf);
    }
    c = fminf(fmaxf(cn, __uint_as_float(lok)), __uint_as_float(hik));
    if (!(c > 0.f)) c = hi;
  }
  // the classification's exact sum on the list and its closed form in FP64;
  // it stands when the exact values classify the same at that c
  C3 z;
  z.cc = (double)c;
  bool done = false;
  if (settled && nm > 0) {
    A v;
    const float T = key_of(c) < kc.krho ? c * kc.kTc_f : c + kc.M;
#pragma unroll 1
    for (int i = lane; i < n3; i += 32) {
      const float x = s.f3[i];
      if (x > c && !(x >= T)) v.add(__longlong_as_double((long long)s.srt3[i]));
    }
    if (nm > nm0) warp_merge<(K != PK_PAIR)>(v);
    const bool low = key_of(c) < kc.krho;
    const double Se = smd + v.val(), kr = (double)(s.kb - (int)nt), n = (double)nm;
    const double cn = (low ? s.a.rho * Se : Se - s.a.M * kr) / (low ? kr + s.a.rho * n : n);
    const double Tn = low ? cn * kc.kTc : cn + s.a.M;
    const unsigned long long ck = (unsigned long long)__double_as_longlong(cn), tk = (unsigned long long)__double_as_longlong(Tn);
    unsigned mt = 0, mm = 0;
#pragma unroll 2
    for (int i = lane; i < n3; i += 32) {
      const unsigned long long x = s.srt3[i];
      mt += x >= tk;
      mm += x > ck && x < tk;
    }
    mt = nt0 + __reduce_add_sync(0xffffffffu, mt);
    mm = nm0 + __reduce_add_sync(0xffffffffu, mm);
    const float cf = (float)cn;
    // (positive and finite; on the side of rho M that the form assumed)
    done = mt == nt && mm == nm && cf > 0.f && cf < 3e38f && (low ? key_of(cf) < kc.krho : key_of(cf) > kc.krho);
    z.cc = pn_flat(cn, kr, n, Se);
  }
  if (!done) {   // search on in FP64
    z.cl = (double)__uint_as_float(lok);
    z.ch = (double)__uint_as_float(hik);
    z.n = 0;
    z.cc = (double)c;
  }
#pragma unroll 1
  for (int it = 0; it < 100 && !done; ++it) {
    const unsigned long long ck = (unsigned long long)__double_as_longlong(z.cc);
    const unsigned long long tk = (unsigned long long)__double_as_longlong(pn_T(z.cc));
    unsigned mt = 0, mm = 0;
    A v;
#pragma unroll 1
    for (int i = lane; i < n3; i += 32) {
      const unsigned long long x = s.srt3[i];
      if (x >= tk) ++mt;
      else if (x > ck) {
        ++mm;
        v.add(__longlong_as_double((long long)x));
      }
    }
    mt = __reduce_add_sync(0xffffffffu, mt);
    mm = __reduce_add_sync(0xffffffffu, mm);
    warp_merge<(K != PK_PAIR)>(v);
    done = pn_step3(z, (double)(nt0 + mt), (double)(nm0 + mm), smd + v.val());
  }
  if (lane == 0) {
    s.c = z.cc;
    s.ccd = __double2float_rd(z.cc);
    // no root, or one at the bracket's very end (up to where a bisection towards
    // that end stops): the bracket missed it
    s.miss3 = !(done && z.cc > (double)__uint_as_float(lok) * (1.0 + 0x1p-40) &&
                z.cc < (double)__uint_as_float(hik) * (1.0 - 0x1p-40));
  }
}
// S3 by cluster-wide classifications (ties that no bracket separates)
template <int K>
__device__ __noinline__ int pn_fallback3(int nx) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0, nw = s.nw[warp];
  C3 z;
  z.cl = 0.0;
  z.ch = K == PK_F64 ? DBL_MAX : (double)FLT_MAX;
  z.cc = (double)__uint_as_float(min(s.hi3, kInfKey - 1));
  z.n = 0;
#pragma unroll 1
  for (int it = 0; it < 200; ++it) {
    const double T = pn_T(z.cc);
    A v;
    unsigned nt = 0, nm = 0;
#pragma unroll 1
    for (int u = lane; u < (w1 - w0) + nw; u += 32) {
      const int i = u < w1 - w0 ? w0 + u : s.wl[w0 + u - (w1 - w0)];
      const uint8_t f8 = s.fl[i];
      if (u < w1 - w0 ? (f8 & 6) != 4 : !(f8 & 4)) continue;
      const double m = u < w1 - w0 ? (double)s.mv[i] : fabs(s.vw[w0 + u - (w1 - w0)]);
      if (m >= T) ++nt;
      else if (m > z.cc) {
        ++nm;
        v.add(m);
      }
    }
    nx = pn_small_sum<K>(nx, v.word(), A().word(), nt, nm);
    const bool done = pn_step3(z, (double)s.cnt0, (double)s.cnt1, s.red_[0]);   // the same on every thread
    __syncthreads();
    if (done) break;
  }
  if (threadIdx.x == 0) {
    s.c = z.cc;
    s.ccd = __double2float_rd(z.cc);
  }
  __syncthreads();
  return nx;
}

// --------------------------------------------------------- finishing of S1
// TopSum through its variational form at t* = the kbar-th largest |a_j|:
// kbar H(t*) + sum (H(|a_j|) - H(t*))_+.  On FP32 data, where FP32 cannot
// tell the kbar-th and the next |a_j| apart, t* is their common FP32 value: an
// upper bound of TopSum, so that Psi stays a lower bound.  (warp 0)
template <int K>
__device__ __noinline__ void pn_finish1(int nx, int n1) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31;
  const double sumH = xacc<A>(nx, 0).val();
  const int r = s.kb - (int)xcnt(nx, 2);
  double ts = r >= 1 && r <= n1 ? __longlong_as_double((long long)s.srt1[r - 1]) : 0.0;
  if (K != PK_F64 && r >= 1 && r < n1 && (float)__longlong_as_double((long long)s.srt1[r]) == (float)ts) ts = (double)(float)ts;
  const double ht = huber_d<double>(ts, s.a.M);
  A v;
#pragma unroll 1
  for (int i = lane; i < n1; i += 32) {
    const double hv = huber_d<double>(__longlong_as_double((long long)s.srt1[i]), s.a.M) - ht;
    if (hv > 0.0) v.add(hv);
  }
  warp_merge<(K != PK_PAIR)>(v);
  if (lane == 0) {
    s.top = (double)r * ht + sumH + v.val();
    s.t1 = ts;
    s.miss1 = !(r >= 1 && r <= n1);   // the bracket missed: left to the fallback
  }
}
// S1 by bisection over the FP64 bits of |a|
template <int K>
__device__ __noinline__ int pn_fallback1(int nx) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0;
  unsigned long long lo = s.lo1 > 4 ? (unsigned long long)__double_as_longlong((double)__uint_as_float(s.lo1 - 4)) : 0ull;
  unsigned long long hi = (unsigned long long)__double_as_longlong((double)__uint_as_float(min(s.hi1 + 4, kInfKey))) + 1;
  const unsigned long long zero = A().word();
  // (the certificate of FP32 data ranks by the stored pairs: t* may be any value
  // near the kbar-th, and near an optimum, where the pooled block ties, the
  // search comes here often)
  auto rank = [&](int64_t j) { return K == PK_PAIR64 && s.a.mode == PM_EVAL ? fabs(pn_G64<K>(j)) * s.a.kc.inv2l : pn_a64<K>(j); };
  while (hi - lo > 1) {
    const unsigned long long mid = lo + (hi - lo) / 2;
    unsigned n = 0;
#pragma unroll 1
    for (int i = w0 + lane; i < w1; i += 32)
      if (s.fl[i] & 4) n += (unsigned long long)__double_as_longlong(rank(s.cb + i)) >= mid ? 1u : 0u;
    nx = pn_small_sum<K>(nx, zero, zero, n, 0u);
    if (s.cnt0 >= (unsigned)s.kb) lo = mid;
    else hi = mid;
    __syncthreads();
  }
  double ts = __longlong_as_double((long long)lo);
  if (K != PK_F64) ts = (double)(float)ts;   // (ties in FP32 brought the search here)
  const double ht = huber_d<double>(ts, s.a.M);
  A v;
#pragma unroll 1
  for (int i = w0 + lane; i < w1; i += 32)
    if ((s.fl[i] & 4) && rank(s.cb + i) > ts * (1.0 - 0x1p-40)) {
      const double ad = pn_a64<K>(s.cb + i);
      if (ad > ts) v.add(huber_d<double>(ad, s.a.M) - ht);
    }
  nx = pn_small_sum<K>(nx, v.word(), zero, 0u, 0u);
  if (threadIdx.x == 0) {
    s.top = (double)s.kb * ht + s.red_[0];
    s.t1 = ts;
  }
  __syncthreads();
  return nx;
}

// ---------------------------------------------------- stage 2, exchange 2
__device__ __forceinline__ void pn_list(int* n, unsigned long long* l, double x) {
  const int at = atomicAdd(n, 1);
  if (at < pn().a.lc) l[at] = (unsigned long long)__double_as_longlong(x);
}
// Exact sums over the coordinates beyond the brackets (margins cover the FP32
// rounding of the keys), the others into lists, to every CTA
template <int K>
__device__ __noinline__ void pn_stage2(int nx, bool d1, bool d3) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0, nw = s.nw[warp];
  const PConst& kc = s.a.kc;
  const uint32_t a1 = s.lo1 > 4 ? s.lo1 - 4 : 1u, b1 = s.hi1 + 4;
  const uint32_t a3 = s.lo3 > 2 ? s.lo3 - 2 : 0u, b3 = min(s.hi3 + 2, kInfKey - 1);
  // a coordinate is surely at z = 1 (not at z = 1) for every c of the bracket
  // when |v_j| is at least T(upper end) (below T(lower end)), with a margin
  // over the FP32 evaluation of T
  const float cl = __uint_as_float(a3), ch = __uint_as_float(b3);
  const float Tl = (a3 < kc.krho ? cl * kc.kTc_f : cl + kc.M) * (1.f - 0x1p-20f);
  const float Th = (b3 < kc.krho ? ch * kc.kTc_f : ch + kc.M) * (1.f + 0x1p-20f);
  A v1, v3;
  unsigned ndef = 0, ntop = 0, nmid = 0;
#pragma unroll 1
  for (int i = w0 + lane; i < w1; i += 32) {
    if (d1) {
      const uint32_t key = s.ka[i];
      if (key >= a1) {
        const double ad = pn_a64<K>(s.cb + i);
        if (key >= b1) {
          ++ndef;
          v1.add(huber_d<double>(ad, s.a.M));
        } else pn_list(&s.n1, s.loc1, ad);
      }
    }
    if (d3 && (s.fl[i] & 6) == 4) {
      const float m = s.mv[i];
      const uint32_t mk = key_of(m);
      if (mk > a3) {
        if (mk > b3 && m > Th) ++ntop;
        else if (mk > b3 && m < Tl) {
          ++nmid;
          v3.add(m);
        } else pn_list(&s.n3, s.loc3, (double)m);
      }
    }
  }
  if (d3) {
#pragma unroll 1
    for (int e = lane; e < nw; e += 32) {
      const int i = s.wl[w0 + e];
      if (!(s.fl[i] & 4)) continue;
      const double md = fabs(s.vw[w0 + e]);
      if (is_zero_bits(md)) continue;
      const float m = s.mv[i];
      const uint32_t mk = key_of(m);
      if (mk > a3 || a3 == 0) {
        if (mk > b3 && m > Th) ++ntop;
        else if (mk > b3 && m < Tl && m < FLT_MAX) {   // (FLT_MAX: a magnitude beyond FP32)
          ++nmid;
          v3.add(md);
        } else pn_list(&s.n3, s.loc3, md);
      }
    }
  }
  ndef = __reduce_add_sync(0xffffffffu, ndef);
  ntop = __reduce_add_sync(0xffffffffu, ntop);
  nmid = __reduce_add_sync(0xffffffffu, nmid);
  if (ndef) warp_merge<(K != PK_PAIR)>(v1);
  if (nmid) warp_merge<(K != PK_PAIR)>(v3);
  if (lane == 0) {
    unsigned long long* rw = s.red + warp * XW_WORDS;
    rw[0] = v1.word();
    rw[1] = v3.word();
    rw[2] = ndef;
    rw[3] = pack2(ntop, nmid);
    rw[4] = 0ull;
  }
  __syncthreads();
  // the lists go out with the sums: each CTA's into its segment everywhere
  const int S = s.a.cl, lc = s.a.lc, n1 = min(s.n1, lc), n3 = min(s.n3, lc);
#pragma unroll 1
  for (int e = tid; e < n1 + n3; e += blockDim.x) {
    const unsigned long long x = e < n1 ? s.loc1[e] : s.loc3[e - n1];
    const uint32_t dst = smem_u32(e < n1 ? s.seg1 + s.rank * lc + e : s.seg3 + s.rank * lc + (e - n1));
#pragma unroll 4
    for (int r = 0; r < S; ++r) st_cluster_u64(pn_remote(dst, r), x);
  }
  if (tid == 0) s.red[4] = pack2((unsigned)s.n1, (unsigned)s.n3);
  pn_exchange<K>(nx, 0, 2, 5);
}

// The lists of the cluster, flat in CTA order and then sorted (descending) by
// counting: the order inside a CTA's list is arbitrary, the sorted one is not.
// Returns the entries of both lists (low and high half), or ~0 for one that
// overflowed somewhere.
__device__ __noinline__ unsigned long long pn_sort(int nx, bool d1, bool d3) {
  PnSh& s = pn();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, S = s.a.cl, lc = s.a.lc;
  // every warp scans the CTAs' counts (lane r: CTA r), then copies its CTAs' lists
  const unsigned long long n = lane < S ? *pn_slot(nx, lane, 4) : 0ull;
  const unsigned n1 = (unsigned)n, n3 = (unsigned)(n >> 32);
  unsigned e1 = n1, e3 = n3;   // inclusive sums
#pragma unroll
  for (int o = 1; o < PN_MAXCL; o <<= 1) {
    const unsigned a = __shfl_up_sync(0xffffffffu, e1, o), b = __shfl_up_sync(0xffffffffu, e3, o);
    if (lane >= o) {
      e1 += a;
      e3 += b;
    }
  }
  const unsigned t1 = __shfl_sync(0xffffffffu, e1, PN_MAXCL - 1), t3 = __shfl_sync(0xffffffffu, e3, PN_MAXCL - 1);
  const bool o1 = __any_sync(0xffffffffu, n1 > (unsigned)lc) || t1 > PN_CAP;
  const bool o3 = __any_sync(0xffffffffu, n3 > (unsigned)lc) || t3 > PN_CAP;
  const unsigned m1 = d1 && !o1 ? t1 : 0u, m3 = d3 && !o3 ? t3 : 0u;
  for (int r = warp; r < S; r += blockDim.x >> 5) {
    const unsigned c1 = __shfl_sync(0xffffffffu, n1, r), b1 = __shfl_sync(0xffffffffu, e1, r) - c1;
    const unsigned c3 = __shfl_sync(0xffffffffu, n3, r), b3 = __shfl_sync(0xffffffffu, e3, r) - c3;
    if (m1)
      for (unsigned e = lane; e < c1; e += 32) s.flat1[b1 + e] = s.seg1[r * lc + e];
    if (m3)
      for (unsigned e = lane; e < c3; e += 32) s.flat3[b3 + e] = s.seg3[r * lc + e];
  }
  __syncthreads();
#pragma unroll 1
  for (unsigned e = tid; e < m1 + m3; e += blockDim.x) {
    const bool one = e < m1;
    const unsigned k = one ? m1 : m3, i0 = one ? e : e - m1;
    const unsigned long long* f = one ? s.flat1 : s.flat3;
    const unsigned long long x = f[i0];
    unsigned at = 0;
#pragma unroll 4
    for (unsigned i = 0; i < k; ++i) {
      const unsigned long long y = f[i];
      at += (y > x || (y == x && i < i0)) ? 1u : 0u;
    }
    (one ? s.srt1 : s.srt3)[at] = x;
    if (!one) s.f3[at] = (float)__longlong_as_double((long long)x);
  }
  __syncthreads();
  return pack2(o1 ? ~0u : t1, o3 ? ~0u : t3);
}

// Both searches to their ends once the brackets are narrow; the searches of a
// list that overflowed go on by rounds, or without lists
template <int K>
__device__ __noinline__ int pn_repair(int nx, bool d1, bool d3, bool o1, bool o3) {
  PnSh& s = pn();
  for (;;) {
    const bool again1 = d1 && o1 && s.hi1 - s.lo1 > 1, again3 = d3 && o3 && s.hi3 - s.lo3 > 1;
    __syncthreads();
    if (d1 && !again1) nx = pn_fallback1<K>(nx);
    if (d3 && !again3) nx = pn_fallback3<K>(nx);
    d1 = again1;
    d3 = again3;
    if (!d1 && !d3) return nx;
    if (threadIdx.x == 0) {
      s.more1 = d1;
      s.more3 = d3;
      s.miss1 = s.miss3 = 0;
      s.n1 = s.n3 = 0;
    }
    __syncthreads();
    nx = pn_more_rounds<K>(nx);
    pn_stage2<K>(nx, d1, d3);
    const unsigned long long t = pn_sort(nx, d1, d3);
    o1 = (unsigned)t == ~0u;
    o3 = (unsigned)(t >> 32) == ~0u;
    if (threadIdx.x < 32 && d1 && !o1) pn_finish1<K>(nx, (int)(unsigned)t);
    if (threadIdx.x >= 32 && threadIdx.x < 64 && d3 && !o3) pn_finish3<K>(nx, (int)(t >> 32));
    __syncthreads();
    ++nx;
    d1 = d1 && (o1 || s.miss1);
    d3 = d3 && (o3 || s.miss3);
    if (!d1 && !d3) return nx;
  }
}

// --------------------------------------------------------------- g(beta), S2
// Newton's method on the concave sum_j min(|beta_j|, w) - kbar w from the right
// of its root (w <= S / kbar there): w <- S_below / (kbar - N_above) decreases
// to the root and ends when the classification stands, or w does not fall any
// more (values equal to the level to rounding can fall on either side of it in turn).
template <int K>
__device__ __noinline__ int pn_level(int nx) {
  using A = Acc<(K != PK_PAIR)>;
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = (warp - 1) * s.a.wch, nw = s.nw[warp];
  if (threadIdx.x == 0) {
    s.w = s.tot[XS_B] / (double)s.kb;
    s.go = 1;
    s.mu = -1.0;
  }
  __syncthreads();
  for (int it = 0; s.go && it < 200; ++it) {
    const double w = s.w;
    A v0, v1;
    unsigned na = 0;
#pragma unroll 1
    for (int e = lane; e < nw; e += 32) {
      const int i = s.wl[w0 + e];
      if (!(s.fl[i] & 4)) continue;
      const double ab = fabs(s.a.mode == PM_ITER ? s.bcur[s.cb + i] : s.vw[w0 + e]);
      if (ab > w) {
        ++na;
        v0.add(ab);
        v1.add(ab * ab);
      }
    }
    nx = pn_small_sum<K>(nx, v0.word(), v1.word(), na, 0u);
    if (threadIdx.x == 0) {
      const double Nab = (double)s.cnt0, Sbel = s.tot[XS_B] - s.red_[0];
      if ((double)s.kb - Nab <= 0.5) {   // the budget is filled by the coordinates above
        s.g = 0.5 * (s.tot[XS_J1B2] + s.tot[XS_B2]);
        s.go = 0;
      } else {
        const double wn = Sbel / ((double)s.kb - Nab);
        if (s.mu == Nab || !(wn < s.w)) {
          s.g = 0.5 * (s.tot[XS_J1B2] + s.red_[1] + wn * Sbel);
          s.go = 0;
        }
        s.mu = Nab;
        s.w = wn;
      }
    }
    __syncthreads();
  }
  return nx;
}

// Stage 1 of this warp's coordinates again with momentum 0 (after a restart)
template <int K>
__device__ __noinline__ unsigned pn_again() {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0, nw = s.nw[warp];
  unsigned nzv = 0;
#pragma unroll 1
  for (int i = w0 + lane; i < w1; i += 32) {
    const uint8_t f8 = s.fl[i];
    if ((f8 & 6) != 4) continue;   // narrow and free
    const float v = -(s.a.kc.s_f * static_cast<const float2*>(s.Gcur)[s.cb + i].x);
    s.fl[i] = (f8 & ~1) | (v < 0.f ? 1 : 0);
    s.mv[i] = fabsf(v);
    nzv += v != 0.f;
  }
  __syncwarp();
#pragma unroll 1
  for (int e = lane; e < nw; e += 32) {
    const int i = s.wl[w0 + e];
    const uint8_t f8 = s.fl[i];
    if (!(f8 & 12)) continue;
    const double v = pn_v_wide<K>(s.cb + i, s.bcur[s.cb + i], 0.0);
    s.vw[w0 + e] = v;
    s.fl[i] = (f8 & ~1) | (v < 0.0 ? 1 : 0);
    if (f8 & 4) {
      s.mv[i] = fminf((float)fabs(v), FLT_MAX);
      nzv += !is_zero_bits(v);
    }
  }
  __syncwarp();
  return nzv;
}

// Phi, Psi and the loop's decisions (thread 0).  Everything the others read:
// flags (1 stop, 2 Phi improved, 4 Psi improved, 8 restart)
__device__ __noinline__ void pn_decisions() {
  PnSh& s = pn();
  const NArgs& a = s.a;
  const IterState& st0 = s.st;
  IterState* st = a.st + (a.seg_node ? a.seg_node[s.prob] : s.prob);
  const double gval = s.g;
  const double phi = s.loss[0] + 2.0 * a.lambda2 * gval;
  const double psi = s.loss[1] - 2.0 * a.lambda2 * (s.tot[XS_J1H] + s.top);
  const bool nonfinite = s.bad > 0;
  if (a.mode == PM_GVAL || a.mode == PM_GSTAR) {
    if (s.rank == 0)
      a.out[0] = a.mode == PM_GVAL                                            ? gval
                 : nonfinite                                                 ? __longlong_as_double(0x7ff8000000000000ll)
                 : s.nnz > 0 || (s.dom > 0 && s.kb > 0) ? INFINITY
                                                        : s.tot[XS_J1H] + s.top;
    return;
  }
  if (a.mode != PM_ITER) {
    if (s.rank == 0) {
      double* o = a.out + (size_t)s.item * a.out_stride + 2 * s.q0;
      o[0] = phi;
      o[1] = psi;
      if (nonfinite) atomicCAS(a.status, ST_OK, ST_NUMERIC);
    }
    return;
  }
  const int t = st0.iter;
  bool stop = nonfinite, restart = false, imp_p = false, imp_d = false;
  double gap_ref = st0.gap_ref, phi_best = st0.phi_best, psi_best = st0.psi_best;
  int have_ref = st0.have_ref, restarts = st0.restarts;
  if (phi < phi_best) { phi_best = phi; imp_p = true; }
  if (psi > psi_best) { psi_best = psi; imp_d = true; }
  const double gap = phi - psi;
  if (a.method == 0 && a.restart_rule == 0) {         // duality-gap restart (Sec. 3.4)
    if (!have_ref) {
      if (isfinite(gap)) { gap_ref = gap; have_ref = 1; }
    } else if (t >= 1 && gap <= gap_ref / a.eta) {
      restart = true;
      gap_ref = gap;
      ++restarts;
    }
  } else if (a.method == 0 && a.restart_rule == 1) {  // function value (O'Donoghue and Candes)
    if (t > 1 && phi > st0.phi_t) {
      restart = true;
      ++restarts;
    }
  }
  if (isfinite(phi_best) && phi_best - psi_best <= st0.tol * fmax(1.0, fabs(phi_best))) stop = true;
  if (t >= a.max_iters) stop = true;
  // stall rule (see pphase.cuh)
  double stall_gap = st0.stall_gap;
  int stall_iter = st0.stall_iter, stalled = 0, cut_rule = 0;
  const double gbest = phi_best - psi_best;
  if (!(gbest >= 0.9 * stall_gap)) {
    stall_gap = gbest;
    stall_iter = t;
  } else if (a.stall_min > 0 && t - stall_iter >= max(a.stall_min, t / 4)) {
    stop = true;
    stalled = 1;
  }
  // dynamic termination (Sec. 5.3): prune wins when both rules hold
  if (st0.cutoff_on) {
    if (isfinite(phi_best) && phi_best <= st0.cutoff) { stop = true; cut_rule = 1; }
    if (psi_best >= st0.cutoff) { stop = true; cut_rule = 2; }
  }
  s.flags = (stop ? 1 : 0) | (imp_p ? 2 : 0) | (imp_d ? 4 : 0) | (restart ? 8 : 0);
  if (s.rank != 0) return;
  // this part of the state is read by no other CTA of this launch any more
  if (nonfinite) atomicCAS(a.status, ST_OK, ST_NUMERIC);
  st->phi_t = phi;
  st->psi_t = psi;
  st->g_t = gval;
  st->phi_best = phi_best;
  st->psi_best = psi_best;
  st->gap_ref = gap_ref;
  st->have_ref = have_ref;
  st->restarts = restarts;
  st->stall_gap = stall_gap;
  st->stall_iter = stall_iter;
  st->stalled = stalled;
  st->cut_rule = cut_rule;
}

// Stage 1 of the standalone operations over this warp's coordinates
template <int K>
__device__ __noinline__ void pn_load(Acc<true> (&sum)[XS_NSUM], unsigned& nnz, unsigned& dom, unsigned& bad, unsigned& nzv,
                                     unsigned& j1, unsigned& jf) {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, mode = s.a.mode;
  const int wch = s.a.wch, w0 = (warp - 1) * wch, w1 = min(s.cnt, w0 + wch);
  int nw = 0;
#pragma unroll 1
  for (int i0 = w0; i0 < w0 + wch; i0 += 32) {
    const int i = i0 + lane;
    bool wide = false;
    uint32_t key = 0;
    float m = 0.f;
    uint8_t f8 = 0;
    double x = 0.0;
    if (i < w1) {
      const int64_t j = s.cb + i;
      const int8_t f = s.fix ? s.fix[j] : (int8_t)0;
      x = pn_vin<K>(j);
      f8 = f == 0 ? 4 : f > 0 ? 8 : 0;
      j1 += f > 0;
      jf += f == 0;
      // (an FP64 value beyond FP32's range is finite all the same)
      const bool inf_nan = (((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ffu) == 0x7ffu;
      const float ax = fminf(fabsf((float)x), FLT_MAX);
      if (inf_nan && (mode == PM_PROX || (x != x && f >= 0))) ++bad;
      if (mode == PM_GSTAR) {   // an infinite value: dom on Jf, nnz on J1
        if (f == 0) key = key_of(ax);
        if (inf_nan && f == 0) ++dom;
        if (f > 0) {
          if (inf_nan) ++nnz;
          else sum[XS_J1H].add(huber_d<double>(fabs(x), s.a.M));
        }
      } else if (mode == PM_PROX) {
        wide = K == PK_F64 ? f >= 0 : f > 0;   // (an FP32 |v_j| is exact in its FP32 word)
        if (__double_as_longlong(x) < 0) f8 |= 1;
        if (f == 0) {
          m = ax;
          nzv += !is_zero_bits(x);
        }
      } else if (!is_zero_bits(x)) {   // g's value
        wide = true;
        const double ab = fabs(x);
        if (f < 0 || ab > s.a.kc.Mtol || (inf_nan && x == x)) ++dom;
        if (f > 0) sum[XS_J1B2].add(ab * ab);
        else if (f == 0) {
          sum[XS_B].add(ab);
          sum[XS_B2].add(ab * ab);
          ++nnz;
        }
      }
      if (wide) f8 |= 2;
    }
    s.ka[i] = key;
    s.mv[i] = m;
    s.fl[i] = f8;
    const unsigned wm = __ballot_sync(0xffffffffu, wide);
    if (wide) {
      const int at = w0 + nw + __popc(wm & ((1u << lane) - 1u));
      s.wl[at] = (uint16_t)i;
      s.vw[at] = x;
    }
    nw += __popc(wm);
  }
  if (lane == 0) s.nw[warp] = nw;
  j1 = __reduce_add_sync(0xffffffffu, j1);
  jf = __reduce_add_sync(0xffffffffu, jf);
  __syncwarp();
}

// The standalone prox's output and counts.  A non-finite input poisons them:
// beta all NaN, counts -1.
template <int K>
__device__ __noinline__ void pn_prox_out(int nx, int kb, bool s3, unsigned bad) {
  PnSh& s = pn();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = (warp - 1) * s.a.wch, w1 = warp ? min(s.cnt, w0 + s.a.wch) : w0, nw = s.nw[warp];
  const double c = kb <= 0 ? INFINITY : s3 ? s.c : 0.0, T = pn_T(c), inv1r = s.a.kc.inv1r, M = s.a.M;
  const float ccd = kb <= 0 ? INFINITY : s3 ? s.ccd : 0.f;   // an FP32 m exceeds c iff it exceeds c rounded down
  unsigned ntop = 0, nnz = 0;
#pragma unroll 1
  for (int u = lane; u < (w1 - w0) + nw; u += 32) {
    // the coordinates with FP32 words (FP64: those fixed out), then the others from the list
    const bool narrow = u < w1 - w0;
    const int e = w0 + u - (narrow ? 0 : w1 - w0);
    const int i = narrow ? e : s.wl[e];
    const uint8_t f8 = s.fl[i];
    if (narrow && (f8 & 2)) continue;
    double b = 0.0;
    if (bad) b = __longlong_as_double(0x7ff8000000000000ll);
    else if (f8 & 8) b = fmin(fmax(s.vw[e] * inv1r, -M), M);
    else if ((f8 & 4) && (!narrow || s.mv[i] > ccd)) {
      const double m = narrow ? (double)s.mv[i] : fabs(s.vw[e]);
      const double r = fmax(0.0, fmin(fmin(m - c, m * inv1r), M));
      if (r > 0.0) {
        ++nnz;
        ntop += m >= T;
        b = (f8 & 1) ? -r : r;
      }
    }
    if (K == PK_F64) static_cast<double*>(s.a.vout)[s.cb + i] = b;
    else static_cast<float*>(s.a.vout)[s.cb + i] = (float)b;
  }
  if (s.a.counts) {
    const unsigned long long zero = Acc<true>().word();
    pn_small_sum<K>(nx, zero, zero, ntop, nnz);
    if (s.rank == 0 && threadIdx.x == 0) {
      s.a.counts[0] = bad ? -1 : (int)s.cnt0;
      s.a.counts[1] = bad ? -1 : (int)s.cnt1;
    }
  }
}

// ==================================================================== kernel
template <int K>
__global__ void __launch_bounds__(32 * PN_MAXW, K == PK_F64 ? 1 : 2) pnode_kernel(const __grid_constant__ NArgs args) {
  using A = Acc<(K != PK_PAIR)>;
  constexpr bool F64 = K == PK_F64;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
  PnSh& s = pn();
  {
    const int S = args.cl;
    const int prob = (int)blockIdx.x / S;
    const bool it = args.mode == PM_ITER;
    const int node = args.seg_node ? args.seg_node[prob] : prob;
    const IterState* st = it ? args.st + node : nullptr;
    // the node's state and the launch's arguments, once into shared memory
    static_assert(sizeof(IterState) % 8 == 0 && sizeof(NArgs) % 8 == 0, "copied by 8-byte words");
    if (it) {
      const unsigned long long* sw = reinterpret_cast<const unsigned long long*>(st);
      for (int i = tid; i < (int)(sizeof(IterState) / 8); i += blockDim.x)
        reinterpret_cast<unsigned long long*>(&s.st)[i] = __ldcg(sw + i);
    }
    const unsigned long long* aw = reinterpret_cast<const unsigned long long*>(&args);
    for (int i = tid; i < (int)(sizeof(NArgs) / 8); i += blockDim.x) reinterpret_cast<unsigned long long*>(&s.a)[i] = aw[i];
    if (tid < PN_MAXW) s.nw[tid] = 0;
    __syncthreads();
    if (it && s.st.done) return;   // uniform over the cluster: every CTA reads the same flag
    cluster_arrive();              // completed before the first push: every CTA of the cluster runs
    // (three warps set up side by side)
    if (tid == 0) {
      s.prob = prob;
      s.rank = (int)blockIdx.x - prob * S;
      const bool ev = args.mode == PM_EVAL;
      s.item = it ? node : ev ? prob / args.nq : 0;
      s.q0 = ev ? prob % args.nq : 0;
      const size_t slot = it ? prob : s.item;
      s.bcur = static_cast<const double*>(it ? s.st.beta_cur : ev ? args.ev[s.item].beta : nullptr);
      s.bprev = it ? static_cast<const double*>(s.st.beta_prev) : nullptr;
      s.fix = args.fix ? args.fix + (size_t)s.item * args.fix_stride : nullptr;
      s.part = static_cast<const double*>(args.part) + slot * args.part_stride + (size_t)s.q0 * args.p;   // 8-byte elements
      s.Gprev = it ? s.st.G_prev : nullptr;
      s.Gcur = it ? s.st.G_cur : static_cast<double*>(args.gev) + (size_t)prob * args.p;
      s.kb = it ? s.st.kbar : args.k;
      s.pb = it ? s.st.pbar : (int)args.p;
      if (ev && args.cnt) {
        s.kb = args.k - args.cnt[3 * s.item];
        s.pb = args.cnt[3 * s.item + 1];
      }
      s.cb = (int64_t)s.rank * args.cpc;
      s.cnt = (int)max((int64_t)0, min(args.p, s.cb + args.cpc) - s.cb);
      s.c1lo = (unsigned)s.pb;
    } else if (tid == 32) {
      unsigned char* q = pn_raw + (sizeof(PnSh) + 15) / 16 * 16;
      auto take = [&](size_t bytes) {
        unsigned char* r = q;
        q += bytes;
        return r;
      };
      const size_t cp = (size_t)(W - 1) * args.wch;
      s.xbuf = reinterpret_cast<unsigned long long*>(take((size_t)2 * S * XW_WORDS * 8));
      s.red = reinterpret_cast<unsigned long long*>(take((size_t)W * XW_WORDS * 8));
      s.seg1 = reinterpret_cast<unsigned long long*>(take((size_t)S * args.lc * 8));
      s.seg3 = reinterpret_cast<unsigned long long*>(take((size_t)S * args.lc * 8));
      s.loc1 = reinterpret_cast<unsigned long long*>(take((size_t)args.lc * 8));
      s.loc3 = reinterpret_cast<unsigned long long*>(take((size_t)args.lc * 8));
      s.flat1 = reinterpret_cast<unsigned long long*>(take(PN_CAP * 8));
      s.flat3 = reinterpret_cast<unsigned long long*>(take(PN_CAP * 8));
      s.srt1 = reinterpret_cast<unsigned long long*>(take(PN_CAP * 8));
      s.srt3 = reinterpret_cast<unsigned long long*>(take(PN_CAP * 8));
      s.vw = reinterpret_cast<double*>(take(cp * 8));
      s.ka = reinterpret_cast<uint32_t*>(take(cp * 4));
      s.mv = reinterpret_cast<float*>(take(cp * 4));
      s.wl = reinterpret_cast<uint16_t*>(take(cp * 2));
      s.fl = reinterpret_cast<uint8_t*>(take(cp));
    } else if (tid == 64) {
      s.lo1 = 0;
      s.hi1 = kInfKey + 1;
      s.lo3 = 0;
      s.hi3 = kInfKey;
      s.c1hi = s.cmhi = s.cthi = s.cmlo = s.ctlo = 0;
      s.z3lo = s.z3hi = 0.f;
      s.more1 = s.more3 = s.miss1 = s.miss3 = s.n1 = s.n3 = 0;
      s.c = 0.0;
      s.ccd = 0.f;
      s.t1 = s.top = s.w = 0.0;
      s.tau = 1.0;
      s.mom = 0.0;
    }
    __syncthreads();
    if (args.tiles) {   // slots of the products' partial tiles that this CTA's coordinates meet
      const int t0 = (int)(s.cb / BG_BM), nt = s.cnt > 0 ? (int)((s.cb + s.cnt - 1) / BG_BM) - t0 + 1 : 0;
      for (int e = tid; e < nt * args.NB; e += blockDim.x) {
        const int q = e / nt, o = e - q * nt;
        s.nsl[q][o] = (uint8_t)bg_slots(args.s2, (t0 + o) * args.s2.NT + (q * args.m + prob) / args.s2.BN);
      }
      __syncthreads();
    }
  }
  const int mode = s.a.mode;
  const bool iter = mode == PM_ITER, alone = K != PK_PAIR && mode >= PM_PROX;
  const int64_t cb = s.cb;
  const int wch = s.a.wch, w0 = (warp - 1) * wch, w1 = warp ? min(s.cnt, w0 + wch) : w0;
  const PConst& kc = s.a.kc;
  int kb = s.kb;   // (standalone: known after exchange 1)
  const int t = iter ? s.st.iter : 0;

  // ----------------------------------------------------- stage 1, exchange 1
  // In the loop beta^t (t >= 1) is the prox output of the last iteration, whose
  // threshold c fixes its water level w = min(c / rho, M) (see pphase.cuh)
  const double w_closed = iter ? s.st.w_next : 0.0;
  const bool w_known = !is_zero_bits(w_closed);
  const double mu = iter ? s.st.ps.mom : 0.0;
  A sum[XS_NSUM];
  unsigned c_nnz = 0, c_dom = 0, c_bad = 0, c_nab = 0, c_nzv = 0, c_j1 = 0, c_jf = 0;
  if (alone) {
    if constexpr (K != PK_PAIR)
      if (warp) pn_load<K>(sum, c_nnz, c_dom, c_bad, c_nzv, c_j1, c_jf);
  } else if (warp == 0) {   // the loss sums of the pass, in FP64
    const double* ls = s.a.lsum + (size_t)(iter ? s.prob : s.item) * s.a.lsum_stride;
    double f = 0.0, d = 0.0;
#pragma unroll 4
    for (int i = lane; i < s.a.nl; i += 32) {
      f += __ldcg(ls + (size_t)i * PN_LSUM);
      d += __ldcg(ls + (size_t)i * PN_LSUM + 1 + s.q0);
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      f += __shfl_xor_sync(0xffffffffu, f, o);
      d += __shfl_xor_sync(0xffffffffu, d, o);
    }
    if (lane == 0) {
      s.loss[0] = f;
      s.loss[1] = d;
    }
  } else {
    const float mu32 = iter ? s.st.mu32 : 0.f, opm32 = iter ? s.st.opm32 : 1.f;
    const bool mu0 = is_zero_bits(mu), ls = s.a.loss == 0;
    int nw = 0;
#pragma unroll 1
    for (int i0 = w0; i0 < w0 + wch; i0 += 32) {
      const int i = i0 + lane;
      const int64_t j = cb + i;
      bool wide = false;
      uint32_t key = 0;
      float m = 0.f;
      uint8_t f8 = 0;
      if (i < w1) {
        const int8_t f = s.fix ? s.fix[j] : (int8_t)0;
        const double b = s.bcur[j];
        const double bp = iter ? s.bprev[j] : 0.0;
        float gp = 0.f;
        if (!F64 && iter && ls && !mu0) gp = static_cast<const float2*>(s.Gprev)[j].x;
        f8 = f == 0 ? 4 : f > 0 ? 8 : 0;
        wide = F64 || f > 0 || !is_zero_bits(b) || !is_zero_bits(bp);
        float aa, gf;
        if constexpr (F64) {
          const double G = pn_gdbl<K>(j, 0);
          static_cast<double*>(s.Gcur)[j] = G;
          gf = (float)G;
          const double ad = fabs(G) * kc.inv2l;
          // an FP64 value beyond FP32 is finite all the same: its key is the largest one's
          aa = ad < INFINITY ? fminf((float)ad, FLT_MAX) : INFINITY;
        } else {
          const ffs g = pn_gpair(j, 0);
          static_cast<float2*>(s.Gcur)[j] = make_float2(g.hi, g.lo);
          gf = g.hi;
          aa = fabsf(gf) * kc.inv2l_f;
        }
        if (!(aa < INFINITY)) ++c_bad;
        if (f == 0) key = key_of(aa);
        if (!F64 && iter && !wide && f == 0) {   // y_j = 0: v_j = -s gy_j in FP32
          float gy = gf;
          if (!mu0) gy = ls ? opm32 * gf - mu32 * gp : pn_gpair(j, 1).hi;
          const float v = -(kc.s_f * gy);
          if (v < 0.f) f8 |= 1;
          m = fabsf(v);
          if (m > 0.f) ++c_nzv;
        }
        if (wide) f8 |= 2;
      }
      s.ka[i] = key;
      s.mv[i] = m;
      s.fl[i] = f8;
      const unsigned wm = __ballot_sync(0xffffffffu, wide);
      if (wide) s.wl[w0 + nw + __popc(wm & ((1u << lane) - 1u))] = (uint16_t)i;
      nw += __popc(wm);
    }
    if (lane == 0) s.nw[warp] = nw;
    __syncwarp();
#pragma unroll 1
    for (int e = lane; e < nw; e += 32) {
      const int i = s.wl[w0 + e];
      const int64_t j = cb + i;
      const double b = s.bcur[j];
      const uint8_t f8 = s.fl[i];
      if (f8 & 8) sum[XS_J1H].add(huber_d<double>(pn_a64<K>(j), s.a.M));
      if (!iter) s.vw[w0 + e] = b;
      if (!is_zero_bits(b)) {
        const double ab = fabs(b);
        A a1, a2;   // |b| and b^2 (FP32 data: as pairs, one conversion for both)
        bool above;
        if constexpr (K != PK_PAIR) {
          a1.s = ab;
          a2.s = ab * ab;
          above = w_known && ab > w_closed;
          if (!(ab < INFINITY)) ++c_bad;
        } else {
          a1.s = ff_of(ab);
          const float h = a1.s.hi * a1.s.hi;
          a2.s.hi = h;
          a2.s.lo = fmaf(a1.s.hi, a1.s.hi, -h) + 2.f * a1.s.hi * a1.s.lo;
          above = w_known && (unsigned long long)__double_as_longlong(ab) > (unsigned long long)__double_as_longlong(w_closed);
          if (!(a1.s.hi < INFINITY)) ++c_bad;
        }
        if (!(f8 & 12)) ++c_dom;
        else {
          if ((unsigned long long)__double_as_longlong(ab) > (unsigned long long)__double_as_longlong(kc.Mtol)) ++c_dom;
          if (f8 & 8) sum[XS_J1B2].merge(a2);
          else {
            sum[XS_B].merge(a1);
            sum[XS_B2].merge(a2);
            ++c_nnz;
            if (above) {
              ++c_nab;
              sum[XS_SAB].merge(a1);
              sum[XS_QAB].merge(a2);
            }
          }
        }
      }
      if (iter && (f8 & 12)) {
        const double v = pn_v_wide<K>(j, b, mu);
        s.vw[w0 + e] = v;
        if (__double_as_longlong(v) < 0) s.fl[i] = f8 | 1;
        if (f8 & 4) {
          s.mv[i] = fminf((float)fabs(v), FLT_MAX);
          if (!is_zero_bits(v)) ++c_nzv;
        }
      }
    }
    __syncwarp();
  }
  bool need1 = alone ? mode == PM_GSTAR : kb > 0 && s.pb > kb, can3 = alone ? mode == PM_PROX : iter && kb > 0;
  const uint32_t k1 = iter ? s.st.key1 : 0u, k3 = iter ? s.st.key3 : 0u;
  uint32_t x1 = k1 ? pn_warm(k1, s.st.win1, 0u, kInfKey + 1, lane) : cand<uint32_t>(0u, kInfKey + 1, lane);
  uint32_t x3 = k3 ? pn_warm(k3, s.st.win3, 0u, kInfKey, lane) : cand<uint32_t>(0u, kInfKey, lane);
  pn_count(need1, can3, x1, x3);
  {
    unsigned long long* rw = s.red + warp * XW_WORDS;
    if (s.nw[warp] > 0 || (alone && warp)) {
#pragma unroll 1
      for (int o = 16; o > 0; o >>= 1)   // the six side by side
#pragma unroll
        for (int i = 0; i < XS_NSUM; ++i) sum[i].merge(A(__shfl_xor_sync(0xffffffffu, sum[i].word(), o)));
      if (lane == 0)
#pragma unroll
        for (int i = 0; i < XS_NSUM; ++i) rw[XW_SUM + i] = sum[i].word();
    } else if (lane < XS_NSUM) rw[XW_SUM + lane] = A().word();
    c_nnz = __reduce_add_sync(0xffffffffu, c_nnz);
    c_dom = __reduce_add_sync(0xffffffffu, c_dom);
    c_bad = __reduce_add_sync(0xffffffffu, c_bad);
    c_nab = __reduce_add_sync(0xffffffffu, c_nab);
    c_nzv = __reduce_add_sync(0xffffffffu, c_nzv);
    if (lane == 0) {
      rw[XW_INT] = pack2(c_nnz, c_dom);
      rw[XW_INT + 1] = pack2(c_bad, c_nzv);
      rw[XW_INT + 2] = c_nab;
      rw[XW_INT + 3] = pack2(c_j1, c_jf);   // (per lane sums only in the standalone modes, reduced there)
    }
  }
  cluster_wait();   // every CTA of the cluster runs
  int nx = 0;
  pn_exchange<K>(nx, XW_SUM, XW_SUM + XS_NSUM, XW_WORDS);
  // S3 has a threshold to find when more coordinates of v are nonzero than the
  // budget holds
  const unsigned long long bz = xcnt(nx, XW_INT + 1);
  const unsigned bad = (unsigned)bz, nzv = (unsigned)(bz >> 32);
  if (alone) {
    const unsigned long long jj = xcnt(nx, XW_INT + 3);
    kb = s.a.k - (int)(unsigned)jj;
    const int pb = (int)(jj >> 32);
    if (tid == 0) {
      s.kb = kb;
      s.pb = pb;
      s.c1lo = (unsigned)pb;
    }
    need1 = need1 && kb > 0 && pb > kb;
    can3 = can3 && kb > 0;
    __syncthreads();
  }
  bool s3 = can3 && (int)nzv > kb && bad == 0;
  const bool s1 = need1 && bad == 0;
  if (warp == 2 % W) {
    if (lane < XS_NSUM) s.tot[lane] = xacc<A>(nx, XW_SUM + lane).val();
    else if (lane == XS_NSUM) {
      const unsigned long long v = xcnt(nx, XW_INT);
      s.nnz = (unsigned)v;
      s.dom = (unsigned)(v >> 32);
      s.bad = bad;
      s.nab = (unsigned)xcnt(nx, XW_INT + 2);
    }
  }
  if (tid == 0 && s3) s.cmlo = s.ctlo = nzv;
  __syncwarp();
  pn_decide(nx, s1, s3, x1, x3);
  __syncthreads();
  ++nx;
  if (s.more1 || s.more3) nx = pn_more_rounds<K>(nx);

  const bool need_b = iter || mode == PM_EVAL || mode == PM_GVAL;
  const bool check_dom = !iter || t == 0;
  const bool g_inf = check_dom && (s.dom > 0 || (kb > 0 && s.tot[XS_B] > s.a.M * (double)kb * (1.0 + 1e-6)) ||
                                   (kb <= 0 && s.tot[XS_B] > 0.0));
  const bool level = need_b && !g_inf && kb > 0 && s.nnz > (unsigned)kb;   // a water level to find
  if (level && !w_known) nx = pn_level<K>(nx);
  // g, and FISTA's next t_k and momentum should this iteration not restart:
  // by warps that have nothing else to do while the searches end
  auto g_closed = [&]() {   // one lane
    if (g_inf) s.g = INFINITY;
    else if (kb <= 0) s.g = 0.5 * s.tot[XS_J1B2];
    else if (!level) s.g = 0.5 * (s.tot[XS_J1B2] + s.tot[XS_B2]);
    else if (w_known) {
      // the closed-form level classifies exactly: a coordinate with
      // |beta_j| = w adds beta_j^2 on either side
      const double r = (double)kb - (double)s.nab, Sbel = s.tot[XS_B] - s.tot[XS_SAB];
      s.g = r <= 0.5 ? 0.5 * (s.tot[XS_J1B2] + s.tot[XS_B2]) : 0.5 * (s.tot[XS_J1B2] + s.tot[XS_QAB] + (Sbel / r) * Sbel);
    }
  };
  auto next_tau = [&]() {   // one lane; after a restart t_k is 1, whose momentum is 0
    if (!iter || s.a.method == 1 || t == 0) return;
    const double tau = s.st.tau, tn = 0.5 * (1.0 + sqrt(1.0 + 4.0 * tau * tau));
    s.tau = tn;
    s.mom = (tn - 1.0) / (0.5 * (1.0 + sqrt(1.0 + 4.0 * tn * tn)));
  };

  // ------------------------------------------------------ stage 2, exchange 2
  bool o1 = false, o3 = false;
  if (s1 || s3) {
    pn_stage2<K>(nx, s1, s3);
    const unsigned long long n = pn_sort(nx, s1, s3);
    o1 = s1 && (unsigned)n == ~0u;
    o3 = s3 && (unsigned)(n >> 32) == ~0u;
    if (warp == 0 && s1 && !o1) pn_finish1<K>(nx, (int)(unsigned)n);
    if (warp == 1 && s3 && !o3) pn_finish3<K>(nx, (int)(n >> 32));
  }
  if (warp == 2 && lane == 0) g_closed();
  if (warp == 3 && lane == 0) next_tau();
  __syncthreads();
  ++nx;
  if ((s1 && (o1 || s.miss1)) || (s3 && (o3 || s.miss3)))
    nx = pn_repair<K>(nx, s1 && (o1 || s.miss1), s3 && (o3 || s.miss3), o1, o3);
  if (kb > 0 && s.pb <= kb && mode != PM_PROX && mode != PM_GVAL) {   // a slack budget: the whole free set (at most kbar coordinates)
    A v;
#pragma unroll 1
    for (int i = w0 + lane; i < w1; i += 32)
      if (s.fl[i] & 4) v.add(huber_d<double>(pn_a64<K>(cb + i), s.a.M));
    nx = pn_small_sum<K>(nx, v.word(), A().word(), 0u, 0u);
    if (tid == 0) {
      s.top = s.red_[0];
      s.t1 = 0.0;
    }
    __syncthreads();
  } else if (tid == 0 && bad) {
    s.top = __longlong_as_double(0x7ff8000000000000ll);
  }

  // ---------------------------------------------------------------------- D
  if (!iter) {
    if (alone && mode == PM_PROX) pn_prox_out<K>(nx, kb, s3, bad);
    else if (tid == 0) pn_decisions();
    return;   // (every push to this CTA has been received: no exchange follows)
  }
  // Thread 0 decides while the other warps form the next point for "no
  // restart" (into a buffer of its own: a stop leaves the last points as they
  // are); a restart forms v again and repeats S3
  auto write_next = [&]() {
    const double c = kb <= 0 ? INFINITY : s3 ? s.c : 0.0;
    const float ccd = kb <= 0 ? INFINITY : s3 ? s.ccd : 0.f;   // an FP32 m exceeds c iff it exceeds c rounded down
    double* out = static_cast<double*>(s.st.beta_next);
    const double inv1r = kc.inv1r, M = s.a.M;
    __nv_bfloat16* brow = s.a.Bp ? s.a.Bp + (size_t)s.prob * s.a.ldp : nullptr;
#pragma unroll 1
    for (int u = lane; u < (w1 - w0) + s.nw[warp]; u += 32) {
      // the warp's narrow coordinates, then its wide ones from the list
      const bool narrow = u < w1 - w0;
      const int e = w0 + u - (narrow ? 0 : w1 - w0);
      const int i = narrow ? e : s.wl[e];
      const uint8_t f8 = s.fl[i];
      if (narrow && (f8 & 2)) continue;
      const int64_t j = cb + i;
      double b = 0.0;
      const bool nz = narrow ? (f8 & 4) && s.mv[i] > ccd : (f8 & 12) != 0;
      if (nz) {
        const double v = narrow ? 0.0 : s.vw[e];
        if (f8 & 8) b = fmin(fmax(v * inv1r, -M), M);
        else {
          const double m = narrow ? (double)s.mv[i] : fabs(v);
          b = m > c ? fmax(0.0, fmin(fmin(m - c, m * inv1r), M)) : 0.0;
          if (f8 & 1) b = -b;
          if (!(m > c)) b = 0.0;
        }
      }
      out[j] = b;
      if (brow) {
        __nv_bfloat16 b1 = __ushort_as_bfloat16(0), b2 = b1, b3 = b1;
        if (!is_zero_bits(b)) split3(b, b1, b2, b3);
        brow[j] = b1;
        brow[s.a.bplane + j] = b2;
        brow[2 * s.a.bplane + j] = b3;
      }
    }
  };
  if (warp == 0) {
    if (lane == 0) pn_decisions();
    __syncwarp();
  } else {
    write_next();
  }
  __syncthreads();
  const int flags = s.flags;
  const bool stop = flags & 1, restart = (flags & 8) != 0 && !stop;
  if (restart && !is_zero_bits(mu)) {
    unsigned nz = 0;
    if (warp) nz = pn_again<K>();
    if (tid == 0) {
      s.lo3 = 0;
      s.hi3 = kInfKey;
      s.cmhi = s.cthi = 0;
      s.z3lo = s.z3hi = 0.f;
      s.more1 = s.more3 = s.miss3 = s.n1 = s.n3 = 0;
    }
    x3 = k3 ? pn_warm(k3, 21, 0u, kInfKey, lane) : cand<uint32_t>(0u, kInfKey, lane);
    pn_count(false, can3, 0u, x3);
    nz = __reduce_add_sync(0xffffffffu, nz);
    {
      unsigned long long* rw = s.red + warp * XW_WORDS;
      if (lane < XS_NSUM) rw[XW_SUM + lane] = A().word();
      if (lane < 3) rw[XW_INT + lane] = lane == 1 ? pack2(0u, nz) : 0ull;
    }
    pn_exchange<K>(nx, XW_SUM, XW_SUM + XS_NSUM, XW_WORDS);
    const unsigned nzv2 = (unsigned)(xcnt(nx, XW_INT + 1) >> 32);
    s3 = can3 && (int)nzv2 > kb;
    if (tid == 0 && s3) s.cmlo = s.ctlo = nzv2;
    __syncwarp();
    pn_decide(nx, false, s3, 0u, x3);
    __syncthreads();
    ++nx;
    if (s3) {
      if (s.more3) nx = pn_more_rounds<K>(nx);
      pn_stage2<K>(nx, false, true);
      const unsigned long long n = pn_sort(nx, false, true);
      o3 = (unsigned)(n >> 32) == ~0u;
      if (warp == 1 && !o3) pn_finish3<K>(nx, (int)(n >> 32));
      __syncthreads();
      ++nx;
      if (o3 || s.miss3) nx = pn_repair<K>(nx, false, true, false, o3);
    }
    if (warp) write_next();
  }

  // -------------------------------------------- best iterates, next pass's area
  const int rk = s.rank * blockDim.x + tid, nk = s.a.cl * blockDim.x;
  if (flags & 6) {
    double* bbest = static_cast<double*>(s.st.beta_best) + cb;
    double* bdbest = static_cast<double*>(s.st.beta_dbest) + cb;
    const double* b = s.bcur + cb;
#pragma unroll 2
    for (int i = tid; i < s.cnt; i += blockDim.x) {
      const double x = b[i];
      if (flags & 2) bbest[i] = x;
      if (flags & 4) bdbest[i] = x;
    }
  }
  if (flags & 4) {
    // the loop's own dual point of the best Psi (its z), for the certificate
    const double* zt = static_cast<const double*>(s.st.z_cur);
    double* zb = static_cast<double*>(s.st.z_dbest);
#pragma unroll 2
    for (int64_t i = rk; i < s.a.n; i += nk) zb[i] = zt[i];
  }
  if (s.a.zero) {
    int4* z = static_cast<int4*>(s.a.zero);
#pragma unroll 2
    for (int64_t i = rk; i < s.a.zero_bytes / 16; i += nk) z[i] = make_int4(0, 0, 0, 0);
  }

  // --------------------------------------------------------------- epilogue
  // (every CTA has read the state: it has been through an exchange since)
  if (s.rank != 0) return;
  IterState* st = s.a.st + (s.a.seg_node ? s.a.seg_node[s.prob] : s.prob);
  if (tid == 32) {
    // predictions of the next thresholds: the last change again, in FP32, with
    // a window of candidates four times the last deviation
    const double c = kb <= 0 ? INFINITY : s3 ? s.c : 0.0;
    const float cf = (float)c, clf = (float)s.st.c_last;
    auto next = [](float x, float last) { return x * (last > 0.f && last < 1e30f ? fminf(fmaxf(x / last, 0.8f), 1.25f) : 1.f); };
    auto window = [](uint32_t pred, float x, int old) {
      if (!pred) return 21;
      const int64_t d = (int64_t)key_of(x) - (int64_t)pred;
      const int e = 34 - __clz((int)min((int64_t)0x3fffffff, d < 0 ? -d : d));
      return min(21, max(max(e, old - 1), 12));
    };
    const bool cok = s3 && cf > 0.f && cf < 1e30f;
    st->key3 = cok ? key_of(next(cf, clf)) : 0u;
    st->win3 = cok ? window(k3, cf, s.st.win3) : 21;
    st->w_next = !stop && s3 ? fmin(c * kc.inv_rho, s.a.M) : 0.0;
    st->c_last = stop ? 0.0 : c;
    st->rho_last = s.a.rho;
  } else if (tid == 64 % blockDim.x) {
    const float tf = (float)s.t1, tlf = (float)s.st.t1_last;
    const bool tok = tf > 0.f && tf < 1e30f;
    const float pr = tf * (tlf > 0.f && tlf < 1e30f ? fminf(fmaxf(tf / tlf, 0.8f), 1.25f) : 1.f);
    st->key1 = tok ? key_of(pr) : 0u;
    int e = 21;
    if (tok && k1) {
      const int64_t d = (int64_t)key_of(tf) - (int64_t)k1;
      e = min(21, max(max(34 - __clz((int)min((int64_t)0x3fffffff, d < 0 ? -d : d)), s.st.win1 - 1), 12));
    }
    st->win1 = e;
    st->t1_last = s.t1;
  } else if (tid == 0) {
    if (stop) {
      st->done = 1;
      st->ps.done = 1;
    } else {
      // rotate: beta_prev <- beta^t, beta_cur <- beta^{t+1}; the old prev is the next spare
      st->beta_prev = s.st.beta_cur;
      st->beta_cur = s.st.beta_next;
      st->beta_next = s.st.beta_prev;
      st->G_prev = s.st.G_cur;
      st->G_cur = s.st.G_prev;
      st->z_prev = s.st.z_cur;
      st->z_cur = s.st.z_prev;
      const bool reset = restart || t == 0 || s.a.method == 1;   // t_k = 1, whose momentum is 0
      const double mo = reset ? 0.0 : s.mom;
      st->tau = reset ? (t == 0 && !restart && s.a.method == 0 ? s.st.tau : 1.0) : s.tau;
      st->iter = t + 1;
      st->ps.beta = s.st.beta_next;
      st->ps.zout = s.st.z_prev;
      st->ps.zprev = s.st.z_cur;
      st->ps.mom = mo;   // the momentum of the next iteration unless it restarts
      st->mu32 = (float)mo;
      st->mu_lo = (float)(mo - (double)(float)mo);
      st->opm32 = (float)(1.0 + mo);
    }
  }
}

}  // namespace

namespace {

// the plan's sizes for clusters of `cl` CTAs; false: a CTA's share does not fit
bool sized(NPlan& pl, int64_t p, int cl, size_t limit) {
  const int64_t cpc = ((p + cl - 1) / cl + 31) / 32 * 32;
  if (cpc > 65536 || (cpc + BG_BM - 1) / BG_BM + 1 > PN_TILES) return false;
  pl.cl = cl;
  pl.cpc = (int)cpc;
  pl.lc = std::min(PN_CAP, 1024 / cl);
  pl.warps = cpc <= 7 * 64 ? 8 : PN_MAXW;
  pl.wch = (int)((cpc + (pl.warps - 1) * 32 - 1) / ((pl.warps - 1) * 32) * 32);
  pl.smem = pn_smem(cl, pl.warps, pl.wch, pl.lc);
  return pl.smem <= limit && (pl.warps - 1) * pl.wch <= 65536;
}

cudaLaunchConfig_t config(const NPlan& pl, int nprob, cudaLaunchAttribute* attr, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)pl.cl;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(nprob * pl.cl), 1, 1);
  cfg.blockDim = dim3((unsigned)(32 * pl.warps), 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// Cluster size.  One problem: latency counts, so a CTA gets few coordinates
// (the FP64 pipe is the narrowest: 64 per CTA where all of them take FP64,
// else 224, one per lane), on up to 16 CTAs (measured when the kernel came in, at 1000 x 1000 FP32:
// 1 / 2 / 4 / 8 / 16 CTAs 50 / 41 / 38 / 31 / 34 us; p = 20000: 4 / 8 / 16 CTAs
// 110 / 76 / 59 us).  Many problems: about two CTAs per SM, but four per
// problem where the sizes allow (256 problems of p = 10000, whole call: 1 / 2 /
// 4 / 8 CTAs 62.8 / 63.1 / 60.7 / 63.7 ms; 48 of p = 5000: 2 / 4 / 8 CTAs 7.59 /
// 6.97 / 7.62 ms).  A CTA's coordinates must fit its shared memory either way.
cudaError_t pnode_plan(NPlan& pl, int kind, int64_t p, int nprob) {
  pl = NPlan{};
  pl.kernel = kind == PK_F64      ? reinterpret_cast<const void*>(&pnode_kernel<PK_F64>)
              : kind == PK_PAIR64 ? reinterpret_cast<const void*>(&pnode_kernel<PK_PAIR64>)
                                  : reinterpret_cast<const void*>(&pnode_kernel<PK_PAIR>);
  if (p < 1 || nprob < 1) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t target = kind == PK_F64 ? 64 : 224;
  int share = 4;
  while (share < PN_MAXCL && 2 * share * nprob <= 2 * nsm) share *= 2;
  const int64_t want = std::min<int64_t>((p + target - 1) / target, share);
  int cl = 1;
  while (cl < want) cl *= 2;
  cudaError_t e;
  for (; cl <= PN_MAXCL; cl *= 2) {
    if (!sized(pl, p, cl, (size_t)optin)) continue;
    if (cl > 8 && (e = cudaFuncSetAttribute(pl.kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
      return e;
    if ((e = raise_smem(pl.kernel, pl.smem)) != cudaSuccess) return e;
    if (cl <= 8) return cudaSuccess;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = config(pl, 1, attr, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, pl.kernel, &cfg) == cudaSuccess && n >= 1) return cudaSuccess;
    (void)cudaGetLastError();
    // no 16 SMs to place one: the largest portable size, if the share fits it
    if (sized(pl, p, 8, (size_t)optin)) return raise_smem(pl.kernel, pl.smem);
  }
  return cudaErrorNotSupported;
}

cudaError_t pnode_launch(const NPlan& pl, NArgs a, int nprob, cudaStream_t st) {
  if (!pl.kernel || nprob < 1) return cudaErrorInvalidValue;
  a.cl = pl.cl;
  a.cpc = pl.cpc;
  a.lc = pl.lc;
  a.wch = pl.wch;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = config(pl, nprob, attr, st);
  void* args[1] = {(void*)&a};
  return cudaLaunchKernelExC(&cfg, pl.kernel, args);
}

}  // namespace relax
