// Node p-phase: everything an iteration does on p-vectors (the steps P0, S1,
// S2, D, P1, S3, P2 of pphase.cuh), the certificate's evaluation of Phi and Psi,
// or a standalone prox, g or g*, by one thread-block cluster per problem.
//
// What bounds it is latency: the arithmetic is a few microseconds' worth of
// one cluster, and every grid-wide sum of the iteration is a round trip
// between its CTAs.  So the work is arranged around as few exchanges as the
// dependences allow, two in a usual iteration:
//  * stage 1, local: G^t (sum of the pass's partials), the keys |a_j|, the
//    sums of Phi and Psi, g's classification at the known water level, and v
//    at the momentum of "no restart" (known from the last iteration);
//  * exchange 1: those sums, and for 32 candidate thresholds around the
//    predicted ones the counts that bracket the kbar-th largest |a_j| (S1)
//    and the counts and sums that bracket the prox threshold c (S3);
//  * stage 2, local: exact sums over the coordinates beyond the brackets, the
//    few inside collected into lists;
//  * exchange 2: those sums and lists.  Every CTA then finishes both searches
//    on the sorted lists by itself and takes the loop's decisions; one that
//    turns out to restart forms v again (momentum 0) and repeats S3.
// An exchange pushes each CTA's words into every CTA's shared memory
// (distributed shared memory) ahead of one hardware cluster barrier, so its
// latency is one way; sums run over the CTAs in rank order (deterministic).
//
// FP64 arithmetic, comparisons and conversions issue at about 1.6 lanes per
// clock per SM here (FP32: about 112), so on FP32 data (PK_PAIR) the
// coordinates with beta^t_j = beta^{t-1}_j = 0 that are not fixed in take FP32
// arithmetic only, gradients travel as FP32 pairs (hi + lo) and sums are
// float-float; the others ("wide") are collected per warp and take FP64 with
// full warps.  (A dependent FP64 operation takes 64 cycles here, a division
// about 580: thread 0 decides while the other warps write the next point.)
// PK_F64 (FP64 data, the last rungs of the precision ladder): every coordinate is
// wide and sums are FP64.  PK_PAIR64 (FP32 data: the certificate, the standalone
// operations): FP32 per coordinate, FP64 sums.
//
// Measured per iteration, against the cooperative grid of pphase.cuh that ran
// before (seven or more grid barriers): p = 1000 45 -> 29 us, p = 4000
// (logistic) 53 -> 39 us, p = 20000 81 -> 44 us, p = 50000 85 -> 58 us (47 over a
// solve of 577 iterations), FP64 p = 1000 66 -> 32 us; whole calls at this step:
// 256 nodes of 5000 x 10000 110 -> 61 ms (with the certificates evaluated
// together), 48 of 2000 x 5000 14.5 -> 7.0 ms.
#pragma once
#include "bgemm.cuh"
#include "pphase.cuh"

namespace relax {

// the kernel's instantiations: FP32 data with float-float sums (the loop), FP64,
// FP32 data with FP64 sums (the certificate, the standalone operations)
enum PNKind : int { PK_PAIR = 0, PK_F64 = 1, PK_PAIR64 = 2 };

constexpr int PN_MAXW = 16;          // warps per CTA at most (warp 0 takes the decisions, the others coordinates)
constexpr int PN_MAXCL = 16;         // CTAs per cluster at most (16: a non-portable size)
constexpr int PN_CAP = 256;          // bracket entries finished in place, per search
constexpr int PN_TILES = 128;        // product tiles (of BG_BM coordinates) a CTA's coordinates meet at most
constexpr int PN_LSUM = 4;           // doubles per CTA of the pass's loss sums: F, dual term, second dual term, -

// exchange words: [0, 32) S3 sums per candidate (float-float), then the sums
// of Phi and Psi, then counts (packed pairs of 32-bit ones)
enum : int { XW_S3 = 0, XW_SUM = 32, XW_N3 = 38, XW_N1 = 70, XW_INT = 102, XW_WORDS = 106 };
enum : int { XS_J1H = 0, XS_J1B2 = 1, XS_B = 2, XS_B2 = 3, XS_SAB = 4, XS_QAB = 5, XS_NSUM = 6 };

struct NArgs {
  PConst kc;
  int mode;                     // PMode
  int loss, cl, cpc;            // CTAs per problem, coordinates per CTA
  int lc, wch;                  // list entries per CTA and search; coordinates per warp
  int64_t p, n;
  int k;
  double lambda2, M, step, rho, eta;
  int max_iters, stall_min, method, restart_rule;
  const int8_t* fix;            // NULL = root; row fix_stride per problem
  int64_t fix_stride;
  // gradient partials [ncl][NB][p] per problem, as FP32 pairs (float2) or FP64
  const void* part;
  int64_t part_stride;
  int ncl, NB, gpair;
  // batched FP32 products instead: FP32 partial tiles [slot][NB m][p]
  const float* tiles;
  BGSplit s2;
  int m;
  // PM_ITER: state, problem s is node seg_node[s] (NULL: s)
  IterState* st;
  const int* seg_node;
  const double* lsum;           // [nl][PN_LSUM] loss sums per problem
  int nl;
  int64_t lsum_stride;
  void* zero;                   // PM_ITER: cleared for the next pass (16-byte multiple), or NULL
  int64_t zero_bytes;
  __nv_bfloat16* Bp;            // batched FP32 products: planes of the next point, row = problem
  int64_t ldp, bplane;
  // PM_EVAL: problem s is the dual point s % nq of item s / nq (part offset
  // by s % nq right-hand sides); beta = ev[item].beta
  const PassState* ev;
  int nq;
  void* gev;                    // [problem][p] scratch: the summed gradients (8 bytes each)
  const int* cnt;               // [items][3] fixing counts {|J1|, |Jf|, .}; NULL: root
  double* out;                  // item's values at out_stride item + 2 (s % nq); PM_GVAL, PM_GSTAR: one value
  int64_t out_stride;
  // the standalone operations, one problem, FP64 vectors (PK_F64) or FP32 ones
  // (PK_PAIR64: their sums and products need FP64's range and precision too)
  const void* vin;              // PM_PROX: v, PM_GVAL: beta, PM_GSTAR: alpha
  void* vout;                   // PM_PROX
  int* counts;                  // PM_PROX: {n_top, n_nz} or NULL
  int* status;
};

}  // namespace relax
