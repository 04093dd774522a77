// Shell-quartet kernel with runtime angular momenta, one CTA per quartet (paper
// Sec. 2.3.4 Eq. twoe-final, Sec. 2.5 Eq. eri-tensor-contracted; J/K digestion
// Eq. fock): every class pair that contains an f shell, and the FP64 class
// pairs whose arrays outgrow one thread (gen64_default).  Same mathematics and
// conventions as eri_core.cuh (pair data with the contraction coefficients,
// Cartesian normalisation and sqrt(2) pi^{5/4}/p folded into E; degeneracy-
// weighted accumulators symmetrised by the caller).
//
// Layout of the work, for groups of nbg bra primitive pairs at a time:
//   1. thread p owns the p-th of the group's primitive quartets that can matter
//      (prim_mask): Boys function, sources, then the whole in-place R recursion in
//      its own column of a shared-memory array R[h][p] (Eq. R-recursion from a
//      table of parents; no barrier);
//   2. W[b][c][h] = sum_k sum_{h' in nz(c)} (-1)^{|h'|} E^{cd,k}_{c,h'} R[h + h'],
//      elements over all threads with h fastest, so a warp shares c (and with
//      it E, a broadcast) and the row of the sum table h + h';
//   3. out[a][c] += sum_b sum_{h in nz(a)} E^{ab,b}_{a,h} W[b][c][h];
// and per quartet the digestion: each thread sums one element of the J/K
// blocks over the quartet block and adds it with one FP64 atomic.
// Four barriers per group and two per quartet, none per primitive quartet or
// recursion level.  An FP64 launch with fewer quartets than resident CTAs shares each quartet's bra
// primitive pairs out over several CTAs, which digest their partial blocks
// (six (dd|dd) quartets: 0.77 ms with one CTA each).
//
// Why this shape: GB300 issues two FP64 FMAs per clock and SM, so one DFMA
// leaves its scheduler 64 issue slots, and what counts in FP64 is the number
// of FP64 instructions, not the loads and index arithmetic around them.
// Operands come from shared memory by table, every Boys function and R is
// evaluated once, and no thread holds a quartet-sized array.  The unrolled
// kernel of eri_core.cuh repeats R for every ket chunk and, at one warp per
// scheduler, waits on its local-memory arrays: it used 50-65 % of the FP64 pipe.
// 64 registers a thread let a fourth CTA onto the SM where its shared memory fits,
// to fill the others' barriers ((H2O)_8 FP64 build -1.7 %, (H2O)_3 with f shells -7 %);
// groups cut down so that four always fit gain nothing more (+0.8, +1 %).  On a
// 7-atom cloud it uses 78-91 % of the FP64 pipe.
#pragma once
#include "eri_core.cuh"

namespace fsim {

constexpr int kGenThreads = 256;
constexpr int kGenMaxL = 12;     // (ff|ff)
constexpr int kGenMaxH1 = nherm(6);  // Hermite terms of an (f f) pair
constexpr int kGenMaxNC = 100;       // components of an (f f) pair
constexpr unsigned kGenMaxSmem = 226 * 1024;  // no layout is larger

// Shared-memory layout of a class pair (byte offsets).
struct GenLayout {
  int nbg, nkg;         // bra and ket primitive pairs per group (all of the ket's, but for the largest classes)
  int npad;             // row length of R: nbg * nkg, odd against bank conflicts
  int stage_k, stage_b; // E of the ket / bra pair staged in shared memory
  unsigned R, W, out, Ek, Eb, coef, col, par, sum, nzc, nza, offc, offa, bytes;
};

template <typename Real>
struct GenParams {
  PairView<Real> bra, ket;
  int la, lb, lc, ld;
  int same;                          // bra class == ket class
  int list_mode;
  const int* __restrict__ prefix;    // JK mode: [nbra + 1] cumulative screened kets per bra
  const int2* __restrict__ items;    // list mode: (bra, ket) pair indices
  int nitems;                        // quartets (JK mode) or items (list mode)
  int nsplit;                        // CTAs a quartet's bra primitive pairs are shared out over (set by launch_gen)
  double* out;                       // list mode: block of item q at out + q * NA*NB * NC*ND
  int N;
  const Real* __restrict__ D;
  double* J;
  double* K;
  const Real* __restrict__ boys;     // full table, rows of kBoysCols
  float boys64_T;
  int prim_lt;                       // log2 of the build's primitive-quartet threshold (prim_theta)
  GenLayout lay;                     // filled by launch_gen
};

inline int gen_pair_nnz(int la, int lb) { return pair_cls_nnz(pair_cls_index(la, lb)); }

// nbg: the fewest warps over all groups in step 1, then the largest group, that
// keeps three CTAs on an SM (or the smallest group where even that does not fit).
template <typename Real>
GenLayout gen_layout(int la, int lb, int lc, int ld, int ppb, int ppk) {
  const int L = la + lb + lc + ld, H1 = nherm(la + lb), H2 = nherm(lc + ld), NH = nherm(L);
  const int A = ncart(la) * ncart(lb), C = ncart(lc) * ncart(ld);
  const int za = gen_pair_nnz(la, lb), zc = gen_pair_nnz(lc, ld);
  constexpr unsigned kThree = 74 * 1024, kStage = 16 * 1024;
  int nkg = ppk;
  auto make = [&](int nbg) {
    GenLayout y{};
    y.nbg = nbg;
    y.nkg = nkg;
    y.npad = (nbg * nkg) | 1;
    y.stage_k = (size_t)zc * ppk * sizeof(Real) <= kStage;
    y.stage_b = (size_t)za * ppb * sizeof(Real) <= kStage;
    unsigned o = 0;
    auto take = [&](size_t n) {
      const unsigned at = o;
      o += (unsigned)((n + 15) / 16 * 16);
      return at;
    };
    y.R = take((size_t)NH * y.npad * sizeof(Real));
    y.W = take((size_t)nbg * C * H1 * sizeof(Real));
    y.out = take((size_t)A * C * sizeof(Real));
    y.Ek = take(y.stage_k ? (size_t)zc * ppk * sizeof(Real) : 0);
    y.Eb = take(y.stage_b ? (size_t)za * ppb * sizeof(Real) : 0);
    y.coef = take(16 * sizeof(Real));
    y.col = take((size_t)(nbg * nkg + 16 + 8 + 1) * sizeof(int));
    y.par = take((size_t)NH * sizeof(int));
    y.sum = take((size_t)H1 * H2 * sizeof(short));
    y.nzc = take((size_t)zc * sizeof(short));
    y.nza = take((size_t)za * sizeof(short));
    y.offc = take((size_t)(C + 1) * sizeof(short));
    y.offa = take((size_t)(A + 1) * sizeof(short));
    y.bytes = o;
    return y;
  };
  GenLayout best = make(1);
  while (best.bytes > kGenMaxSmem && nkg > 1) {
    nkg = (nkg + 1) / 2;
    best = make(1);
  }
  int best_warps = 1 << 30;
  for (int nbg = 1; nbg <= ppb && nbg * nkg <= kGenThreads / 2; ++nbg) {
    const GenLayout y = make(nbg);
    if (y.bytes > kThree) break;
    int warps = 0;
    for (int b = 0; b < ppb; b += nbg) warps += ((b + nbg < ppb ? nbg : ppb - b) * nkg + 31) / 32;
    if (warps <= best_warps) {
      best_warps = warps;
      best = y;
    }
  }
  return best;
}

}  // namespace fsim
