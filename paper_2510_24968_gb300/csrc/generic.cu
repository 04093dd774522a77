// The runtime-angular-momentum quartet kernel (described in generic.cuh), used
// for every class pair that contains an f shell, in FP32 and FP64, and for the
// heavy FP64 class pairs of s, p and d shells.
#include <algorithm>

#include "fsim_internal.h"
#include "generic.cuh"

namespace fsim {

// F_0..F_L from the full table in global memory, at T (FP64: at u = -2T)
template <typename Real, int L>
__device__ __forceinline__ void gen_boys_to(Real T, Real* F, const Real* tab, float t64) {
  Real f[L + 1];
  if constexpr (std::is_same<Real, double>::value) boys_fp64_u<L, false>(T, f, tab + L, kBoysCols, kBoysCols - 1 - L);
  else Boys<Real>::template eval<L>(T, f, tab + L, kBoysCols, t64);
#pragma unroll
  for (int n = 0; n <= L; ++n) F[n] = f[n];
}

template <typename Real>
__device__ void gen_boys(int L, Real T, Real* F, const Real* tab, float t64) {
  switch (L) {
    case 0: gen_boys_to<Real, 0>(T, F, tab, t64); break;
    case 1: gen_boys_to<Real, 1>(T, F, tab, t64); break;
    case 2: gen_boys_to<Real, 2>(T, F, tab, t64); break;
    case 3: gen_boys_to<Real, 3>(T, F, tab, t64); break;
    case 4: gen_boys_to<Real, 4>(T, F, tab, t64); break;
    case 5: gen_boys_to<Real, 5>(T, F, tab, t64); break;
    case 6: gen_boys_to<Real, 6>(T, F, tab, t64); break;
    case 7: gen_boys_to<Real, 7>(T, F, tab, t64); break;
    case 8: gen_boys_to<Real, 8>(T, F, tab, t64); break;
    case 9: gen_boys_to<Real, 9>(T, F, tab, t64); break;
    case 10: gen_boys_to<Real, 10>(T, F, tab, t64); break;
    case 11: gen_boys_to<Real, 11>(T, F, tab, t64); break;
    default: gen_boys_to<Real, 12>(T, F, tab, t64); break;
  }
}

// Index tables of every pair class, constants of the program: a CTA copies the
// parts of its class pair into shared memory.  (Built by each CTA, they cost
// more than a small launch's quartets.)
struct GenTables {
  int par[nherm(kGenMaxL)];  // R recursion: first parent | second << 10 | axis << 20 | coefficient << 22
  short sum[kGenMaxH1][kGenMaxH1];               // [h'][h]: index of h + h'
  short off[kNumPairClsAll][kGenMaxNC + 1];      // first non-zero of each component; [NC]: their number
  short nz[kNumPairClsAll][pair_cls_nnz(kNumPairClsAll - 1)];  // Hermite index | parity << 14
};

constexpr GenTables make_gen_tables() {
  GenTables T{};
  int t[nherm(kGenMaxL)] = {}, u[nherm(kGenMaxL)] = {}, v[nherm(kGenMaxL)] = {};
  for (int n = 0, h = 0; n <= kGenMaxL; ++n)
    for (int m = 0; m <= n; ++m)
      for (int w = 0; w <= m; ++w, ++h) {
        t[h] = n - m;
        u[h] = m - w;
        v[h] = w;
      }
  for (int h = 1; h < nherm(kGenMaxL); ++h) {
    const int ax = t[h] > 0 ? 0 : (u[h] > 0 ? 1 : 2);
    const int dt = ax == 0, du = ax == 1, dv = ax == 2;
    const int cf = (ax == 0 ? t[h] : (ax == 1 ? u[h] : v[h])) - 1;
    const int p1 = hidx(t[h] - dt, u[h] - du, v[h] - dv);
    const int p2 = cf > 0 ? hidx(t[h] - 2 * dt, u[h] - 2 * du, v[h] - 2 * dv) : p1;
    T.par[h] = p1 | (p2 << 10) | (ax << 20) | (cf << 22);
  }
  for (int a = 0; a < kGenMaxH1; ++a)
    for (int b = 0; b < kGenMaxH1; ++b) T.sum[a][b] = (short)hidx(t[a] + t[b], u[a] + u[b], v[a] + v[b]);
  for (int c = 0; c < kNumPairClsAll; ++c) {
    const int la = pair_cls_la(c), lb = pair_cls_lb(c), nc = ncart(la) * ncart(lb);
    int k = 0;
    for (int a = 0; a < nc; ++a) {
      int e[3] = {};
      for (int x = 0; x < 3; ++x) e[x] = cart_comp(la, a / ncart(lb), x) + cart_comp(lb, a % ncart(lb), x);
      T.off[c][a] = (short)k;
      for (int i = 0; i <= e[0]; ++i)
        for (int j = 0; j <= e[1]; ++j)
          for (int w = 0; w <= e[2]; ++w, ++k) T.nz[c][k] = (short)(hidx(i, j, w) | (((i + j + w) & 1) << 14));
    }
    T.off[c][nc] = (short)k;
  }
  return T;
}
__device__ const GenTables kGenTables = make_gen_tables();

template <typename Real>
__global__ void __launch_bounds__(kGenThreads, 4) gen_kernel(GenParams<Real> P) {
  extern __shared__ __align__(16) unsigned char gen_smem[];
  const GenLayout& Y = P.lay;
  const int la = P.la, lb = P.lb, lc = P.lc, ld = P.ld;
  const int NB = ncart(lb), NDc = ncart(ld), NA = ncart(la), NCc = ncart(lc);
  const int A = NA * NB, C = NCc * NDc;
  const int L = la + lb + lc + ld;
  const int NH = nherm(L), H1 = nherm(la + lb), H2 = nherm(lc + ld);
  Real* sR = reinterpret_cast<Real*>(gen_smem + Y.R);      // [h][p]
  Real* sW = reinterpret_cast<Real*>(gen_smem + Y.W);      // [b][c][h]
  Real* sOut = reinterpret_cast<Real*>(gen_smem + Y.out);  // [a][c]
  Real* sEk = reinterpret_cast<Real*>(gen_smem + Y.Ek);    // [nz][k], signed
  Real* sEb = reinterpret_cast<Real*>(gen_smem + Y.Eb);    // [nz][b]
  Real* sCoef = reinterpret_cast<Real*>(gen_smem + Y.coef);
  int* sCol = reinterpret_cast<int*>(gen_smem + Y.col);    // [p]: bra << 8 | ket primitive pair
  int* sBeg = sCol + Y.nbg * Y.nkg;                        // [b]: first p of bra primitive pair b of the group
  int* sCnt = sBeg + 17;                                   // kept primitive quartets of each warp
  int* sPar = reinterpret_cast<int*>(gen_smem + Y.par);    // first parent | second << 10 | axis << 20 | coefficient << 22
  short* sSum = reinterpret_cast<short*>(gen_smem + Y.sum);  // [h'][h]: index of h + h'
  short* sNzc = reinterpret_cast<short*>(gen_smem + Y.nzc);  // h' | parity << 14
  short* sNza = reinterpret_cast<short*>(gen_smem + Y.nza);
  short* sOffc = reinterpret_cast<short*>(gen_smem + Y.offc);
  short* sOffa = reinterpret_cast<short*>(gen_smem + Y.offa);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int cb = pair_cls_index(la, lb), ck = pair_cls_index(lc, ld);
  for (int h = tid; h < NH; h += nth) sPar[h] = kGenTables.par[h];
  for (int x = tid; x < H1 * H2; x += nth) sSum[x] = kGenTables.sum[x / H1][x % H1];
  for (int a = tid; a <= A; a += nth) sOffa[a] = kGenTables.off[cb][a];
  for (int c = tid; c <= C; c += nth) sOffc[c] = kGenTables.off[ck][c];
  const int zA = kGenTables.off[cb][A], zC = kGenTables.off[ck][C];
  for (int z = tid; z < zA; z += nth) sNza[z] = kGenTables.nz[cb][z];
  for (int z = tid; z < zC; z += nth) sNzc[z] = kGenTables.nz[ck][z];
  if (tid < 16) sCoef[tid] = Real(tid);
  __syncthreads();
  const size_t bstride = (size_t)P.bra.ppmax * P.bra.n, kstride = (size_t)P.ket.ppmax * P.ket.n;
  for (ItemLoop at(blockIdx.x, gridDim.x, P.nitems * P.nsplit); at.more(); at.next()) {
    const int q = (int)at.i / P.nsplit, share = (int)at.i - q * P.nsplit;
    int i, j;
    if (P.list_mode) {
      const int2 it = P.items[q];
      i = it.x;
      j = it.y;
    } else {
      i = find_bra(P.prefix, P.bra.n, q);
      j = q - __ldg(P.prefix + i);
    }
    const int nppb = P.bra.npp[i], nppk = P.ket.npp[j];
    const int b_lo = share * nppb / P.nsplit, b_hi = (share + 1) * nppb / P.nsplit;  // this CTA's bra primitive pairs
    if (b_lo == b_hi) continue;
    const int prim_lt = P.prim_lt == kPrimKeepAll  // (the bounds themselves are made so, before Q exists)
                            ? kPrimKeepAll
                            : prim_theta<Real>(P.prim_lt, bound_word(P.bra.Q, i), bound_word(P.ket.Q, j));
    const Real* bp = P.bra.pd + i;
    const Real* kp = P.ket.pd + j;
    const int4 bi = P.bra.idx[i], ki = P.ket.idx[j];
    const Real deg = P.list_mode
                         ? Real(1)
                         : Real((bi.z == bi.w ? 1 : 2) * (ki.z == ki.w ? 1 : 2) * ((P.same && i == j) ? 1 : 2));
    if (Y.stage_k)
      for (int x = tid; x < zC * nppk; x += nth) {
        const int z = x / nppk, k = x - z * nppk;
        const Real e = ldg_r(kp + (size_t)(4 + z) * kstride + (size_t)k * P.ket.n);
        sEk[x] = (sNzc[z] & 0x4000) ? -e : e;
      }
    if (Y.stage_b)
      for (int x = tid; x < zA * nppb; x += nth) {
        const int z = x / nppb, b = x - z * nppb;
        sEb[x] = ldg_r(bp + (size_t)(4 + z) * bstride + (size_t)b * P.bra.n);
      }
    for (int b0 = b_lo; b0 < b_hi; b0 += Y.nbg) {
      const int nb = min(Y.nbg, b_hi - b0);
      for (int k0 = 0; k0 < nppk; k0 += Y.nkg) {
        const int nk = min(Y.nkg, nppk - k0);
        // the primitive quartets to evaluate, in order
        int np;
        {
          const int b = tid / nk, k = k0 + tid % nk;
          bool keep = false;
          if (tid < nb * nk)
            keep = prim_lt == kPrimKeepAll || prim_byte(P.ket.ub + j, k) >= prim_least(prim_lt, prim_byte(P.bra.ub + i, b0 + b));
          const unsigned bal = __ballot_sync(0xffffffffu, keep);
          if ((tid & 31) == 0) sCnt[tid >> 5] = __popc(bal);
          __syncthreads();  // (also: the previous step's columns have been read)
          int p = __popc(bal & ((1u << (tid & 31)) - 1u));
          np = 0;
          for (int w = 0; w < nth / 32; ++w) {
            if (w < tid >> 5) p += sCnt[w];
            np += sCnt[w];
          }
          if (tid < nb * nk) {
            if (keep) sCol[p] = b << 8 | k;
            if (tid % nk == 0) sBeg[b] = p;
          }
          if (tid == 0) sBeg[nb] = np;
          __syncthreads();
        }
        // 1. one primitive quartet per thread: sources and the in-place recursion
        if (tid < np) {
          const int b = b0 + (sCol[tid] >> 8), k = sCol[tid] & 255;
          const auto p4 = P.bra.pq[(size_t)b * P.bra.n + i];
          const Real p = p4.x, Px = p4.y, Py = p4.z, Pz = p4.w;
          const auto q4 = P.ket.pq[(size_t)k * P.ket.n + j];
          const Real qq = q4.x;
          const Real s = p + qq;
          const Real X = Px - q4.y, Yy = Py - q4.z, Z = Pz - q4.w;
          Real F[kGenMaxL + 1], fac, m2a;
          if constexpr (std::is_same<Real, double>::value) {
            fac = rsqrt_fp64(s);
            m2a = -2.0 * p * qq * (fac * fac);
            gen_boys<Real>(L, m2a * (X * X + Yy * Yy + Z * Z), F, P.boys, P.boys64_T);
          } else {
            fac = rsqrt_r<Real>(s);
            const Real al = p * qq * (fac * fac);
            gen_boys<Real>(L, al * (X * X + Yy * Yy + Z * Z), F, P.boys, P.boys64_T);
            m2a = Real(-2) * al;
          }
          for (int n = 0; n <= L; ++n) {
            F[n] = fac * F[n];
            fac *= m2a;
          }
          Real* R = sR + tid;
          R[0] = F[L];
          for (int n = L - 1; n >= 0; --n) {
            // level n from level n + 1, higher orders first: order s reads s - 1 and s - 2 only
            for (int o = L - n; o >= 1; --o) {
              const int hi = nherm(o);
              for (int h = nherm(o - 1); h < hi; h += 4) {
                int w[4];
                Real c1[4], c2[4];
  #pragma unroll
                for (int x = 0; x < 4; ++x) {
                  w[x] = sPar[min(h + x, hi - 1)];
                  c1[x] = R[(w[x] & 1023) * Y.npad];
                  c2[x] = R[((w[x] >> 10) & 1023) * Y.npad];
                }
  #pragma unroll
                for (int x = 0; x < 4; ++x) {
                  const int ax = (w[x] >> 20) & 3, cf = w[x] >> 22;
                  const Real a = ax == 0 ? X : (ax == 1 ? Yy : Z);
                  Real r;  // the branch is uniform: every thread is at the same h
                  if (h + x >= hi) break;
                  if (cf == 0) r = a * c1[x];
                  else if (cf == 1) r = fma(a, c1[x], c2[x]);
                  else r = fma(a, c1[x], sCoef[cf] * c2[x]);
                  R[(h + x) * Y.npad] = r;
                }
              }
            }
            R[0] = F[n];
          }
        }
        __syncthreads();
        // 2. ket transform
        const int nW = C * nb * H1;
        for (int x = tid; x < nW; x += nth) {
          const int bh = x / H1, h = x - bh * H1, c = bh / nb, b = bh - c * nb;
          const int p0 = sBeg[b], p1 = sBeg[b + 1];
          const short* sum = sSum + h;
          const int z0 = sOffc[c], z1 = sOffc[c + 1];
          Real& Wx = sW[(b * C + c) * H1 + h];
          Real acc = k0 == 0 ? Real(0) : Wx;
          if constexpr (std::is_same<Real, float>::value) {
            for (int p = p0; p < p1; ++p) {
              const int k = sCol[p] & 255;
              Real part = Real(0);
              for (int z = z0; z < z1; ++z) {
                const int w = sNzc[z], hz = w & 0x3fff;
                Real e;
                if (Y.stage_k) {
                  e = sEk[z * nppk + k];
                } else {
                  e = ldg_r(kp + (size_t)(4 + z) * kstride + (size_t)k * P.ket.n);
                  e = (w & 0x4000) ? -e : e;
                }
                part = fma(e, sR[sum[hz * H1] * Y.npad + p], part);
              }
              acc += part;
            }
          } else {
            for (int z = z0; z < z1; ++z) {
              const int w = sNzc[z], hz = w & 0x3fff;
              const Real* Rz = sR + sum[hz * H1] * Y.npad;
              if (Y.stage_k && np == nb * nk) {  // nothing left out: no list to follow
                const Real* E = sEk + z * nppk + k0 - p0;
  #pragma unroll 3
                for (int p = p0; p < p1; ++p) acc = fma(E[p], Rz[p], acc);
              } else if (Y.stage_k) {
                const Real* E = sEk + z * nppk;
  #pragma unroll 3
                for (int p = p0; p < p1; ++p) acc = fma(E[sCol[p] & 255], Rz[p], acc);
              } else {
                const Real* E = kp + (size_t)(4 + z) * kstride;
                const Real sg = (w & 0x4000) ? Real(-1) : Real(1);
                Real part = Real(0);
  #pragma unroll 3
                for (int p = p0; p < p1; ++p) part = fma(ldg_r(E + (size_t)(sCol[p] & 255) * P.ket.n), Rz[p], part);
                acc = fma(sg, part, acc);
              }
            }
          }
          Wx = acc;
        }
        __syncthreads();
      }
      // 3. bra transform into the block (the next group's step 1 only writes R)
      for (int x = tid; x < A * C; x += nth) {
        const int a = x / C, c = x - a * C;
        const int z0 = sOffa[a], z1 = sOffa[a + 1];
        Real tot = b0 == b_lo ? Real(0) : sOut[x];
        for (int b = 0; b < nb; ++b) {
          const Real* W = sW + (b * C + c) * H1;
          Real acc = Real(0);
          for (int z = z0; z < z1; ++z) {
            const Real e = Y.stage_b ? sEb[z * nppb + b0 + b]
                                     : ldg_r(bp + (size_t)(4 + z) * bstride + (size_t)(b0 + b) * P.bra.n);
            acc = fma(e, W[sNza[z] & 0x3fff], acc);
          }
          tot += acc;
        }
        sOut[x] = b0 + nb == b_hi ? deg * tot : tot;
      }
    }
    __syncthreads();
    if (P.list_mode) {
      double* o = P.out + (size_t)q * A * C;
      for (int x = tid; x < A * C; x += nth) o[x] = (double)sOut[x];
    } else {
      const int N = P.N;
      const int oJk = A, oK1 = oJk + C, oK2 = oK1 + NA * NCc, oK3 = oK2 + NA * NDc, oK4 = oK3 + NB * NCc,
                nout = oK4 + NB * NDc;
      // element (row, col) of J or K: sum over n0 x n1 block elements of D(r0 + x0, r1 + x1) v
      for (int x = tid; x < nout; x += nth) {
        int row, col, r0, r1, n0, n1, at, s0, s1;  // block index of (x0, x1): at + x0 s0 + x1 s1
        if (x < oJk) {  // J_bra[a] += D_{la si} v
          row = bi.x + x / NB; col = bi.y + x % NB;
          r0 = ki.x; r1 = ki.y; n0 = NCc; n1 = NDc;
          at = x * C; s0 = NDc; s1 = 1;
        } else if (x < oK1) {  // J_ket[c] += D_{mu nu} v
          const int c = x - oJk;
          row = ki.x + c / NDc; col = ki.y + c % NDc;
          r0 = bi.x; r1 = bi.y; n0 = NA; n1 = NB;
          at = c; s0 = NB * C; s1 = C;
        } else if (x < oK2) {  // K(mu la) += D_{nu si} v
          const int y = x - oK1, m = y / NCc, l = y % NCc;
          row = bi.x + m; col = ki.x + l;
          r0 = bi.y; r1 = ki.y; n0 = NB; n1 = NDc;
          at = m * NB * C + l * NDc; s0 = C; s1 = 1;
        } else if (x < oK3) {  // K(mu si) += D_{nu la} v
          const int y = x - oK2, m = y / NDc, l = y % NDc;
          row = bi.x + m; col = ki.y + l;
          r0 = bi.y; r1 = ki.x; n0 = NB; n1 = NCc;
          at = m * NB * C + l; s0 = C; s1 = NDc;
        } else if (x < oK4) {  // K(nu la) += D_{mu si} v
          const int y = x - oK3, m = y / NCc, l = y % NCc;
          row = bi.y + m; col = ki.x + l;
          r0 = bi.x; r1 = ki.y; n0 = NA; n1 = NDc;
          at = m * C + l * NDc; s0 = NB * C; s1 = 1;
        } else {  // K(nu si) += D_{mu la} v
          const int y = x - oK4, m = y / NDc, l = y % NDc;
          row = bi.y + m; col = ki.y + l;
          r0 = bi.x; r1 = ki.x; n0 = NA; n1 = NCc;
          at = m * C + l; s0 = NB * C; s1 = NDc;
        }
        double acc = 0.0;
        for (int x0 = 0; x0 < n0; ++x0) {
          const Real* Dr = P.D + (size_t)(r0 + x0) * N + r1;
          for (int x1 = 0; x1 < n1; ++x1) {
            const Real v = sOut[at + x0 * s0 + x1 * s1];
            if constexpr (std::is_same<Real, float>::value) acc += (double)(Dr[x1] * v);
            else acc = fma(Dr[x1], v, acc);
          }
        }
        atomicAdd((x < oK1 ? P.J : P.K) + (size_t)row * N + col, acc);
      }
    }
    __syncthreads();  // block and E read before the next quartet overwrites them
  }
}

template <typename Real>
cudaError_t launch_gen(const GenParams<Real>& in, cudaStream_t s) {
  auto k = gen_kernel<Real>;
  GenParams<Real> p = in;
  p.lay = gen_layout<Real>(p.la, p.lb, p.lc, p.ld, p.bra.ppmax, p.ket.ppmax);
  const size_t smem = p.lay.bytes;
  // one kernel for every class pair and the limit is the process's: always the
  // largest layout, so that no other thread's launch can lower it in between
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGenMaxSmem);
  if (e != cudaSuccess || p.nitems == 0) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kGenThreads, smem);
  if (e != cudaSuccess) return e;
  const int slots = std::max(1, occ) * device_sm_count();
  p.nsplit = 1;
  if (std::is_same<Real, double>::value && !p.list_mode && p.nitems < slots) {
    // as many shares as fill the device, evened out (9 pairs: 9, 5, 3 or 2 CTAs)
    const int per = (p.bra.ppmax + slots / p.nitems - 1) / (slots / p.nitems);
    p.nsplit = (p.bra.ppmax + per - 1) / per;
  }
  const int grid = std::min(p.nitems * p.nsplit, slots);
  k<<<grid, kGenThreads, smem, s>>>(p);
  return cudaGetLastError();
}

template cudaError_t launch_gen<float>(const GenParams<float>&, cudaStream_t);
template cudaError_t launch_gen<double>(const GenParams<double>&, cudaStream_t);

}  // namespace fsim
