/*
 * dg_element.cu -- the float64 element kernel of one stage (k_element_sf): the
 * volume integral (Eq. volume, Algorithm 1) sum-factorised on the collapsed
 * volume grid (or contracted directly on a symmetric rule of Q points), the lift
 * of the three edge fluxes (Algorithms 2-3), the 1/det J
 * scaling (Eq. 2ddg0), the Runge-Kutta stage update (with, for the classical
 * RK4, the running sum of its stages as a second output) and the next stage's
 * edge traces, for one tile of elements per CTA; and the fused stepper of small
 * meshes (k_rk_small), whose phases are this kernel's.  Larger meshes take
 * k_element_split (dg_split.cuh).
 */
#include <cuda_runtime.h>

#include <cstdint>

#include "dg_device.cuh"
#include "dg_internal.h"
#include "dg_limiter.cuh"

namespace dg {
namespace {

// ---------------------------------------------------------------------------
// element kernel, sum-factorised volume term (float64 path)
//
// The volume rule is a tensor grid in the collapsed coordinates (alpha, beta)
// and the basis factors as phi_j = P_a(alpha) chi_j(beta), so
//   interpolation  U(ia,ib) = sum_a P_a(alpha_ia) W(a,ib),  W(a,ib) = sum_{j:a(j)=a} chi_j(beta_ib) c_j
//   projection     V_j = sum_ib chiA_j(ib) Xa(a,ib) + dchiB_j(ib) Xb(a,ib),
//                  Xa(a,ib) = sum_ia wa P_a'(alpha_ia) Ha(ia,ib),  Xb(a,ib) = sum_ia wa P_a(alpha_ia) Hb(ia,ib),
// with Ha = G_r + (1+alpha)/2 G_s, Hb = G_s at the points and the weights and
// chain-rule factors of the collapsed map, d/dr = 2/(1-s) d/dalpha and
// d/ds = (1+alpha)/(1-s) d/dalpha + 2 d/dbeta, folded into the tables
// (chiA = chi wb / (4 (1-s)), dchiB = chi' wb / 4).  This is the same sum as the
// direct projection (Eq. volume), in (p+1)(N_p + (p+1)^2) instead of
// (p+1)^2 N_p products per variable for each of the two contractions.  The
// reference fluxes (G_r, G_s) = J^tau (F1, F2) are formed as the Euler flux
// along the two rows of J^tau, which are constant on the element.
// ---------------------------------------------------------------------------
//
// Q > 0 (a volume rule of Q points without tensor structure: the symmetric
// rules) contracts the volume term directly instead,
//   U(k) = sum_j phi_j(r_k) c_j,   V_j = sum_k w_k (d_r phi_j(r_k) G_r(k) + d_s phi_j(r_k) G_s(k)),
// Q N_p products per variable for each; the lift, the stage update and the
// traces are the same in both forms.
// ---------------------------------------------------------------------------
// EBX > 0 overrides the elements per tile (the fused small-mesh stepper's small
// tiles spread a small mesh over many SMs)
template <int P, int NE, int Q, int EBX = 0>
struct SfCfg {
  using C = Cfg<P, NE, Q>;
  static constexpr bool DIRECT = Q > 0;
  static constexpr int NP = C::NP, ND = C::ND, NQ = C::NQ, NF = C::NF;
  // the volume points in mirror pairs of the Gauss-Legendre nodes (p >= 3; at
  // p = 1 the pairing saves nothing, at p = 2 its registers would cost the
  // third resident CTA per SM).  The small-mesh stepper's tiles take the same
  // arithmetic, so that its results stay bitwise those of k_element_sf.
  static constexpr bool PAIRS = !DIRECT && P >= 3;
  // tiles of 32 elements on 128 threads at p = 1 (64 on 256 measured 2.5 %
  // slower there), 32 on 256 threads at p = 2 (16 on 128: 6 % slower), 16 on
  // 128 at p = 3 (four CTAs per SM instead of two with 32 on 256: 8 % faster;
  // 8 on 64: 8 % slower), 16 on 256 at p = 4-5 (8 on 128: 7 % slower at p = 4,
  // and at p = 5 no faster on the collapsed grid, 6 % slower on the symmetric
  // rule)
  static constexpr int EB = EBX > 0 ? EBX : (P <= 2 ? 32 : 16);
  static constexpr int THREADS = (P <= 1 || P == 3) ? 128 : kThreads;
  // per element and variable, the edge-flux buffer holds the NF gathered fluxes,
  // then (in place) the LW sums of the factorised lift
  static constexpr int LW = ND + 2 * NE;
  static constexpr int RS = NF > LW ? NF : LW;
  static constexpr int TAB = 3 * ND * ND + 3 * NP * ND + ND + 2 * NP * NE + 2 * ND * NE + NP + (DIRECT ? 3 * NP * NQ : 0);
  // per element: the sum-factorisation buffer (8 ND^2), or for the direct form
  // the new state (its point buffer is read until the last mode is done)
  static constexpr int XS = DIRECT ? M * NP : 8 * ND * ND;
  // per element (collapsed grid, p >= 3): the flux directions of H_alpha at the
  // ND alpha nodes and of H_beta, [ND + 1][2], formed once per tile (at p <= 2
  // the few points' FMAs are not worth the registers: at p = 2 they cost a
  // third resident CTA per SM)
  static constexpr bool PREDIR = !DIRECT && P >= 3;
  static constexpr int DS = PREDIR ? 2 * (ND + 1) : 0;
  // SPREAD (the fused small-mesh stepper's tiles): a float64 instruction takes a
  // warp as long with few lanes as with 32, and the tile leaves most lanes idle, so
  // the lift, the modes and the mirror pairs go to more threads: one per variable
  // and sum, one per mode and variable, one per point of a pair (where the items
  // of the pairs and of the middle nodes fit in the block at once).
  static constexpr bool SPREAD = EBX > 0;
  static constexpr int NHALF = 2 * EB * ND * (ND / 2), MIDAT = (NHALF + 31) / 32 * 32;
  static constexpr bool SPREAD_PAIRS = SPREAD && PAIRS && MIDAT + ((ND & 1) ? EB * ND : 0) <= 128;
  static constexpr int LS = SPREAD ? LW : RS;               // stride of the lift sums
  static constexpr int TILE = EB * (M * NP + XS + 8 * NQ + RS * M + DS + (SPREAD ? LW * M : 0));
  static constexpr int SMEM = (TAB + TILE) * 8;
  static_assert(DIRECT || 8 * NQ >= M * NP, "the new state reuses the point buffer");
};

// The Euler flux of U along two directions a and b (Fa = F1 a_x + F2 a_y, ...).
// The Euler flux along a direction d is (rho v_d, rho u v_d + p d_x,
// rho v v_d + p d_y, (E + p) v_d) with v_d = (rho u d_x + rho v d_y) / rho.
__device__ __forceinline__ void flux_two_dirs(const double U[M], double ax, double ay, double bx, double by,
                                              double gamma, int *err, double Fa[M], double Fb[M]) {
  const double inv = recip(U[0]);
  const double p = (gamma - 1.0) * fma(fma(U[1], U[1], U[2] * U[2]), -0.5 * inv, U[3]);
  if (!(positive_finite(U[0]) & positive_finite(p))) atomicOr(err, kErrNonPhysical);
  const double Ep = U[3] + p;
  {
    const double mn = fma(U[1], ax, U[2] * ay), vd = mn * inv;
    Fa[0] = mn; Fa[1] = fma(U[1], vd, p * ax); Fa[2] = fma(U[2], vd, p * ay); Fa[3] = Ep * vd;
  }
  {
    const double mn = fma(U[1], bx, U[2] * by), vd = mn * inv;
    Fb[0] = mn; Fb[1] = fma(U[1], vd, p * bx); Fb[2] = fma(U[2], vd, p * by); Fb[3] = Ep * vd;
  }
}
// Reference fluxes at one volume point: G_r = J^tau row 0 . (F1, F2), G_s = row 1
// . (F1, F2).
__device__ __forceinline__ void ref_flux(const double U[M], const double *g, double gamma, int *err, double Gr[M],
                                         double Gs[M]) {
  flux_two_dirs(U, g[0], g[1], g[2], g[3], gamma, err, Gr, Gs);
}

// mode j -> a (first Dubiner index); modes are ordered by degree d = a+b, then b
__device__ __forceinline__ int mode_a(int j) {
  int d = 0;
  while ((d + 1) * (d + 2) / 2 <= j) ++d;
  return d - (j - d * (d + 1) / 2);
}

// the r-th mode (in mode order) whose first index a is >= 1: degree d holds d of
// them (b = 0 .. d-1), so it lies in the degree d with d(d-1)/2 <= r < d(d+1)/2
__device__ __forceinline__ int mode_a_ge1(int r) {
  int d = 1;
  while (d * (d + 1) / 2 <= r) ++d;
  return d * (d + 1) / 2 + (r - d * (d - 1) / 2);
}

// One tile of the element stage in shared memory (SfCfg::SMEM bytes), in phases that
// the element kernel and the fused small-mesh stepper put together in different
// orders; each phase leaves the synchronisation before the next to its caller
// unless it says otherwise.
template <int P, int NE, int Q, int EBX = 0>
struct SfTile {
  using S = SfCfg<P, NE, Q, EBX>;
  static constexpr int NP = S::NP, ND = S::ND, NQ = S::NQ, NF = S::NF, EB = S::EB, RS = S::RS;
  double *sPa, *sPaW, *sdPaW, *sChi, *sChiA, *sdChiB, *sHalf, *sEChi, *sEWChi, *sEWPa, *sEChiM1, *sEPa;
  double *sBvT, *sDr, *sDs, *sC, *sX, *sH, *sF, *sDir, *sL, *sO;

  __device__ __forceinline__ explicit SfTile(double *smem) {
    sPa = smem;                  // [ND][ND]   P_a(alpha_ia)
    sPaW = sPa + ND * ND;        // [ND][ND]   wa P_a
    sdPaW = sPaW + ND * ND;      // [ND][ND]   wa P_a'
    sChi = sdPaW + ND * ND;      // [NP][ND]   chi_j(beta_ib)
    sChiA = sChi + NP * ND;      // [NP][ND]   chi_j wb / (4 (1-s))
    sdChiB = sChiA + NP * ND;    // [NP][ND]   chi_j' wb / 4
    sHalf = sdChiB + NP * ND;    // [ND]       (1 + alpha_ia) / 2
    sEChi = sHalf + ND;          // [NP][NE]   chi_j(xi_k)
    sEWChi = sEChi + NP * NE;    // [NP][NE]   omega_k chi_j(xi_k)
    sEWPa = sEWChi + NP * NE;    // [ND][NE]   omega_k P_a(xi_k)
    sEChiM1 = sEWPa + ND * NE;   // [NP]       chi_j(-1)
    sEPa = sEChiM1 + NP;         // [ND][NE]   P_a(xi_k)
    sBvT = sEPa + ND * NE;       // direct form: [NP][NQ] phi_j(r_k)
    sDr = sBvT + (S::DIRECT ? NP * NQ : 0);   //  [NQ][NP] w_k d_r phi_j(r_k)
    sDs = sDr + (S::DIRECT ? NQ * NP : 0);    //  [NQ][NP] w_k d_s phi_j(r_k)
    sC = sDs + (S::DIRECT ? NQ * NP : 0);     // [EB][M][NP]        stage input
    sX = sC + EB * M * NP;       // [EB][ND][ND][8]    W (first 4), then Xa, Xb (direct: the new state)
    sH = sX + EB * S::XS;        // [EB][NQ][8]        Ha, Hb (direct: G_r, G_s); later the new state
    sF = sH + EB * NQ * 8;       // [EB][RS][M]        -F_hat_out * l, then the lift sums
    sDir = sF + EB * RS * M;     // [EB][ND+1][2]      J^tau row 0 + half_ia row 1 (ia < ND), row 1
    sL = S::SPREAD ? sDir + EB * S::DS : sF;  // [EB][LS][M]  the lift sums (else in place of the fluxes)
    sO = S::DIRECT ? sX : sH;    // the new state
  }

  __device__ __forceinline__ void load_tables(const DevTables &tab) {
    for (int i = threadIdx.x; i < ND * ND; i += blockDim.x) {
      sPa[i] = tab.SPa[i]; sPaW[i] = tab.SPaW[i]; sdPaW[i] = tab.SdPaW[i];
    }
    for (int i = threadIdx.x; i < NP * ND; i += blockDim.x) {
      sChi[i] = tab.SChi[i]; sChiA[i] = tab.SChiA[i]; sdChiB[i] = tab.SdChiB[i];
    }
    for (int i = threadIdx.x; i < ND; i += blockDim.x) sHalf[i] = tab.SHalf[i];
    for (int i = threadIdx.x; i < NP * NE; i += blockDim.x) { sEChi[i] = tab.EChi[i]; sEWChi[i] = tab.EWChi[i]; }
    for (int i = threadIdx.x; i < ND * NE; i += blockDim.x) sEWPa[i] = tab.EWPa[i];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) sEChiM1[i] = tab.EChiM1[i];
    for (int i = threadIdx.x; i < ND * NE; i += blockDim.x) sEPa[i] = tab.EPa[i];
    if constexpr (S::DIRECT) {
      for (int i = threadIdx.x; i < NP * NQ; i += blockDim.x) {
        sBvT[i] = tab.BvT[i]; sDr[i] = tab.Dr[i]; sDs[i] = tab.Ds[i];
      }
    }
  }

  // the stage input
  __device__ __forceinline__ void load_state(const double *c, int e0, int ecount) {
    const double *src = c + (size_t)e0 * M * NP;
    for (int i = threadIdx.x; i < EB * M * NP; i += blockDim.x) sC[i] = i < ecount * M * NP ? src[i] : 0.0;
  }

  // the flux is linear in its direction: H_alpha = G_r + half G_s is the flux
  // along J^tau row 0 + half row 1, H_beta = G_s the flux along row 1
  __device__ __forceinline__ void load_dirs(const double *__restrict__ geo, int e0, int ecount) {
    if constexpr (S::PREDIR) {
      for (int i = threadIdx.x; i < EB * (ND + 1); i += blockDim.x) {
        const int el = i / (ND + 1), ia = i - el * (ND + 1);
        double dx = 0.0, dy = 0.0;
        if (el < ecount) {
          const double *g = geo + (size_t)(e0 + el) * GEO;
          if (ia < ND) {
            const double half = sHalf[ia];
            dx = fma(half, g[2], g[0]);
            dy = fma(half, g[3], g[1]);
          } else {
            dx = g[2];
            dy = g[3];
          }
        }
        sDir[2 * i] = dx;
        sDir[2 * i + 1] = dy;
      }
    }
  }

  // the element's edge fluxes in its own order, -F_hat_out l; edge(el, q) = 2 f + side
  template <class Edge>
  __device__ __forceinline__ void gather(const double *fhat, Edge &&edge, int ecount, int64_t F, int *err) {
    for (int i = threadIdx.x; i < EB * NF; i += blockDim.x) {
      const int el = i / NF, qk = i - el * NF;
      double v[M] = {0.0, 0.0, 0.0, 0.0};
      if (el < ecount) {
        const int q = qk / NE, k = qk - q * NE;
        const int ef = edge(el, q);
        const int64_t f = checked(ef >> 1, F, err);
        const int side = ef & 1;
        const double *fp = fhat + ((size_t)f * NE + (side ? NE - 1 - k : k)) * M;
#pragma unroll
        for (int m = 0; m < M; ++m) v[m] = side ? fp[m] : tc::neg_bits(fp[m]);
      }
#pragma unroll
      for (int m = 0; m < M; ++m) sF[(el * RS + qk) * M + m] = v[m];
    }
  }

  __device__ __forceinline__ void lift() {
    // the lift's edge sums, in place of the element's fluxes of one variable:
    //   Q_a = sum_k omega_k P_a(xi_k) F0_k                            (face 0)
    //   G_even,k / G_odd,k = F1_k +/- F2_{NE-1-k}                   (faces 1, 2)
    // so that the lift of mode j = (a, b) is
    //   chi_j(-1) Q_a + sum_k omega_k chi_j(xi_k) G_{a mod 2, k}
    if constexpr (S::SPREAD) {
      for (int i = threadIdx.x; i < (ND + NE) * EB * M; i += blockDim.x) {
        const int x = i / (EB * M), r = i - x * (EB * M);
        const double *fe = sF + (r / M) * RS * M + (r % M);
        double *lo = sL + (r / M) * S::LS * M + (r % M);
        if (x < ND) {
          double q = 0.0;
#pragma unroll
          for (int k = 0; k < NE; ++k) q = fma(sEWPa[x * NE + k], fe[k * M], q);
          lo[x * M] = q;
        } else {
          const int k = x - ND;
          const double f1 = fe[(NE + k) * M], f2 = fe[(3 * NE - 1 - k) * M];
          lo[x * M] = f1 + f2;
          lo[(x + NE) * M] = f1 - f2;
        }
      }
    } else {
      for (int i = threadIdx.x; i < EB * M; i += blockDim.x) {
        double *fe = sF + (i / M) * RS * M + (i % M);
        double f[NF];
#pragma unroll
        for (int x = 0; x < NF; ++x) f[x] = fe[x * M];
#pragma unroll
        for (int a = 0; a < ND; ++a) {
          double q = 0.0;
#pragma unroll
          for (int k = 0; k < NE; ++k) q = fma(sEWPa[a * NE + k], f[k], q);
          fe[a * M] = q;
        }
#pragma unroll
        for (int k = 0; k < NE; ++k) {
          fe[(ND + k) * M] = f[NE + k] + f[3 * NE - 1 - k];
          fe[(ND + NE + k) * M] = f[NE + k] - f[3 * NE - 1 - k];
        }
      }
    }
  }

  // the x-th (element, ib) at the middle node alpha = 0 of an odd number of nodes,
  // where P_a(0) = 0 for odd a
  __device__ __forceinline__ void middle_node(int x, int ecount, double gamma, int *err) {
    const int el = x / ND, ib = x - el * ND;
    constexpr int MID = ND / 2;
    const double *w0 = sX + ((el * ND) * ND + ib) * 8;
    double U[M] = {w0[0], w0[1], w0[2], w0[3]};
#pragma unroll
    for (int a = 2; a < ND; a += 2) {
      const double pa = sPa[a * ND + MID];
      const double *w = sX + ((el * ND + a) * ND + ib) * 8;
#pragma unroll
      for (int m = 0; m < M; ++m) U[m] = fma(pa, w[m], U[m]);
    }
    double Ha[M], Hb[M];
    if (el < ecount) {
      const double *dir = sDir + el * 2 * (ND + 1);
      flux_two_dirs(U, dir[2 * MID], dir[2 * MID + 1], dir[2 * ND], dir[2 * ND + 1], gamma, err, Ha, Hb);
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m) { Ha[m] = 0.0; Hb[m] = 0.0; }
    }
    double *h = sH + ((size_t)el * NQ + ib * ND + MID) * 8;
#pragma unroll
    for (int m = 0; m < M; ++m) { h[m] = Ha[m]; h[4 + m] = Hb[m]; }
  }

  // interpolation and the fluxes at the volume points; synchronised on return
  __device__ __forceinline__ void points(const double *__restrict__ geo, int e0, int ecount, double gamma, int *err) {
    if constexpr (S::DIRECT) {
      // volume points: U = sum_j phi_j c_j, then G_r, G_s; one item per (element, point)
      for (int i = threadIdx.x; i < EB * NQ; i += blockDim.x) {
        const int el = i / NQ, k = i - el * NQ;
        double U[M] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          const double b = sBvT[j * NQ + k];
#pragma unroll
          for (int m = 0; m < M; ++m) U[m] = fma(b, sC[(el * M + m) * NP + j], U[m]);
        }
        double Gr[M] = {0.0, 0.0, 0.0, 0.0}, Gs[M] = {0.0, 0.0, 0.0, 0.0};
        if (el < ecount) ref_flux(U, geo + (size_t)(e0 + el) * GEO, gamma, err, Gr, Gs);
        double *h = sH + (size_t)i * 8;
#pragma unroll
        for (int m = 0; m < M; ++m) { h[m] = Gr[m]; h[4 + m] = Gs[m]; }
      }
      __syncthreads();
    } else {
      // W(a, ib) = sum over the modes with first index a of chi_j(beta_ib) c_j; one
      // item per (element, ib, variable) runs over all modes (the same unrolled
      // sequence in every lane)
      for (int i = threadIdx.x; i < EB * ND * M; i += blockDim.x) {
        const int el = i / (ND * M), ib = (i / M) % ND, m = i % M;
        const double *cm = sC + (el * M + m) * NP;
        double w[ND];
#pragma unroll
        for (int a = 0; a < ND; ++a) w[a] = 0.0;
#pragma unroll
        for (int d = 0; d <= P; ++d)
#pragma unroll
          for (int b = 0; b <= d; ++b) {
            const int j = d * (d + 1) / 2 + b;
            w[d - b] = fma(sChi[j * ND + ib], cm[j], w[d - b]);
          }
#pragma unroll
        for (int a = 0; a < ND; ++a) sX[((el * ND + a) * ND + ib) * 8 + m] = w[a];
      }
      __syncthreads();

      // volume points: U = sum_a P_a W; Euler flux; Ha, Hb.
      // PAIRS (p >= 3): one item per (element, ib, mirror pair ia, ia' = ND-1-ia
      // of the Gauss-Legendre nodes), then (p + 1 odd) one per (element, ib) for
      // the middle node.  With P_a(alpha_ia') = (-1)^a P_a(alpha_ia) the pair's
      // states are E +/- O, E = sum_{a even} P_a W, O = sum_{a odd} P_a W, and the
      // point slots of the pair receive the sums and differences the folded
      // projection takes: slot ia (Ha + Ha', Hb + Hb'), slot ia' (Ha - Ha',
      // Hb - Hb'); the middle slot keeps (Ha, Hb).
      if constexpr (S::SPREAD_PAIRS) {
        // a thread per point of a pair (neighbouring lanes), the middle nodes in
        // warps of their own: the sums of the form below, each formed by both
        // threads of a pair or by one of them
        constexpr int NH = ND / 2;
        const int i = threadIdx.x;
        if (i < S::NHALF) {
          const int left = S::NHALF - (i & ~31);
          const unsigned mask = left >= 32 ? 0xFFFFFFFFu : (1u << left) - 1u;
          const int hf = i & 1, pr = i >> 1;
          const int el = pr / (ND * NH), r = pr - el * (ND * NH), ib = r / NH, ia = r - ib * NH;
          const int ia2 = ND - 1 - ia;
          const double *w0 = sX + ((el * ND) * ND + ib) * 8;
          double E[M] = {w0[0], w0[1], w0[2], w0[3]}, O[M];
#pragma unroll
          for (int a = 1; a < ND; ++a) {
            const double pa = sPa[a * ND + ia];
            const double *w = sX + ((el * ND + a) * ND + ib) * 8;
#pragma unroll
            for (int m = 0; m < M; ++m) {
              if (a == 1) O[m] = pa * w[m];
              else if (a & 1) O[m] = fma(pa, w[m], O[m]);
              else E[m] = fma(pa, w[m], E[m]);
            }
          }
          double Ha[M] = {0.0, 0.0, 0.0, 0.0}, Hb[M] = {0.0, 0.0, 0.0, 0.0};
          if (el < ecount) {
            double U[M];
#pragma unroll
            for (int m = 0; m < M; ++m) U[m] = hf ? E[m] - O[m] : E[m] + O[m];
            const double *dir = sDir + el * 2 * (ND + 1), *da = dir + 2 * (hf ? ia2 : ia);
            flux_two_dirs(U, da[0], da[1], dir[2 * ND], dir[2 * ND + 1], gamma, err, Ha, Hb);
          }
          double *h = sH + ((size_t)el * NQ + ib * ND + (hf ? ia2 : ia)) * 8;
#pragma unroll
          for (int m = 0; m < M; ++m) {
            const double oa = __shfl_xor_sync(mask, Ha[m], 1), ob = __shfl_xor_sync(mask, Hb[m], 1);
            h[m] = hf ? __dsub_rn(oa, Ha[m]) : __dadd_rn(Ha[m], oa);
            h[4 + m] = hf ? __dsub_rn(ob, Hb[m]) : __dadd_rn(Hb[m], ob);
          }
        } else if ((ND & 1) && i >= S::MIDAT && i < S::MIDAT + EB * ND) {
          middle_node(i - S::MIDAT, ecount, gamma, err);
        }
      } else if constexpr (S::PAIRS) {
        constexpr int NH = ND / 2, NPAIR = EB * ND * NH, NMID = (ND & 1) ? EB * ND : 0;
        for (int i = threadIdx.x; i < NPAIR + NMID; i += blockDim.x) {
          if ((ND & 1) && i >= NPAIR) {
            // the middle node alpha = 0 (p + 1 odd), after all the pairs so that
            // warps stay uniform
            middle_node(i - NPAIR, ecount, gamma, err);
            continue;
          }
          const int el = i / (ND * NH), r = i - el * (ND * NH), ib = r / NH, ia = r - ib * NH;
          const int ia2 = ND - 1 - ia;
          const double *w0 = sX + ((el * ND) * ND + ib) * 8;
          double E[M] = {w0[0], w0[1], w0[2], w0[3]}, O[M];
#pragma unroll
          for (int a = 1; a < ND; ++a) {
            const double pa = sPa[a * ND + ia];
            const double *w = sX + ((el * ND + a) * ND + ib) * 8;
#pragma unroll
            for (int m = 0; m < M; ++m) {
              if (a == 1) O[m] = pa * w[m];
              else if (a & 1) O[m] = fma(pa, w[m], O[m]);
              else E[m] = fma(pa, w[m], E[m]);
            }
          }
          double S1[M], D1[M], S2[M], D2[M];
          if (el < ecount) {
            const double *dir = sDir + el * 2 * (ND + 1);
            const double bx = dir[2 * ND], by = dir[2 * ND + 1];
            double U[M], Ha[M], Hb[M], Ha2[M], Hb2[M];
#pragma unroll
            for (int m = 0; m < M; ++m) U[m] = E[m] + O[m];
            flux_two_dirs(U, dir[2 * ia], dir[2 * ia + 1], bx, by, gamma, err, Ha, Hb);
#pragma unroll
            for (int m = 0; m < M; ++m) U[m] = E[m] - O[m];
            flux_two_dirs(U, dir[2 * ia2], dir[2 * ia2 + 1], bx, by, gamma, err, Ha2, Hb2);
#pragma unroll
            for (int m = 0; m < M; ++m) {
              // (not contracted with the products they add: SPREAD_PAIRS adds them
              // in another thread than the one that formed them)
              S1[m] = __dadd_rn(Ha[m], Ha2[m]); D1[m] = __dsub_rn(Ha[m], Ha2[m]);
              S2[m] = __dadd_rn(Hb[m], Hb2[m]); D2[m] = __dsub_rn(Hb[m], Hb2[m]);
            }
          } else {
#pragma unroll
            for (int m = 0; m < M; ++m) { S1[m] = 0.0; D1[m] = 0.0; S2[m] = 0.0; D2[m] = 0.0; }
          }
          double *h1 = sH + ((size_t)el * NQ + ib * ND + ia) * 8, *h2 = sH + ((size_t)el * NQ + ib * ND + ia2) * 8;
#pragma unroll
          for (int m = 0; m < M; ++m) {
            h1[m] = S1[m]; h1[4 + m] = S2[m];
            h2[m] = D1[m]; h2[4 + m] = D2[m];
          }
        }
      } else {
        for (int i = threadIdx.x; i < EB * NQ; i += blockDim.x) {
          const int el = i / NQ, k = i - el * NQ, ib = k / ND, ia = k - ib * ND;
          // P_0 = 1: the a = 0 term is W(0, ib) itself
          const double *w0 = sX + ((el * ND) * ND + ib) * 8;
          double U[M] = {w0[0], w0[1], w0[2], w0[3]};
#pragma unroll
          for (int a = 1; a < ND; ++a) {
            const double pa = sPa[a * ND + ia];
            const double *w = sX + ((el * ND + a) * ND + ib) * 8;
#pragma unroll
            for (int m = 0; m < M; ++m) U[m] += pa * w[m];
          }
          double Ha[M], Hb[M];
          if (el < ecount) {
            if constexpr (S::PREDIR) {
              const double *dir = sDir + el * 2 * (ND + 1);
              flux_two_dirs(U, dir[2 * ia], dir[2 * ia + 1], dir[2 * ND], dir[2 * ND + 1], gamma, err, Ha, Hb);
            } else {
              // the flux along J^tau row 0 + half row 1 and along row 1
              const double *g = geo + (size_t)(e0 + el) * GEO;
              const double half = sHalf[ia];
              flux_two_dirs(U, fma(half, g[2], g[0]), fma(half, g[3], g[1]), g[2], g[3], gamma, err, Ha, Hb);
            }
          } else {
#pragma unroll
            for (int m = 0; m < M; ++m) { Ha[m] = 0.0; Hb[m] = 0.0; }
          }
          double *h = sH + (size_t)i * 8;
#pragma unroll
          for (int m = 0; m < M; ++m) { h[m] = Ha[m]; h[4 + m] = Hb[m]; }
        }
      }
      __syncthreads();
    }
  }

  // the sums over the points of a row (collapsed grid); synchronised on return
  __device__ __forceinline__ void row_sums() {
    if constexpr (!S::DIRECT) {
      if constexpr (P >= 2 && P <= 4) {
        // Xa(a, ib) = sum_ia Ha wa P_a', Xb(a, ib) = sum_ia Hb wa P_a, one item per
        // (element, ib, variable) over every a, folded on the mirror pairs of the
        // Gauss-Legendre nodes (alpha_{ND-1-ia} = -alpha_ia, the same weight):
        // P_a(-x) = (-1)^a P_a(x) and P_a'(-x) = (-1)^(a+1) P_a'(x), so
        //   Xb(a) = sum_{ia < ND/2} wa P_a(alpha_ia) (Hb_ia +/- Hb_ia'),  + for a even
        //   Xa(a) = sum_{ia < ND/2} wa P_a'(alpha_ia) (Ha_ia -/+ Ha_ia'), - for a even,
        // and for ND odd the middle node alpha = 0 enters Xb of the even a and Xa
        // of the odd a only (P_a(0) = 0 for a odd, P_a'(0) = 0 for a even).  Per item
        // that is 4 (ND / 2) additions (already formed by the point phase when
        // PAIRS) and about half the products of the plain sums; Xa(0, ib) = 0
        // (P_0' = 0) costs no arithmetic.
        constexpr int NH = ND / 2, MID = ND / 2;
        for (int i = threadIdx.x; i < EB * ND * M; i += blockDim.x) {
          const int el = i / (ND * M), ib = (i / M) % ND, m = i % M;
          const double *hrow = sH + ((el * NQ) + ib * ND) * 8;
          double ea[NH], oa[NH], eb[NH], ob[NH];
#pragma unroll
          for (int ia = 0; ia < NH; ++ia) {
            const double *h1 = hrow + ia * 8, *h2 = hrow + (ND - 1 - ia) * 8;
            const double a1 = h1[m], a2 = h2[m], b1 = h1[4 + m], b2 = h2[4 + m];
            if constexpr (S::PAIRS) {
              ea[ia] = a1; oa[ia] = a2;
              eb[ia] = b1; ob[ia] = b2;
            } else {
              ea[ia] = a1 + a2; oa[ia] = a1 - a2;
              eb[ia] = b1 + b2; ob[ia] = b1 - b2;
            }
          }
          double xa[ND], xb[ND];
#pragma unroll
          for (int a = 0; a < ND; ++a) {
            const double *fb = (a & 1) ? ob : eb, *fa = (a & 1) ? ea : oa;
            double sb = 0.0, sa = 0.0;
            if ((ND & 1) && !(a & 1)) sb = hrow[MID * 8 + 4 + m] * sPaW[a * ND + MID];
            if ((ND & 1) && (a & 1)) sa = hrow[MID * 8 + m] * sdPaW[a * ND + MID];
#pragma unroll
            for (int ia = 0; ia < NH; ++ia) {
              sb = fma(fb[ia], sPaW[a * ND + ia], sb);
              if (a > 0) sa = fma(fa[ia], sdPaW[a * ND + ia], sa);
            }
            xa[a] = sa;
            xb[a] = sb;
          }
#pragma unroll
          for (int a = 0; a < ND; ++a) {
            double *x = sX + ((el * ND + a) * ND + ib) * 8;
            x[m] = xa[a];
            x[4 + m] = xb[a];
          }
        }
      } else if constexpr (P <= 4) {
        // p = 1: the plain sums (the folding would add more than it saves)
        for (int i = threadIdx.x; i < EB * ND * M; i += blockDim.x) {
          const int el = i / (ND * M), ib = (i / M) % ND, m = i % M;
          double xa[ND], xb[ND];
#pragma unroll
          for (int a = 0; a < ND; ++a) { xa[a] = 0.0; xb[a] = 0.0; }
#pragma unroll
          for (int ia = 0; ia < ND; ++ia) {
            const double *h = sH + ((el * NQ) + ib * ND + ia) * 8;
            const double ha = h[m], hb = h[4 + m];
#pragma unroll
            for (int a = 1; a < ND; ++a) xa[a] = fma(ha, sdPaW[a * ND + ia], xa[a]);
#pragma unroll
            for (int a = 0; a < ND; ++a) xb[a] = fma(hb, sPaW[a * ND + ia], xb[a]);
          }
#pragma unroll
          for (int a = 0; a < ND; ++a) {
            double *x = sX + ((el * ND + a) * ND + ib) * 8;
            x[m] = xa[a];
            x[4 + m] = xb[a];
          }
        }
      } else {
        // p = 5: one item per (element, a, ib) for all four variables (the
        // per-variable form above would spill at this size), on the pair sums and
        // differences of the point phase (PAIRS): Xa(a) takes the sums of Ha for
        // a odd and the differences for a even, Xb(a) the sums of Hb for a even
        // and the differences for a odd, over the ND / 2 pairs
        static_assert(S::PAIRS && S::PREDIR, "p = 5 has mirror pairs");
        constexpr int NH = ND / 2;
        for (int i = threadIdx.x; i < EB * ND * ND; i += blockDim.x) {
          const int el = i / (ND * ND), a = (i / ND) % ND, ib = i % ND;
          double xa[M] = {0.0, 0.0, 0.0, 0.0}, xb[M] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
          for (int ia = 0; ia < NH; ++ia) {
            const double dp = sdPaW[a * ND + ia], pa = sPaW[a * ND + ia];
            const double *hs = sH + ((el * NQ) + ib * ND + ia) * 8, *hd = sH + ((el * NQ) + ib * ND + ND - 1 - ia) * 8;
            const double *fa = (a & 1) ? hs : hd, *fb = (a & 1) ? hd : hs;
#pragma unroll
            for (int m = 0; m < M; ++m) { xa[m] = fma(fa[m], dp, xa[m]); xb[m] = fma(fb[4 + m], pa, xb[m]); }
          }
          double *x = sX + (size_t)i * 8;
#pragma unroll
          for (int m = 0; m < M; ++m) { x[m] = xa[m]; x[4 + m] = xb[m]; }
        }
      }
      __syncthreads();

    }
  }

  // update(el, j, m, acc): the new value of mode j, variable m of element el from its
  // projection and lift acc
  template <class Update>
  __device__ __forceinline__ void modes(int ecount, Update &&update) {
    // V_j + lifted edge fluxes, then the caller's update.  Sum-factorised: the items
    // of the modes with a >= 1 come first and those of the modes with a = 0 (b = d)
    // last, so that warps take one branch of the projection (for a = 0,
    // Xa(0, .) = 0 and only the Xb term is formed).  An item has all four variables;
    // SPREAD: one.
    constexpr int NV = S::SPREAD ? 1 : M, IV = M / NV;
    for (int i = threadIdx.x; i < EB * NP * IV; i += blockDim.x) {
      const int it = i / IV, m0 = i - it * IV;
      int el, j;
      if constexpr (S::DIRECT) {
        el = it / NP;
        j = it - el * NP;
      } else {
        constexpr int NB = NP - ND;                   // modes with a >= 1
        if (it < EB * NB) {
          el = it / NB;
          j = mode_a_ge1(it - el * NB);
        } else {
          const int i2 = it - EB * NB;
          el = i2 / ND;
          const int d = i2 - el * ND;
          j = d * (d + 1) / 2 + d;
        }
      }
      const int a = mode_a(j);
      double acc[NV];
#pragma unroll
      for (int m = 0; m < NV; ++m) acc[m] = 0.0;
      if constexpr (S::DIRECT) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
          const double dr = sDr[k * NP + j], ds = sDs[k * NP + j];
          const double *h = sH + (el * NQ + k) * 8 + m0;
#pragma unroll
          for (int m = 0; m < NV; ++m) acc[m] = fma(ds, h[4 + m], fma(dr, h[m], acc[m]));
        }
      } else if (a > 0) {
#pragma unroll
        for (int ib = 0; ib < ND; ++ib) {
          const double ch = sChiA[j * ND + ib], dch = sdChiB[j * ND + ib];
          const double *x = sX + ((el * ND + a) * ND + ib) * 8 + m0;
#pragma unroll
          for (int m = 0; m < NV; ++m) acc[m] = fma(dch, x[4 + m], fma(ch, x[m], acc[m]));
        }
      } else {
#pragma unroll
        for (int ib = 0; ib < ND; ++ib) {
          const double dch = sdChiB[j * ND + ib];
          const double *x = sX + (el * ND * ND + ib) * 8 + m0;
#pragma unroll
          for (int m = 0; m < NV; ++m) acc[m] = fma(dch, x[4 + m], acc[m]);
        }
      }
      {
        const double *fl = sL + el * S::LS * M + m0;
        const double c1 = sEChiM1[j];
#pragma unroll
        for (int m = 0; m < NV; ++m) acc[m] = fma(c1, fl[a * M + m], acc[m]);
        const double *g = fl + (ND + (a & 1) * NE) * M;
#pragma unroll
        for (int k = 0; k < NE; ++k) {
          const double l = sEWChi[j * NE + k];
#pragma unroll
          for (int m = 0; m < NV; ++m) acc[m] = fma(l, g[k * M + m], acc[m]);
        }
      }
      // the new state, for the next stage's traces (sum-factorised: sH is free,
      // every thread has passed the barrier after the row sums, the last reader of
      // sH; direct: a buffer of its own, the modes still read sH)
#pragma unroll
      for (int m = 0; m < NV; ++m)
        sO[(el * M + m0 + m) * NP + j] = el < ecount ? update(el, j, m0 + m, acc[m]) : 0.0;
    }
  }

  // the edge traces of the state sS, sO or sC (synchronises before its first read)
  __device__ __forceinline__ void traces(const double *sS, double *trace_out, int e0, int ecount) {
      __syncthreads();
      // Z_a of the new state (face 0 lies on beta = -1), one item per (element,
      // variable), in the buffer the modes have finished reading (sX; direct: sH)
      double *sZ = S::DIRECT ? sH : sX;
      for (int i = threadIdx.x; i < ecount * M; i += blockDim.x) {
        double z[ND + 1];
        face_sums<P>(sS + i * NP, sEChiM1, sEChi[0], z);
#pragma unroll
        for (int a = 0; a <= ND; ++a) sZ[i * (ND + 1) + a] = z[a];
      }
      __syncthreads();
      // edge traces of the new state, one item per (element, variable, edge point k):
      //   T0_k = sum_a P_a(xi_k) Z_a,
      //   T1_k = sum_a Y_a(xi_k),  T2_{NE-1-k} = sum_a (-1)^a Y_a(xi_k),
      //   Y_a(xi) = sum_b chi_ab(xi) c_ab
      for (int i = threadIdx.x; i < ecount * M * NE; i += blockDim.x) {
        const int el = i / (M * NE), m = (i / NE) % M, k = i % NE;
        const double *cj = sS + (el * M + m) * NP;
        double *dst = trace_out + (size_t)(e0 + el) * NF * M + m;
        double t0, t1, t2;
        edge_traces_unit<P, NE>(cj, sZ + (el * M + m) * (ND + 1), sEPa, sEChi, k, t0, t1, t2);
        dst[k * M] = t0;
        dst[(NE + k) * M] = t1;
        dst[(3 * NE - 1 - k) * M] = t2;
      }
  }
};

// a0 u0 + b0 c + g dt R with R = acc / det J, as b0 c + a0 u0 + (g dt / det J) acc
__device__ __forceinline__ double stage_value(const StageUpdate &su, double kap, double c, double u0, double acc) {
  double t = su.b0 * c;
  if (su.a0 != 0.0) t = fma(su.a0, u0, t);
  return fma(kap, acc, t);
}
// x acc2 + y v + (w dt / det J) acc, the running sum of the classical RK4
__device__ __forceinline__ double stage_sum(const StageUpdate &su, double inv, double v, double acc2, double acc) {
  double t2 = su.y * v;
  if (su.x != 0.0) t2 = fma(su.x, acc2, t2);
  return fma(su.w * su.dt * inv, acc, t2);
}

template <int P, int NE, int Q>
__global__ void __launch_bounds__(kThreads, 2)
k_element_sf(const double *c, const double *u0, double *out, double *__restrict__ trace_out,
             const double *__restrict__ fhat, const double *__restrict__ geo,
             const int32_t *__restrict__ elem_face, DevTables tab, int N, int64_t F, StageUpdate su, int mode,
             double gamma, int *err) {
  extern __shared__ double smem[];
  SfTile<P, NE, Q> t(smem);
  constexpr int NP = SfCfg<P, NE, Q>::NP, EB = SfCfg<P, NE, Q>::EB;
  t.load_tables(tab);
  const int ntiles = (N + EB - 1) / EB;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int e0 = tile * EB, ecount = min(EB, N - e0);
    __syncthreads();
    t.load_state(c, e0, ecount);
    t.load_dirs(geo, e0, ecount);
    t.gather(fhat, [&](int el, int q) { return elem_face[(size_t)(e0 + el) * 3 + q]; }, ecount, F, err);
    __syncthreads();
    t.lift();
    t.points(geo, e0, ecount, gamma, err);
    t.row_sums();
    t.modes(ecount, [&](int el, int j, int m, double acc) {
      const size_t e = (size_t)(e0 + el), idx = (e * M + m) * NP + j;
      const double inv = geo[e * GEO + 4];
      const double kap = su.g * su.dt * inv;
      double v;
      if (mode == 0) {
        v = acc * inv;
      } else {
        v = stage_value(su, kap, t.sC[(el * M + m) * NP + j], su.a0 != 0.0 ? u0[idx] : 0.0, acc);
        if (su.out2) su.out2[idx] = stage_sum(su, inv, v, su.x != 0.0 ? su.acc[idx] : 0.0, acc);
      }
      out[idx] = v;
      return v;
    });
    if (trace_out) t.traces(t.sO, trace_out, e0, ecount);
  }
}

// CTAs of k_element_sf per SM (the kernel's shared memory attribute set first)
template <int P, int NE, int Q>
int element_sf_per_sm(const dg_mesh *m, int *per_sm) {
  using S = SfCfg<P, NE, Q>;
  static PerDevice attr_set;
  if (!attr_set.test(m->device)) {
    cudaError_t e = cudaFuncSetAttribute(k_element_sf<P, NE, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
    if (e != cudaSuccess) return (int)e;
    e = cudaFuncSetAttribute(k_element_sf<P, NE, Q>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return (int)e;
    attr_set.set(m->device);
  }
  *per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_element_sf<P, NE, Q>, S::THREADS, S::SMEM);
  if (e != cudaSuccess) return (int)e;
  if (*per_sm < 1) *per_sm = 1;
  return (int)cudaSuccess;
}

// Elements [e0, e1) of the mesh (e1 < 0: all): the kernel runs on the views of
// the arrays that start at element e0.  Each element's arithmetic does not
// depend on the tile it falls in, so a range launch gives the same bits.
template <int P, int NE, int Q>
int run_element_sf(const dg_mesh *m, const double *c, const double *u0, double *out, double *trace_out,
                   const double *fhat, const StageUpdate &su0, int mode, cudaStream_t s, int64_t e0 = 0,
                   int64_t e1 = -1) {
  using S = SfCfg<P, NE, Q>;
  int per_sm = 0;
  int err = element_sf_per_sm<P, NE, Q>(m, &per_sm);
  if (err != (int)cudaSuccess) return err;
  if (e1 < 0) e1 = m->N;
  const int64_t n = e1 - e0;
  if (n <= 0) return (int)cudaSuccess;
  const size_t so = (size_t)e0 * M * S::NP;           // state rows of the range
  StageUpdate su = su0;
  if (su.acc) su.acc += so;
  if (su.out2) su.out2 += so;
  const int ntiles = (int)((n + S::EB - 1) / S::EB);
  const int grid = ntiles < m->num_sms * per_sm ? ntiles : m->num_sms * per_sm;
  k_element_sf<P, NE, Q><<<grid, S::THREADS, S::SMEM, s>>>(
      c + so, u0 ? u0 + so : nullptr, out + so, trace_out ? trace_out + (size_t)e0 * S::NF * M : nullptr, fhat,
      m->geo + (size_t)e0 * GEO, m->elem_face + (size_t)e0 * 3, m->tab, (int)n, m->F, su, mode, m->gamma,
      m->err_flag);
  return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// fused small-mesh stepper
//
// On a mesh whose element tiles fit in one wave of the GPU, a stage's two
// launches (edge flux, element) do a few microseconds of work each and the step
// is bound by launch latency (the paper's Section 7.1 finds its small meshes
// alike).  This kernel runs every stage of a whole call inside one cooperative
// launch, one tile per block: the edge phase (face_flux_points) and the phases of
// SfTile, the code of k_face and k_element_sf, with barriers over the grid between
// them, so the results are bitwise those of the separate launches.
//
// A block keeps its tile's state, the step's first state, the classical RK4's
// running sum, geometry and connectivity in shared memory from one stage to the
// next; only traces and edge fluxes pass through memory.  The volume integral needs
// neither, so it runs between a block's arrival at a barrier and its wait: the
// points of the next stage behind the barrier after the traces, the row sums
// behind the one after the edge fluxes.  (Cycles of a stage, p = 4, 800 elements:
// 52,500 with whole barriers and the tile read back from memory at each stage, of
// which 11,500 the barriers, 5,000 the loads and 11,000 the update that waited for
// its operands; 33,900 now.  p = 1, 512 elements: 30,000 -> 17,800.)
// ---------------------------------------------------------------------------
constexpr uint64_t kGridWaitNs = 2000000000ull;    // 2 s per barrier before giving up

// A barrier over all blocks of the (co-resident) grid in two parts.  Arrival: the
// block's writes so far, then one more on the counter; wait: until the counter
// reaches target (nblocks times the barriers so far; it starts at 0).  The wait is
// bounded: after kGridWaitNs it records kErrTimeout and returns false, and the
// caller leaves the kernel.
__device__ __forceinline__ void grid_arrive(unsigned *bar) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();                                  // this block's writes before its arrival
    atomicAdd(bar, 1u);
  }
}
__device__ __forceinline__ bool grid_wait(unsigned *bar, unsigned target, int *err) {
  __shared__ int ok_s;
  if (threadIdx.x == 0) {
    int ok = 1;
    uint64_t t0 = 0;
    for (unsigned it = 1;; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((it & 255u) == 0u) {
        const uint64_t t = tc::global_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > kGridWaitNs) {
          atomicOr(err, kErrTimeout);
          ok = 0;
          break;
        }
      }
    }
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

constexpr int kSmallThreads = 128;
constexpr int kSmallTiles[2] = {4, 8};          // elements per tile of the two variants

// Blocks per SM that the stepper's registers are held to.  At p = 1 the 8-element
// tiles take five (96 registers, no spills, instead of 122-128), which serves meshes
// up to 6,080 elements on 152 SMs: ten SSP-RK3 steps at 5,000-6,050 elements 0.30-0.32
// ms against 0.56 with separate launches (0.53-0.58 before the split-product kernel).
// At p >= 2 the separate launches are the faster ones beyond four blocks.
constexpr int small_blocks(int p, int tile) { return p == 1 && tile == 8 ? 5 : 4; }

// shared memory of the stepper: the tile's phases, then the step's first state and
// the RK4 sum [EB][M][NP], 1/det J [EB] and the elements' edges [EB][3]
template <int P, int NE, int Q, int EBX>
struct SmallCfg {
  using S = SfCfg<P, NE, Q, EBX>;
  static constexpr int ROWS = S::EB * M * S::NP;
  static constexpr int SMEM = S::SMEM + (2 * ROWS + S::EB) * 8 + (3 * S::EB + 1) / 2 * 8;
};

template <int P, int NE, int Q, int EBX>
__global__ void __launch_bounds__(kSmallThreads, small_blocks(P, EBX))
k_rk_small(double *c, double *S, double *A, double *trace, double *fhat, const double *__restrict__ geo,
           const int32_t *__restrict__ elem_face, const FaceConn *__restrict__ conn, const FaceGeo *__restrict__ fg,
           const FaceFix *__restrict__ ff, const double *__restrict__ bstate, const int32_t *__restrict__ elem_nbr,
           DevTables tab, int N, int64_t F, GammaFix gf, double phi1, double dt, int nsteps, int method, int limit, unsigned *bar, int *err) {
  extern __shared__ double smem[];
  using Sm = SmallCfg<P, NE, Q, EBX>;
  constexpr int NP = Sm::S::NP, EB = Sm::S::EB, ROWS = Sm::ROWS;
  SfTile<P, NE, Q, EBX> t(smem);
  double *sU0 = smem + Sm::S::SMEM / 8, *sA = sU0 + ROWS, *sInv = sA + ROWS;
  int32_t *sEf = reinterpret_cast<int32_t *>(sInv + EB);
  const unsigned nb = gridDim.x;
  unsigned target = 0;
  const int ns = rk_num_stages(method);
  const int e0 = blockIdx.x * EB, ecount = min(EB, N - e0);

  t.load_tables(tab);
  t.load_state(c, e0, ecount);
  for (int i = threadIdx.x; i < ecount * 3; i += blockDim.x) sEf[i] = elem_face[(size_t)e0 * 3 + i];
  for (int i = threadIdx.x; i < ecount; i += blockDim.x) sInv[i] = geo[(size_t)(e0 + i) * GEO + 4];
  __syncthreads();
  t.load_dirs(geo, e0, ecount);
  t.traces(t.sC, trace, e0, ecount);
  grid_arrive(bar);
  target += nb;
  t.points(geo, e0, ecount, gf.gamma, err);
  if (!grid_wait(bar, target, err)) return;
  bool have_points = true;
  for (int step = 0; step < nsteps; ++step)
    for (int i = 0; i < ns; ++i) {
      const RkStage st = rk_stage(method, i, dt, c, S, A);
      const bool last = step == nsteps - 1 && i == ns - 1;
      if (i == 0)
        for (int x = threadIdx.x; x < ROWS; x += blockDim.x) sU0[x] = t.sC[x];
      face_flux_points<NE>(trace, fhat, conn, fg, ff, bstate, N, F, gf, err, blockIdx.x, nb);
      grid_arrive(bar);
      target += nb;
      if (!have_points) t.points(geo, e0, ecount, gf.gamma, err);
      t.row_sums();
      if (!grid_wait(bar, target, err)) return;
      t.gather(fhat, [&](int el, int q) { return sEf[el * 3 + q]; }, ecount, F, err);
      __syncthreads();
      t.lift();
      __syncthreads();
      const double *u0 = method == DG_RK4 && i == 3 ? sA : sU0;
      const StageUpdate &su = st.su;
      t.modes(ecount, [&](int el, int j, int m, double acc) {
        const double inv = sInv[el], kap = su.g * su.dt * inv;
        const int x = (el * M + m) * NP + j;
        const double v = stage_value(su, kap, t.sC[x], u0[x], acc);
        if (su.out2) sA[x] = stage_sum(su, inv, v, sA[x], acc);
        if (limit || last) st.out[(size_t)e0 * M * NP + x] = v;
        return v;
      });
      t.traces(t.sO, trace, e0, ecount);
      if (last && !limit) return;
      grid_arrive(bar);
      target += nb;
      have_points = !limit;
      if (have_points) {
        for (int x = threadIdx.x; x < ROWS; x += blockDim.x) t.sC[x] = x < ecount * M * NP ? t.sO[x] : 0.0;
        __syncthreads();
        t.points(geo, e0, ecount, gf.gamma, err);
      }
      if (!grid_wait(bar, target, err)) return;
      if constexpr (P == 1) {
        // with the limiter on, every stage value is limited in place (and the
        // traces of the elements it limits rewritten) before the next stage, which
        // reads its tile back
        if (limit) {
          limit_p1_items<true>(st.out, trace, elem_nbr, tab.EPa, tab.EChiM1, tab.EChi, phi1, N, err, blockIdx.x, nb);
          if (last) return;
          grid_arrive(bar);
          target += nb;
          if (!grid_wait(bar, target, err)) return;
          t.load_state(st.out, e0, ecount);
          __syncthreads();
        }
      }
    }
}

// Resident blocks per SM of the two variants on the mesh's device (0: not
// launchable), asked once per device.
template <int P, int NE, int Q>
const int *small_per_sm(int dev) {
  static PerDevice ready;
  static int per_sm[64][2];
  static int fallback[2];
  int *r = dev >= 0 && dev < 64 ? per_sm[dev] : fallback;
  if (dev >= 0 && dev < 64 && ready.test(dev)) return r;
  auto k0 = k_rk_small<P, NE, Q, kSmallTiles[0]>;
  auto k1 = k_rk_small<P, NE, Q, kSmallTiles[1]>;
  const int s0 = SmallCfg<P, NE, Q, kSmallTiles[0]>::SMEM, s1 = SmallCfg<P, NE, Q, kSmallTiles[1]>::SMEM;
  int v[2] = {0, 0};           // (r is written once complete: two threads may ask at the same time)
  if (cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, s0) != cudaSuccess ||
      cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, s1) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v[0], k0, kSmallThreads, s0) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v[1], k1, kSmallThreads, s1) != cudaSuccess) {
    cudaGetLastError();
    v[0] = v[1] = 0;
  }
  r[0] = v[0];
  r[1] = v[1];
  if (dev >= 0 && dev < 64) ready.set(dev);
  return r;
}

// the variant whose tiles of the mesh fit in one wave (its blocks all resident),
// the smaller tiles first; -1 if neither
template <int P, int NE, int Q>
int small_variant(const dg_mesh *m) {
  const int *per_sm = small_per_sm<P, NE, Q>(m->device);
  for (int v = 0; v < 2; ++v) {
    const int64_t nb = (m->N + kSmallTiles[v] - 1) / kSmallTiles[v];
    if (per_sm[v] > 0 && nb <= (int64_t)m->num_sms * per_sm[v]) return v;
  }
  return -1;
}

template <int P, int NE, int Q, int EBX>
int run_rk_small(dg_mesh *m, double *c, double dt, int nsteps, int method, cudaStream_t s) {
  using Sc = SmallCfg<P, NE, Q, EBX>;
  auto kern = k_rk_small<P, NE, Q, EBX>;
  // one tile per block (the variant was chosen so that they are all resident);
  // the edge phase spreads its points over the same blocks
  const int64_t nb = (m->N + EBX - 1) / EBX;
  cudaError_t e = cudaMemsetAsync(m->gbar, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return (int)e;
  double *S = m->stage, *A = m->rk_acc, *tr = m->trace, *fh = m->fhat;
  const double *geo = m->geo, *bst = m->bstate;
  const int32_t *ef = m->elem_face;
  const FaceConn *conn = m->face_conn;
  const FaceGeo *fg = m->face_geo;
  const FaceFix *ff = m->face_fix;
  DevTables tab = m->tab;
  int N = (int)m->N;
  int64_t F = m->F;
  GammaFix gf = gamma_fix(m->gamma);
  unsigned *bar = m->gbar;
  int *err = m->err_flag;
  const int32_t *nbr = m->elem_nbr;
  double phi1 = m->phi1;
  int limit = m->limiter ? 1 : 0;
  void *args[] = {&c,   &S, &A, &tr,    &fh,   &geo, &ef,     &conn,  &fg,   &ff, &bst, &nbr, &tab,
                  &N,   &F, &gf, &phi1, &dt,   &nsteps, &method, &limit, &bar, &err};
  return (int)cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)nb), dim3(kSmallThreads), args,
                                          Sc::SMEM, s);
}

template <int P, int NE, int Q>
int run_small(dg_mesh *m, double *c, double dt, int nsteps, int method, cudaStream_t s) {
  switch (small_variant<P, NE, Q>(m)) {
    case 0: return run_rk_small<P, NE, Q, kSmallTiles[0]>(m, c, dt, nsteps, method, s);
    case 1: return run_rk_small<P, NE, Q, kSmallTiles[1]>(m, c, dt, nsteps, method, s);
    default: return (int)cudaErrorCooperativeLaunchTooLarge;
  }
}

template <int P, int NE, int Q>
bool fits_small(const dg_mesh *m) {
  return small_variant<P, NE, Q>(m) >= 0;
}

}  // namespace

bool small_rk_fits(const dg_mesh *m) {
#define CALL(P, NE) (m->rule == DG_RULE_SYMMETRIC ? fits_small<P, NE, sym_points(P)>(m) : fits_small<P, NE, 0>(m))
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return false;
}

int launch_rk_small(dg_mesh *m, double *c, double dt, int nsteps, int method, void *stream) {
  cudaStream_t s = (cudaStream_t)stream;
#define CALL(P, NE)                                                                        \
  (m->rule == DG_RULE_SYMMETRIC ? run_small<P, NE, sym_points(P)>(m, c, dt, nsteps, method, s) \
                                : run_small<P, NE, 0>(m, c, dt, nsteps, method, s))
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

int element_wave(const dg_mesh *m, int *tiles, int *elems_per_tile) {
  if (m->split_img) {
    *tiles = split_wave(m);
    *elems_per_tile = 32;
    return (int)cudaSuccess;
  }
#define CALL(P, NE)                                                                                 \
  (m->rule == DG_RULE_SYMMETRIC                                                                     \
       ? (*elems_per_tile = SfCfg<P, NE, sym_points(P)>::EB, element_sf_per_sm<P, NE, sym_points(P)>(m, tiles)) \
       : (*elems_per_tile = SfCfg<P, NE, 0>::EB, element_sf_per_sm<P, NE, 0>(m, tiles)))
  int e = (int)cudaErrorInvalidValue;
  if (m->p == 1 && m->ne == 2) e = CALL(1, 2);
  else if (m->p == 2 && m->ne == 3) e = CALL(2, 3);
  else if (m->p == 3 && m->ne == 4) e = CALL(3, 4);
  else if (m->p == 3 && m->ne == 3) e = CALL(3, 3);
  else if (m->p == 4 && m->ne == 5) e = CALL(4, 5);
  else if (m->p == 5 && m->ne == 6) e = CALL(5, 6);
#undef CALL
  if (e == (int)cudaSuccess) *tiles *= m->num_sms;
  return e;
}

int launch_element(const dg_mesh *m, const double *c, const double *u0, double *out, double *trace_out,
                   const double *fhat, const StageUpdate &su, int mode, void *stream, int64_t e0, int64_t e1) {
  cudaStream_t s = (cudaStream_t)stream;
  if (m->split_img) return launch_split(m, c, u0, out, trace_out, fhat, su, mode, nullptr, stream, e0, e1);
#define CALL(P, NE)                                                                                        \
  (m->rule == DG_RULE_SYMMETRIC                                                                            \
       ? run_element_sf<P, NE, sym_points(P)>(m, c, u0, out, trace_out, fhat, su, mode, s, e0, e1)        \
       : run_element_sf<P, NE, 0>(m, c, u0, out, trace_out, fhat, su, mode, s, e0, e1))
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

}  // namespace dg
