/*
 * dg_adj_split.cu -- the discrete adjoint's element kernels with their contractions
 * on the tensor cores, by the exact digit products of dg_split.cuh: the transposes
 * k_adj_element_sf / k_adj_element and k_adj_combine_sf / k_adj_combine of meshes
 * that use the split-product kernel, p <= 3 (further up the three point buffers of
 * a group leave room for one group per SM).
 *
 *   k_adj_split      u's values at the volume points and edge traces T = B_f u; from
 *                    lb = lam / det J the cotangents of G_r, G_s at the points
 *                    (transposed projection) and G, those of the lifted fluxes
 *                    (transposed lift); the pull-back through J^tau and the Euler
 *                    flux Jacobians in float64, one (element, point) a thread; then
 *                    uvol, the transposed interpolation
 *   k_adj_sum_split  out = x0 X + x1 Y + x2 Z + s (uvol + B_f^T TB)
 *
 * The float64 pipe bounds both as it bounds the forward kernel; here it keeps the
 * pull-back (52 operations a point) and the sums, of about 1,435 + 200 float64
 * instructions per element at p = 2 (131,072 elements: k_adj_split 359 -> 196 us,
 * k_adj_sum_split 73 -> 51 us against the factorised kernels).  Tiles, groups,
 * digits and turns as in k_element_split.
 */
#include "dg_split.cuh"

namespace dg {
namespace {

// the tables of the adjoint's contractions
enum { kTabU, kTabT, kTabR, kTabS, kTabG, kTabV, kTabB, kAdjTabs };

template <int P, int NE, int Q>
struct Ap {
  using T = Sp<P, NE, Q>;
  static constexpr int SUBS = 3, THREADS = SUBS * kSubThreads, SUBCOLS = 168;
  static constexpr int NP = T::NP, NQ = T::NQ, NF = T::NF, NPH = T::NPH, NFH = T::NFH, QH = T::QH;
  static constexpr int N1 = T::N1, N2 = T::N2, N3 = T::N3, K1H = T::K1H, K1 = T::K1;
  static constexpr int KQ = up8(QH), KV = 2 * KQ;           // points as K slots
  static constexpr int KF = up8(NFH), KB = 2 * KF;          // face points as K slots
  static constexpr int CA = max2(max2(K1, KV), KB) / 2, ND = T::ND;
  static_assert(T::NB1 == 1 && ND + kDigits * CA <= SUBCOLS, "TMEM columns of a group");
  // image of k_adj_split: the first six tables, then their exponents; the seventh
  // (k_adj_sum_split) and its exponent after it
  static constexpr int bytes(int n, int k) { return kDigits * n * k * 2; }
  static constexpr int oU = 0, oT = oU + bytes(N1, K1), oR = oT + bytes(N3, K1), oS = oR + bytes(N1, K1),
                       oG = oS + bytes(N1, K1), oV = oG + bytes(N3, K1), oEx = oV + bytes(N2, KV);
  static constexpr int IMG = oEx + 32;
  static constexpr int oB = IMG, IMGB = bytes(N2, KB) + 16, ALL = IMG + IMGB;
  static constexpr int LD = T::LD, PT = NQ * M * LD * 8;
  static constexpr int oGeo = 3 * PT, oMx = oGeo + 4 * 32 * 8;
  static constexpr int SUB = oMx + 5 * 128 * 4;
  static constexpr int oSub = (IMG + 127) / 128 * 128, oBar = oSub + SUBS * SUB, SMEM = oBar + 64;
  static constexpr int oSubB = (IMGB + 127) / 128 * 128, oBarB = oSubB + SUBS * 1024, SMEMB = oBarB + 64;
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

// One tile group of a CTA: its place, barriers and TMEM columns (as in
// k_element_split, whose comments give the reasons).
struct Group {
  int sub, tid, warp, lane, quarter, h, row, rel, rm, subs;
  uint32_t mbar, phase, tmem, tD;
  volatile int *fail;
  int *turn, *err;
  bool in_flight;
  int waits;

  __device__ __forceinline__ bool sync() const {
    bar_sync(1 + sub, kSubThreads);
    return fail[sub] == 0;
  }
  __device__ __forceinline__ bool operands_ready() const {
    tc::wait_st();
    tc::fence_before_sync();
    const bool ok = sync();
    tc::fence_after_sync();
    return ok;
  }
  // every thread has read the accumulator
  __device__ __forceinline__ bool results_read() const {
    tc::fence_before_sync();
    const bool ok = sync();
    tc::fence_after_sync();
    return ok;
  }
  __device__ __forceinline__ bool wait_mma() {
    in_flight = true;
    const bool done = tc::mbar_wait_sleep(mbar, phase, kSplitWaitNs, kSplitSuspendNs) && !expire_wait(err, waits++);
    if (!done) {
      fail[sub] = 1;
      atomicOr(err, kErrTimeout);
    }
    phase ^= 1u;
    tc::fence_after_sync();
    return done;
  }
  __device__ __forceinline__ uint32_t pair_max(uint32_t *s, uint32_t v) const {
    s[h * 128 + row] = v;
    bar_sync(1 + subs + sub * 4 + quarter, 64);
    return max(v, s[(h ^ 1) * 128 + row]);
  }
  // CTA start: TMEM, mbarriers, the image's bulk copy; false: the copy's wait expired
  __device__ __forceinline__ bool begin(unsigned char *sm, int oBar, int nsubs, int subcols, const unsigned char *img,
                                        uint32_t img_bytes, int *err_) {
    subs = nsubs;
    err = err_;
    sub = threadIdx.x / kSubThreads;
    tid = threadIdx.x % kSubThreads;
    warp = tid >> 5;
    lane = tid & 31;
    quarter = warp & 3;
    h = warp >> 2;
    row = quarter * 32 + lane;
    rel = row >> 2;
    rm = row & 3;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + oBar);
    uint32_t *slot = reinterpret_cast<uint32_t *>(sm + oBar + 36);
    turn = reinterpret_cast<int *>(sm + oBar + 40);
    fail = reinterpret_cast<volatile int *>(sm + oBar + 48);
    const uint32_t mbar_img = tc::smem_u32(bars + subs);
    mbar = tc::smem_u32(bars + sub);
    phase = 0;
    in_flight = false;
    waits = 0;
    if (threadIdx.x < 32) tc::tmem_alloc(tc::smem_u32(slot), 512);
    if (threadIdx.x == 0) {
      for (int i = 0; i <= subs; ++i) tc::mbar_init(tc::smem_u32(bars + i), 1);
      for (int i = 0; i < subs; ++i) fail[i] = 0;
      *turn = 0;
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    tmem = *slot + (uint32_t)(sub * subcols);
    tD = tmem + ((uint32_t)(quarter * 32) << 16);
    if (threadIdx.x == 0) {
      tc::mbar_arrive_expect_tx(mbar_img, img_bytes);
      tc::bulk_g2s(tc::smem_u32(sm), img, img_bytes, mbar_img);
    }
    const bool ok = tc::mbar_wait_sleep(mbar_img, 0, kSplitWaitNs, kSplitSuspendNs);
    if (!ok) {
      for (int i = 0; i < subs; ++i) fail[i] = 1;
      atomicOr(err, kErrTimeout);
    }
    __syncthreads();
    return ok;
  }
  __device__ __forceinline__ void end(unsigned char *sm, int oBar, bool img_ok) {
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + oBar);
    uint32_t *slot = reinterpret_cast<uint32_t *>(sm + oBar + 36);
    if (fail[sub] && in_flight) tc::mbar_wait_sleep(mbar, phase ^ 1u, kSplitWaitNs, kSplitSuspendNs);
    if (!img_ok) tc::mbar_wait_sleep(tc::smem_u32(bars + subs), 0, kSplitWaitNs, kSplitSuspendNs);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (threadIdx.x < 32) tc::tmem_dealloc(*slot, 512);
  }
};

template <int N>
__device__ __forceinline__ uint32_t max_hi(const double *v) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) m = max(m, (uint32_t)__double2hiint(v[i]) & 0x7FFFFFFFu);
  return m;
}
// this half's n values -> its K slots (KH of them) in the operand columns
template <int KH, int N>
__device__ __forceinline__ void store_half(const Group &g, uint32_t tA, int ca, const double *v, int E) {
#pragma unroll
  for (int s = 0; s < KH; s += 8) {
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = s + i < N ? v[s + i] : 0.0;
    store_digits8(tA + (uint32_t)((g.h * KH + s) / 2), ca, x, E);
  }
}
// put(i, value) for the CNT outputs of this half (level blocks of N columns)
template <int N, int CNT, class Put>
__device__ __forceinline__ void read_half(const Group &g, int xb, uint32_t nan, Put &&put) {
#pragma unroll
  for (int q = 0; q < N / 2; q += 4) {
    if (q >= CNT) break;
    float d[4][kDigits];
    load_levels4(g.tD, N, g.h * (N / 2) + q, d);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (q + i < CNT) put(q + i, from_levels(d[i], xb, nan));
  }
}

// ub = A_x(U)^T bx + A_y(U)^T by (flux_jac_t_xy) of the cotangents r, s of G_r, G_s:
// bx = g0 r + g2 s, by = g1 r + g3 s
__device__ __forceinline__ void pull_back(const double U[M], const double r[M], const double s[M], const double g[4],
                                          double gamma, double ub[M]) {
  double bx[M], by[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    bx[m] = fma(g[0], r[m], g[2] * s[m]);
    by[m] = fma(g[1], r[m], g[3] * s[m]);
  }
  flux_jac_t_xy(U, gamma, bx, by, ub);
}

template <int P, int NE, int Q>
__global__ void __launch_bounds__(Ap<P, NE, Q>::THREADS, 1)
k_adj_split(const double *__restrict__ u, const double *__restrict__ lam, double *__restrict__ uvol,
            double *__restrict__ G, double *__restrict__ Tr, const double *__restrict__ geo,
            const unsigned char *__restrict__ img, int N, double gamma, int *err) {
  using A = Ap<P, NE, Q>;
  constexpr int NP = A::NP, NQ = A::NQ, NF = A::NF, LD = A::LD, NPH = A::NPH, NFH = A::NFH, QH = A::QH, EB = 32;
  extern __shared__ __align__(1024) unsigned char sm[];
  Group g;
  const bool img_ok = g.begin(sm, A::oBar, A::SUBS, A::SUBCOLS, img, (uint32_t)A::IMG, err);
  unsigned char *mine = sm + A::oSub + g.sub * A::SUB;
  double *sU = reinterpret_cast<double *>(mine), *sR = sU + NQ * M * LD, *sS = sR + NQ * M * LD;   // [NQ][4][LD]
  double *sGeo = reinterpret_cast<double *>(mine + A::oGeo);                                    // [4][32]
  uint32_t *sMxA = reinterpret_cast<uint32_t *>(mine + A::oMx), *sMxB = sMxA + 256, *sMxG = sMxB + 256;
  const uint32_t tA = g.tD + (uint32_t)A::ND, aD = g.tmem + (uint32_t)A::ND, uB = tc::smem_u32(sm);
  const int *ex = reinterpret_cast<const int *>(sm + A::oEx);
  const int h = g.h, rel = g.rel, rm = g.rm;

  auto issue = [&](auto n, auto k, int off) {
    if (g.tid == 0) {
      gemm_digits<decltype(n)::v, decltype(k)::v>(g.tmem, aD, A::CA, uB + (uint32_t)off, true);
      tc::commit(g.mbar);
    }
  };
  struct C1 { enum { v = A::N1 }; };
  struct C2 { enum { v = A::N2 }; };
  struct C3 { enum { v = A::N3 }; };
  struct CK { enum { v = A::K1 }; };
  struct CV { enum { v = A::KV }; };

  auto tile_body = [&](int tile) -> bool {
    const int e0 = tile * EB, ecount = min(EB, N - e0);
    bool live = rel < ecount;                                // (and no wait has expired: nothing is stored after one)
    const size_t orow = ((size_t)(e0 + rel) * M + rm) * NP + h * NPH;
    double v[NPH], lb[NPH];
    const double inv = live ? geo[(size_t)(e0 + rel) * GEO + 4] : 0.0;
#pragma unroll
    for (int i = 0; i < NPH; ++i) {
      const bool on = live && h * NPH + i < NP;
      v[i] = on ? u[orow + i] : 0.0;
      lb[i] = on ? lam[orow + i] : 0.0;
    }
    if (g.warp < 4) sGeo[g.warp * 32 + g.lane] = g.lane < ecount ? geo[(size_t)(e0 + g.lane) * GEO + g.warp] : 0.0;
    else if (g.warp == 4)
#pragma unroll
      for (int m = 0; m < M; ++m) sMxG[m * 32 + g.lane] = 0u;
    // ---- u: values at the points, edge traces ----
    uint32_t mx = g.pair_max(sMxA, max_hi<NPH>(v));
    int E = row_exp(mx);
    uint32_t nan = row_nan(mx);
    store_half<A::K1H, NPH>(g, tA, A::CA, v, E);
    if (!g.operands_ready()) return false;
    issue(C1{}, CK{}, A::oU);
    g.wait_mma();
    auto to_points = [&](double *s, int xb) {
      read_half<A::N1, QH>(g, xb, nan, [&](int i, double x) {
        if (h * QH + i < NQ) s[((h * QH + i) * M + rm) * LD + rel] = x;
      });
    };
    auto to_faces = [&](double *dst, int xb) {
      double *d = dst + (size_t)(e0 + rel) * NF * M + rm;
      read_half<A::N3, NFH>(g, xb, nan, [&](int i, double x) {
        if (h * NFH + i < NF && live) d[(h * NFH + i) * M] = x;
      });
    };
    to_points(sU, E + ex[kTabU] + 5);
    if (!g.results_read()) return false;
    issue(C3{}, CK{}, A::oT);
#pragma unroll
    for (int i = 0; i < NPH; ++i) lb[i] *= inv;
    const uint32_t mxl = g.pair_max(sMxB, max_hi<NPH>(lb));
    live = g.wait_mma() && live;
    to_faces(Tr, E + ex[kTabT] + 5);
    // ---- lb: cotangents of the edge fluxes and of G_r, G_s ----
    E = row_exp(mxl);
    nan = row_nan(mxl);
    store_half<A::K1H, NPH>(g, tA, A::CA, lb, E);
    if (!g.operands_ready()) return false;
    issue(C3{}, CK{}, A::oG);
    live = g.wait_mma() && live;
    to_faces(G, E + ex[kTabG] + 5);
    if (!g.results_read()) return false;
    issue(C1{}, CK{}, A::oR);
    g.wait_mma();
    to_points(sR, E + ex[kTabR] + 5);
    if (!g.results_read()) return false;
    issue(C1{}, CK{}, A::oS);
    g.wait_mma();
    to_points(sS, E + ex[kTabS] + 5);
    tc::fence_before_sync();
    take_turn(g.turn, g.tid);
    if (!g.sync()) return false;
    tc::fence_after_sync();
    // ---- float64 pull-back, one point per warp and turn, the element across the lanes ----
    {
      uint32_t gm[M] = {0u, 0u, 0u, 0u};
      const double gg[4] = {sGeo[g.lane], sGeo[32 + g.lane], sGeo[64 + g.lane], sGeo[96 + g.lane]};
      for (int k = g.warp; k < NQ; k += kSubThreads / 32) {
        const int o = k * M * LD + g.lane;
        double U[M], r[M], s[M], ub[M];
#pragma unroll
        for (int m = 0; m < M; ++m) { U[m] = sU[o + m * LD]; r[m] = sR[o + m * LD]; s[m] = sS[o + m * LD]; }
        pull_back(U, r, s, gg, gamma, ub);
#pragma unroll
        for (int m = 0; m < M; ++m) {
          if (g.lane >= ecount) ub[m] = 0.0;
          sU[o + m * LD] = ub[m];
          gm[m] = max(gm[m], (uint32_t)__double2hiint(ub[m]) & 0x7FFFFFFFu);
        }
      }
#pragma unroll
      for (int m = 0; m < M; ++m) atomicMax(&sMxG[m * 32 + g.lane], gm[m]);
    }
    if (!g.sync()) return false;
    if (g.tid == 0) atomicExch(g.turn, 0);
    // ---- transposed interpolation ----
    mx = sMxG[rm * 32 + rel];
    E = row_exp(mx);
    nan = row_nan(mx);
    double b[QH];
#pragma unroll
    for (int i = 0; i < QH; ++i) b[i] = h * QH + i < NQ ? sU[((h * QH + i) * M + rm) * LD + rel] : 0.0;
    store_half<A::KQ, QH>(g, tA, A::CA, b, E);
    if (!g.operands_ready()) return false;
    issue(C2{}, CV{}, A::oV);
    live = g.wait_mma() && live;
    read_half<A::N2, NPH>(g, E + ex[kTabV] + 5, nan, [&](int i, double x) {
      if (h * NPH + i < NP && live) uvol[orow + i] = x;
    });
    return g.results_read();                                  // and the next tile may overwrite sGeo, sMxG
  };

  const int ntiles = (N + EB - 1) / EB;
  bool ok = img_ok && g.fail[g.sub] == 0;
  for (int tile = g.sub * (int)gridDim.x + (int)blockIdx.x; ok && tile < ntiles; tile += A::SUBS * (int)gridDim.x)
    ok = tile_body(tile);
  g.end(sm, A::oBar, img_ok);
}

template <int P, int NE, int Q>
__global__ void __launch_bounds__(Ap<P, NE, Q>::THREADS, 1)
k_adj_sum_split(const double *__restrict__ uvol, const double *__restrict__ TB, const double *X, const double *Y,
                const double *Z, double x0, double x1, double x2, double s, double *out,
                const unsigned char *__restrict__ img, int N, int *err) {
  using A = Ap<P, NE, Q>;
  constexpr int NP = A::NP, NF = A::NF, NPH = A::NPH, NFH = A::NFH, EB = 32;
  extern __shared__ __align__(1024) unsigned char sm[];
  Group g;
  const bool img_ok = g.begin(sm, A::oBarB, A::SUBS, A::SUBCOLS, img + A::oB, (uint32_t)A::IMGB, err);
  uint32_t *sMx = reinterpret_cast<uint32_t *>(sm + A::oSubB + g.sub * 1024);
  const uint32_t tA = g.tD + (uint32_t)A::ND, aD = g.tmem + (uint32_t)A::ND, uB = tc::smem_u32(sm);
  const int ex = *reinterpret_cast<const int *>(sm + A::IMGB - 16);
  const int h = g.h;

  const int ntiles = (N + EB - 1) / EB;
  auto load = [&](int tile, double *f) {
    const int e = tile * EB + g.rel;
#pragma unroll
    for (int i = 0; i < NFH; ++i)
      f[i] = tile < ntiles && e < N && h * NFH + i < NF ? TB[((size_t)e * NF + h * NFH + i) * M + g.rm] : 0.0;
  };
  double f[NFH];
  auto tile_body = [&](int tile, int next) -> bool {
    const int e = tile * EB + g.rel;
    bool live = e < N;
    const size_t o = ((size_t)e * M + g.rm) * NP + h * NPH;
    const uint32_t mx = g.pair_max(sMx, max_hi<NFH>(f));
    const int E = row_exp(mx);
    store_half<A::KF, NFH>(g, tA, A::CA, f, E);
    if (!g.operands_ready()) return false;
    if (g.tid == 0) {
      gemm_digits<A::N2, A::KB>(g.tmem, aD, A::CA, uB, true);
      tc::commit(g.mbar);
    }
    // the rest of the sum while the products run: s uvol + x0 X + x1 Y + x2 Z
    double r[NPH];
#pragma unroll
    for (int i = 0; i < NPH; ++i) {
      const bool on = live && h * NPH + i < NP;
      r[i] = on ? s * uvol[o + i] : 0.0;
      if (X && on) r[i] = fma(x0, X[o + i], r[i]);
      if (Y && on) r[i] = fma(x1, Y[o + i], r[i]);
      if (Z && on) r[i] = fma(x2, Z[o + i], r[i]);
    }
    load(next, f);
    live = g.wait_mma() && live;
    read_half<A::N2, NPH>(g, E + ex + 5, row_nan(mx), [&](int i, double x) {
      if (h * NPH + i < NP && live) out[o + i] = fma(s, x, r[i < NPH ? i : 0]);
    });
    return g.results_read();
  };
  bool ok = img_ok && g.fail[g.sub] == 0;
  const int first = g.sub * (int)gridDim.x + (int)blockIdx.x, step = A::SUBS * (int)gridDim.x;
  load(first, f);
  for (int tile = first; ok && tile < ntiles; tile += step) ok = tile_body(tile, tile + step);
  g.end(sm, A::oBarB, img_ok);
}

// The seven tables' digit blocks (k_split_tables' layout) and exponents.
template <int P, int NE, int Q>
__global__ void __launch_bounds__(256) k_adj_split_tables(DevTables tab, unsigned char *img) {
  using A = Ap<P, NE, Q>;
  constexpr int NP = A::NP, NQ = A::NQ, NF = A::NF;
  __shared__ unsigned long long mx[kAdjTabs];
  __shared__ int ex[kAdjTabs];
  if (threadIdx.x < kAdjTabs) mx[threadIdx.x] = 0ull;
  __syncthreads();
  double big[kAdjTabs] = {};
  for (int i = threadIdx.x; i < NP * NQ; i += blockDim.x) {
    big[kTabU] = fmax(big[kTabU], fabs(tab.BvT[i]));
    big[kTabR] = fmax(big[kTabR], fabs(tab.Dr[i]));
    big[kTabS] = fmax(big[kTabS], fabs(tab.Ds[i]));
  }
  for (int i = threadIdx.x; i < NP * NF; i += blockDim.x) {
    big[kTabT] = fmax(big[kTabT], fabs(tab.BfT[i]));
    big[kTabG] = fmax(big[kTabG], fabs(tab.Lf[i]));
  }
  big[kTabV] = big[kTabU];
  big[kTabB] = big[kTabT];
  for (int t = 0; t < kAdjTabs; ++t) {
    for (int o = 16; o > 0; o >>= 1) big[t] = fmax(big[t], __shfl_down_sync(0xFFFFFFFFu, big[t], o));
    if ((threadIdx.x & 31) == 0) atomicMax(&mx[t], (unsigned long long)__double_as_longlong(big[t]));
  }
  __syncthreads();
  if (threadIdx.x < kAdjTabs) {
    int e;
    frexp(__longlong_as_double((long long)mx[threadIdx.x]), &e);
    ex[threadIdx.x] = e;
    if (blockIdx.x == 0)
      *reinterpret_cast<int *>(threadIdx.x == kTabB ? img + A::ALL - 16 : img + A::oEx + 4 * threadIdx.x) = e;
  }
  if (blockIdx.x == 0 && threadIdx.x >= kAdjTabs && threadIdx.x < kAdjTabs + 2)
    reinterpret_cast<int *>(img + A::oEx)[threadIdx.x - 1] = 0;
  if (blockIdx.x == 0 && threadIdx.x >= 16 && threadIdx.x < 19)
    reinterpret_cast<int *>(img + A::ALL - 16)[threadIdx.x - 15] = 0;
  __syncthreads();
  // slot s of 2 w slots in halves -> item (cnt to a half, n in all), -1: none
  auto item = [](int s, int w, int cnt, int n) {
    const int hh = s / w, x = s % w;
    return x < cnt && hh * cnt + x < n ? hh * cnt + x : -1;
  };
  const int at = blockIdx.x * blockDim.x + threadIdx.x, all = gridDim.x * blockDim.x;
  // rows digit * n + output slot, K-major; value(output, input)
  auto fill = [&](int off, int t, int n, int k, int cn, int nn, int ck, int nk, auto value) {
    for (int i = at; i < kDigits * n * k; i += all) {
      const int r = i / k, kk = i % k, digit = r / n;
      const int o = item(r % n, n / 2, cn, nn), x = item(kk, k / 2, ck, nk);
      const double b = o >= 0 && x >= 0 ? value(o, x) : 0.0;
      *reinterpret_cast<__half *>(img + off + tc::kmaj16(r, kk, k)) = __float2half_rn(table_digit(b, ex[t], digit));
    }
  };
  fill(A::oU, kTabU, A::N1, A::K1, A::QH, NQ, A::NPH, NP, [&](int k, int j) { return tab.BvT[j * NQ + k]; });
  fill(A::oT, kTabT, A::N3, A::K1, A::NFH, NF, A::NPH, NP, [&](int q, int j) { return tab.BfT[j * NF + q]; });
  fill(A::oR, kTabR, A::N1, A::K1, A::QH, NQ, A::NPH, NP, [&](int k, int j) { return tab.Dr[k * NP + j]; });
  fill(A::oS, kTabS, A::N1, A::K1, A::QH, NQ, A::NPH, NP, [&](int k, int j) { return tab.Ds[k * NP + j]; });
  fill(A::oG, kTabG, A::N3, A::K1, A::NFH, NF, A::NPH, NP, [&](int q, int j) { return tab.Lf[q * NP + j]; });
  fill(A::oV, kTabV, A::N2, A::KV, A::NPH, NP, A::QH, NQ, [&](int j, int k) { return tab.BvT[j * NQ + k]; });
  fill(A::oB, kTabB, A::N2, A::KB, A::NPH, NP, A::NFH, NF, [&](int j, int q) { return tab.BfT[j * NF + q]; });
}

template <int P, int NE, int Q>
int adj_tables_pq(dg_mesh *m) {
  cudaError_t e = cudaMalloc((void **)&m->adj_split_img, Ap<P, NE, Q>::ALL);
  if (e != cudaSuccess) return (int)e;
  k_adj_split_tables<P, NE, Q><<<64, 256>>>(m->tab, m->adj_split_img);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return (int)e;
}

template <int P, int NE, int Q>
int adj_attrs(const dg_mesh *m) {
  static PerDevice attr_set;
  if (attr_set.test(m->device)) return (int)cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_adj_split<P, NE, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Ap<P, NE, Q>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_adj_sum_split<P, NE, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             Ap<P, NE, Q>::SMEMB);
  if (e == cudaSuccess) attr_set.set(m->device);
  return (int)e;
}

template <int P, int NE, int Q>
int adj_element_pq(const dg_mesh *m, const double *u, const double *lam, double *uvol, double *G, double *T,
                   cudaStream_t s) {
  using A = Ap<P, NE, Q>;
  if (int e = adj_attrs<P, NE, Q>(m)) return e;
  const int64_t ntiles = (m->N + 31) / 32;
  k_adj_split<P, NE, Q><<<(int)(ntiles < m->num_sms ? ntiles : m->num_sms), A::THREADS, A::SMEM, s>>>(
      u, lam, uvol, G, T, m->geo, m->adj_split_img, (int)m->N, m->gamma, m->err_flag);
  return (int)cudaGetLastError();
}

template <int P, int NE, int Q>
int adj_sum_pq(const dg_mesh *m, const double *uvol, const double *TB, const double *X, const double *Y,
               const double *Z, double x0, double x1, double x2, double s, double *out, cudaStream_t st) {
  using A = Ap<P, NE, Q>;
  if (int e = adj_attrs<P, NE, Q>(m)) return e;
  const int64_t ntiles = (m->N + 31) / 32;
  k_adj_sum_split<P, NE, Q><<<(int)(ntiles < m->num_sms ? ntiles : m->num_sms), A::THREADS, A::SMEMB, st>>>(
      uvol, TB, X, Y, Z, x0, x1, x2, s, out, m->adj_split_img, (int)m->N, m->err_flag);
  return (int)cudaGetLastError();
}

}  // namespace

#define DISPATCH(CALL)                                                                             \
  do {                                                                                             \
    const bool sym = m->rule == DG_RULE_SYMMETRIC;                                                 \
    if (m->p == 1 && m->ne == 2) return sym ? CALL(1, 2, sym_points(1)) : CALL(1, 2, 0);           \
    if (m->p == 2 && m->ne == 3) return sym ? CALL(2, 3, sym_points(2)) : CALL(2, 3, 0);           \
    if (m->p == 3 && m->ne == 4) return sym ? CALL(3, 4, sym_points(3)) : CALL(3, 4, 0);           \
    if (m->p == 3 && m->ne == 3) return sym ? CALL(3, 3, sym_points(3)) : CALL(3, 3, 0);           \
  } while (0)

int adj_split_tables(dg_mesh *m) {
  if (!m->split_img) return (int)cudaSuccess;
#define CALL(P, NE, Q) adj_tables_pq<P, NE, Q>(m)
  DISPATCH(CALL);
#undef CALL
  return (int)cudaSuccess;
}

int launch_adj_split(const dg_mesh *m, const double *u, const double *lam, double *uvol, double *G, double *T,
                     void *stream) {
  cudaStream_t s = (cudaStream_t)stream;
#define CALL(P, NE, Q) adj_element_pq<P, NE, Q>(m, u, lam, uvol, G, T, s)
  DISPATCH(CALL);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

int launch_adj_sum_split(const dg_mesh *m, const double *uvol, const double *TB, const double *X, const double *Y,
                         const double *Z, double x0, double x1, double x2, double s, double *out, void *stream) {
  cudaStream_t st = (cudaStream_t)stream;
#define CALL(P, NE, Q) adj_sum_pq<P, NE, Q>(m, uvol, TB, X, Y, Z, x0, x1, x2, s, out, st)
  DISPATCH(CALL);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

}  // namespace dg
