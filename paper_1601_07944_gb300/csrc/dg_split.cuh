/*
 * dg_split.cuh -- the float64 element kernel of large meshes, k_element_split:
 * the dense contractions of a stage leave the float64 pipe and run, as exact
 * integer products, on the tensor cores (tcgen05.mma kind::f16).
 *
 * Why.  This GPU issues 2 float64 FMAs per clock and SM, 1/64 of its float32 and
 * integer rate, and the sum-factorised kernel (k_element_sf) is bound by that
 * pipe alone.  Here only the Euler flux at the points (23 float64 operations) and
 * the stage update (1-3 per coefficient) use it.
 *
 * How.  A float64 operand row x_0..x_{K-1} (one element, one variable) is taken
 * relative to its largest exponent as 60-bit integers, X_k = x_k 2^(1081-E)
 * truncated (E the largest biased exponent of the row, |X_k| <= 2^59), and cut into
 * six signed digits of ten bits, X = sum_i d_i 2^(10 (5-i)), |d_i| <= 512: integers
 * that float16 holds exactly.  The tables are cut alike, once per mesh, relative to
 * the largest entry of each table.  With level L the sum of all digit products
 * d_i e_j with i + j = L,
 *     sum_k x_k b_k = 2^s sum_L D_L 2^(-10 L),
 * and every D_L is a sum of integers of at most 2^18 that the tensor core forms in
 * float32: exact below 2^24.  Levels 0 and 1 stay below that for any operand (by 5 % at
 * p = 5; tests/test_split_digits.py bounds every table), levels 2 and 3 too except in
 * GEMM 2: level 2 there at p = 4 and 5 (up to 1.2 and 1.7 times 2^24), level 3 from p = 3
 * on.  To pass it an operand has to line up with a table column digit by digit: sums of
 * random sign stay below by ten standard deviations.  (Levels 4 and 5 need not be exact.)
 * Levels above 5 are dropped.  The result is then the exact product to about 2^-58 of
 * (largest input) x (largest table entry), rounded once to float64: closer than the
 * float64 sums it replaces, whose every partial sum is rounded to 2^-53.  (Such an operand
 * would lose a unit of level 2, 2^-38 of the largest product, or of level 3, 2^-48, at
 * each of GEMM 2's K steps.)
 *
 * Measured (256 x 256 mesh, 131,072 elements, one launch of a stage, k_element_sf
 * -> here): p = 1 0.108 -> 0.082 ms, p = 2 0.265 -> 0.127, p = 3 0.498 -> 0.182,
 * p = 4 0.907 -> 0.320, p = 5 1.49 -> 0.463; the symmetric rules 0.101 -> 0.079,
 * 0.242 -> 0.114, 0.593 -> 0.169, 1.08 -> 0.224, 2.07 -> 0.386; the traces alone
 * (mode 2) 0.043 -> 0.032 (p = 2), 0.074 -> 0.039 (p = 3), 0.271 -> 0.074 (p = 5).
 * The float64 pipe is 60-70 % busy; the rest is the latency of a group's phases,
 * which the other groups fill only in part.  The error of the right-hand side
 * against an 80-bit reference falls by 1.5 (p = 2) to 2.9 (p = 5).
 *
 * A row whose largest value is below 2^-959 is taken relative to that number: its
 * results then have an error of 2^-1017 of the largest table entry, near the end of the
 * normal range, instead of one relative to themselves.  A row whose largest value is
 * not finite, or is 2^1007 or more, gives NaN (a sum of 90 products with table entries
 * below 2^8 then stays below the largest float64).
 *
 * Layout.  A tile is 32 elements = 128 rows (row = 4 e + m) = 128 TMEM lanes.  A
 * group of 256 threads works on a tile, two threads (halves h = 0, 1) per row:
 * each cuts half of the row's K slots and reassembles half of its outputs.  A CTA
 * holds three groups (two at p = 5: shared memory) with barriers of their own that
 * share one copy of the tables, so that one group's integer phases run beside
 * another's flux phase (split_groups, take_turn).  Per tile:
 *   GEMM 1  U  = c Phi           interpolation to the volume points
 *           float64 Euler flux, one (element, point) item per thread
 *   GEMM 2  D  = [G_r | G_s | lifted fluxes] [Dr; Ds; Lf]   projection and lift
 *           float64 stage update
 *   GEMM 3  T  = c_new Phi_f     edge traces of the new state
 * (mode 2: GEMM 3 alone, on the input.)  The digits of A are TMEM columns written
 * by the row's threads (tcgen05.st); digit i of A multiplies the digit blocks
 * B_0..B_{5-i} side by side in shared memory in one MMA per K step, whose columns
 * are the levels i..5.
 */
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "dg_device.cuh"
#include "dg_internal.h"
#include "dg_tcgen05.cuh"

namespace dg {
namespace {

constexpr int kSubThreads = 256;                     // threads of a tile group
constexpr int kDigits = 6;
constexpr uint64_t kSplitWaitNs = 2000000000ull;     // 2 s per MMA batch before giving up
constexpr uint32_t kSplitSuspendNs = 1000;

__host__ __device__ constexpr int up8(int x) { return (x + 7) / 8 * 8; }
__host__ __device__ constexpr int up16(int x) { return (x + 15) / 16 * 16; }
constexpr int half_up(int x) { return (x + 1) / 2; }
constexpr int max2(int a, int b) { return a > b ? a : b; }
// accumulator columns of a GEMM with n columns per level: digit i's MMA writes
// up16((6 - i) n) columns from column i n on (those past 6 n are never read)
constexpr int level_cols(int n) {
  int c = 0;
  for (int i = 0; i < kDigits; ++i) c = max2(c, i * n + up16((kDigits - i) * n));
  return c;
}

// Tile groups per CTA: three (80 registers a thread, 168 TMEM columns a group, so
// that GEMM 2 takes its operand in two to five batches) against two (128 registers):
// p = 2 0.128 against 0.173 ms, p = 3 0.187 against 0.221, p = 4 0.331 against
// 0.372.  At p = 5 the point buffers of three groups do not fit in shared memory.
__host__ __device__ constexpr int split_groups(int p) { return p <= 4 ? 3 : 2; }

template <int P, int NE, int Q>
struct Sp {
  using C = Cfg<P, NE, Q>;
  static constexpr int NP = C::NP, NQ = C::NQ, NF = C::NF;
  static constexpr int EB = 32, ROWS = 128;
  static constexpr int SUBS = split_groups(P), THREADS = SUBS * kSubThreads;   // tile groups per CTA
  static constexpr int ROOM = SUBS == 2 ? 256 : 168;        // TMEM columns a group may take
  // outputs and K slots go in halves to a row's two threads
  static constexpr int NPH = half_up(NP), NFH = half_up(NF);
  static constexpr int NB1 = NQ > 16 ? 2 : 1;               // GEMM 1 in batches of points (TMEM columns)
  static constexpr int QB = (NQ + NB1 - 1) / NB1, QH = half_up(QB);
  static constexpr int N1 = up8(2 * QH), N2 = up8(2 * NPH), N3 = up8(2 * NFH);
  static constexpr int K1H = up8(NPH), K1 = 2 * K1H;        // GEMMs 1 and 3
  static constexpr int KH = NQ + NFH;                       // GEMM 2: half 0 G_r, half 1 G_s, and half of the fluxes each
  static constexpr int KROOM = (ROOM - max2(max2(level_cols(N1), level_cols(N2)), level_cols(N3))) / kDigits / 8 * 8;
  static constexpr int NB2 = (up8(KH) + KROOM - 1) / KROOM; // GEMM 2 in batches of K slots
  static constexpr int KC = up8((KH + NB2 - 1) / NB2), K2 = 2 * KC;
  // TMEM columns of a group: the accumulator [0, ND), then the six digit planes
  static constexpr int ND = max2(max2(level_cols(N1), level_cols(N2)), level_cols(N3));
  static constexpr int CA = max2(K1, K2) / 2;
  static constexpr int SUBCOLS = SUBS == 2 ? (ND + kDigits * CA <= 128 ? 128 : 256) : ROOM;
  static_assert(ND + kDigits * CA <= SUBCOLS, "TMEM columns of a group");
  static constexpr int COLS = SUBS == 2 ? 2 * SUBCOLS : 512;
  // shared memory: table image (digit blocks, then the three table exponents)
  static constexpr int B1B = kDigits * N1 * K1 * 2, B2B = kDigits * N2 * K2 * 2, B3B = kDigits * N3 * K1 * 2;
  static constexpr int oB1 = 0, oB2 = oB1 + NB1 * B1B, oB3 = oB2 + NB2 * B2B, oEx = oB3 + B3B;
  static constexpr int IMG = oEx + 16;
  // per group: point values [NQ][4][LD] (element fastest; LD = 36 spreads the four
  // variables' rows over the banks), U then G_r in place, and G_s
  static constexpr int LD = 36;
  static constexpr int PT = NQ * M * LD * 8;
  static constexpr int oG = 2 * PT;                         // geometry [NG][32]
  static constexpr int NG = 10;
  static constexpr int oMx = oG + NG * 32 * 8;              // row exponents: 2 x [2][128], [4][32]
  static constexpr int SUB = oMx + 5 * 128 * 4;
  static constexpr int oSub = (IMG + 127) / 128 * 128;
  static constexpr int oBar = oSub + SUBS * SUB;      // mbarriers: groups, image; TMEM slot; failure flags
  static constexpr int SMEM = oBar + 64;
  static_assert(SMEM <= 227 * 1024, "shared memory");
  static_assert(2 * PT >= ROWS * NP * 8, "mode 2 stages its tile in the point buffers");
};

// ---- digits ---------------------------------------------------------------

// biased exponent that a row's values are taken relative to: 64 at least, so that the
// digits of a zero (exponent 0, its leading bit taken as set) are shifted out
__device__ __forceinline__ int row_exp(uint32_t hi_max) { return max((int)(hi_max >> 20), 64); }
// ones in the exponent for a row out of range (from_levels)
__device__ __forceinline__ uint32_t row_nan(uint32_t hi_max) { return hi_max >= (2030u << 20) ? 0x7FF80000u : 0u; }

// x 2^(1081 - E) truncated, plus 512 in every digit: the digits + 512, ten bits each
// (the top one eleven)
__device__ __forceinline__ void to_fixed(double x, int E, uint32_t &lo, uint32_t &hi) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7FFu);
  const int d = min(E - e, 63);
  const uint32_t mh = (h & 0xFFFFFu) | 0x100000u;
  unsigned long long X = ((unsigned long long)__funnelshift_l(l, mh, 6) << 32) | (l << 6);
  X >>= d;
  const long long s = (long long)((int)h >> 31);
  constexpr unsigned long long BIAS = 512ull * ((1ull << 50) + (1ull << 40) + (1ull << 30) + (1ull << 20) + (1ull << 10) + 1ull);
  X = (X ^ (unsigned long long)s) + (BIAS - (unsigned long long)s);
  lo = (uint32_t)X;
  hi = (uint32_t)(X >> 32);
}

// digits + 512 of two values -> two float16 digits (low half: the first value)
__device__ __forceinline__ uint32_t pack_digit(uint32_t a, uint32_t b, uint32_t mask) {
  const uint32_t w = (__byte_perm(a, b, 0x5410) & mask) + 0x64006400u;   // 1024 + digit + 512
  __half2 v = __hsub2(*reinterpret_cast<const __half2 *>(&w), __half2half2(__ushort_as_half(0x6600)));
  return *reinterpret_cast<const uint32_t *>(&v);
}

// eight values -> four columns of each digit plane of this thread's TMEM lane
__device__ __forceinline__ void make_digits8(uint32_t w[kDigits][4], const double *v, int E) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t al, ah, bl, bh;
    to_fixed(v[2 * c], E, al, ah);
    to_fixed(v[2 * c + 1], E, bl, bh);
    constexpr uint32_t MK = 0x03FF03FFu;
    w[0][c] = pack_digit(ah >> 18, bh >> 18, 0x07FF07FFu);
    w[1][c] = pack_digit(ah >> 8, bh >> 8, MK);
    w[2][c] = pack_digit(__funnelshift_r(al, ah, 30), __funnelshift_r(bl, bh, 30), MK);
    w[3][c] = pack_digit(al >> 20, bl >> 20, MK);
    w[4][c] = pack_digit(al >> 10, bl >> 10, MK);
    w[5][c] = pack_digit(al, bl, MK);
  }
}
__device__ __forceinline__ void store_digits8(uint32_t tA, int ca, const double *v, int E) {
  uint32_t w[kDigits][4];
  make_digits8(w, v, E);
#pragma unroll
  for (int i = 0; i < kDigits; ++i) tc::st4(tA + (uint32_t)(i * ca), w[i]);
}

// sum_L D_L 2^(-10 L) with the row's and the table's exponents -> float64, rounded
// once.  xb = E + table exponent + 5: the result's biased exponent is xb + 1 - clz, at
// least 7 + table exponent.
// nan: all ones in the exponent where the row was out of range.
__device__ __forceinline__ double from_levels(const float *d, int xb, uint32_t nan) {
  // (level 5 joins level 4 in float32: the sum's rounding is below level 5's leading bits)
  long long V = (long long)__float2int_rn(fmaf(d[5], 0x1p-10f, d[4]));
  V += (long long)__float2int_rn(d[3]) * (1 << 10);
  V += (long long)__float2int_rn(d[2]) * (1 << 20);
  V += (long long)__float2int_rn(d[1]) * (1 << 30);
  V += (long long)((unsigned long long)(long long)__float2int_rn(d[0]) << 40);
  const long long s = V >> 63;
  const unsigned long long a = (unsigned long long)((V ^ s) - s);
  const int z = __clzll((long long)a);
  const unsigned long long n = a << (z & 63);
  unsigned long long b = (n >> 11) + ((n >> 10) & 1ull);          // 53 bits, rounded to nearest
  uint32_t hi = (uint32_t)(b >> 32) + ((uint32_t)(xb - z) << 20); // the leading bit adds one to the exponent
  hi = a == 0ull ? 0u : hi;
  hi |= ((uint32_t)(s >> 32) & 0x80000000u) | nan;
  return __hiloint2double((int)hi, (int)(uint32_t)b);
}

// the six levels of four consecutive outputs (accumulator columns col..col+3 of
// level blocks of n columns)
__device__ __forceinline__ void load_levels4(uint32_t tD, int n, int col, float d[4][kDigits]) {
  float t[kDigits][4];
#pragma unroll
  for (int L = 0; L < kDigits; ++L) tc::ld4(tD + (uint32_t)(L * n + col), t[L]);
  tc::wait_ld();
#pragma unroll
  for (int L = 0; L < kDigits; ++L)
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i][L] = t[L][i];
}

// D = sum over digits and K steps of digit i of A (TMEM columns a + i ca) against
// the digit blocks B_0..B_{5-i} (shared memory, n rows each, K columns)
template <int N, int K>
__device__ __forceinline__ void gemm_digits(uint32_t d, uint32_t a, int ca, uint32_t b, bool first) {
#pragma unroll
  for (int i = 0; i < kDigits; ++i)
#pragma unroll
    for (int s = 0; s < K / 16; ++s)
      tc::mma_f16_ts(d + (uint32_t)(i * N), a + (uint32_t)(i * ca + s * 8), tc::desc16(b + (uint32_t)(s * 256), K),
                     tc::idesc_f16(128, up16((kDigits - i) * N)), (i == 0 && s == 0 && first) ? 0u : 1u);
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// One group of the CTA in the float64 phase at a time: the float64 pipe serves one
// group as fast as two, and taking turns keeps the groups out of step, so that
// one's integer phases run beside another's flux (two groups, p = 3: 0.221 against
// 0.274 ms without turns; three groups: 0.202, two of them at once 0.214).  A wait
// that does not end soon goes ahead (the order is for speed only); the holder sets
// *turn to 0 after the phase.
__device__ __forceinline__ void take_turn(int *turn, int tid) {
  if (tid != 0) return;
  for (int i = 0; i < 400; ++i) {
    if (atomicCAS(turn, 0, 1) == 0) break;
    __nanosleep(64);
  }
}

// -x/2 of a normal x on the bit pattern (a float64 multiply would take a slot of
// the float64 pipe)
__device__ __forceinline__ double neg_half_bits(double x) {
  return __hiloint2double((__double2hiint(x) ^ (int)0x80000000) - 0x00100000, __double2loint(x));
}

// Euler flux of U along two directions a, b (ga, gb = (gamma - 1) times them):
// 20 float64 operations (the reciprocal in integers).  False if the state is not physical.
// FIXED_RECIP: the reciprocal in integers (p >= 4: 0.469 against 0.517 ms at p = 5; at
// p <= 3, with 80 registers, it costs more than the three float64 operations).
template <bool FIXED_RECIP>
__device__ __forceinline__ bool flux_dirs(const double U[M], double ax, double ay, double bx, double by, double gax,
                                          double gay, double gbx, double gby, double g1, double Fa[M], double Fb[M]) {
  const double inv = FIXED_RECIP ? fx::recip_fixed(U[0]) : recip3(U[0]);
  const double P = fma(fma(U[1], U[1], U[2] * U[2]), neg_half_bits(inv), U[3]);     // p / (gamma - 1)
  const double Ep = fma(g1, P, U[3]);
  {
    const double mn = fma(U[1], ax, U[2] * ay), vd = mn * inv;
    Fa[0] = mn; Fa[1] = fma(U[1], vd, P * gax); Fa[2] = fma(U[2], vd, P * gay); Fa[3] = Ep * vd;
  }
  {
    const double mn = fma(U[1], bx, U[2] * by), vd = mn * inv;
    Fb[0] = mn; Fb[1] = fma(U[1], vd, P * gbx); Fb[2] = fma(U[2], vd, P * gby); Fb[3] = Ep * vd;
  }
  return positive_finite(U[0]) & positive_finite(P);
}

// edge fluxes of half H of a row's points in the element's order, from its three
// edges; orient negates those of the edges whose left element this is (the flux
// leaves it), on the sign bits
template <int NE, int NFH, int H>
__device__ __forceinline__ void load_edge_fluxes(const double *__restrict__ fhat, const int *ef, int rm, bool live,
                                                 int64_t F, int *err, double *f) {
#pragma unroll
  for (int i = 0; i < NFH; ++i) {
    const int qk = H * NFH + i, q = qk / NE, k = qk - q * NE;
    f[i] = 0.0;
    if (qk < 3 * NE && live) {
      const int64_t fi = checked(ef[q] >> 1, F, err);
      f[i] = fhat[((size_t)fi * NE + ((ef[q] & 1) ? NE - 1 - k : k)) * M + rm];
    }
  }
}
template <int NE, int NFH, int H>
__device__ __forceinline__ void orient_edge_fluxes(uint32_t left, double *f) {
#pragma unroll
  for (int i = 0; i < NFH; ++i) {
    const int qk = H * NFH + i, q = qk / NE;
    if (qk < 3 * NE)
      f[i] = __hiloint2double(__double2hiint(f[i]) ^ (int)((left << (31 - q)) & 0x80000000u), __double2loint(f[i]));
  }
}

// TRACES: mode 2, in an instantiation of its own (its tile held ahead in registers
// would weigh on the other modes)
template <int P, int NE, int Q, bool TRACES>
__global__ void __launch_bounds__(Sp<P, NE, Q>::THREADS, 1)
k_element_split(const double *c, const double *u0, double *out, double *__restrict__ trace_out,
                const double *__restrict__ fhat, const double *__restrict__ geo,
                const int32_t *__restrict__ elem_face, const unsigned char *__restrict__ img, DevTables tab, int N, int64_t F,
                StageUpdate su, int mode, double gamma, double *__restrict__ copy, int *err) {
  using T = Sp<P, NE, Q>;
  constexpr int NP = T::NP, NQ = T::NQ, NF = T::NF, EB = T::EB, LD = T::LD, NPH = T::NPH, NFH = T::NFH;
  extern __shared__ __align__(1024) unsigned char sm[];
  const int sub = threadIdx.x / kSubThreads, tid = threadIdx.x % kSubThreads;
  const int warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, h = warp >> 2;               // this warp's TMEM lanes; its half of the row's work
  const int row = quarter * 32 + lane, rel = row >> 2, rm = row & 3;
  unsigned char *mine = sm + T::oSub + sub * T::SUB;
  double *sU = reinterpret_cast<double *>(mine);             // [NQ][4][LD] U, then G_r
  double *sS = reinterpret_cast<double *>(mine + T::PT);     // [NQ][4][LD] G_s
  double *sGeo = reinterpret_cast<double *>(mine + T::oG);   // [NG][32]
  uint32_t *sMxA = reinterpret_cast<uint32_t *>(mine + T::oMx);   // [2][128] halves' largest high words
  uint32_t *sMxB = sMxA + 256;                               // the same, for the new state
  uint32_t *sMxG = sMxB + 256;                               // [4][32] largest high word of the flux rows
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm + T::oBar);
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + T::oBar + 36);
  volatile int *fail = reinterpret_cast<volatile int *>(sm + T::oBar + 48);
  int *turn = reinterpret_cast<int *>(sm + T::oBar + 40);
  const uint32_t mbar = tc::smem_u32(bars + sub), mbar_img = tc::smem_u32(bars + T::SUBS);

  // ---- once per CTA: TMEM, mbarriers, the table image ----
  if (threadIdx.x < 32) tc::tmem_alloc(tc::smem_u32(slot), T::COLS);
  if (threadIdx.x == 0) {
    for (int i = 0; i <= T::SUBS; ++i) tc::mbar_init(tc::smem_u32(bars + i), 1);
    for (int i = 0; i < T::SUBS; ++i) fail[i] = 0;
    *turn = 0;
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot + (uint32_t)(sub * T::SUBCOLS);
  if (threadIdx.x == 0) {
    tc::mbar_arrive_expect_tx(mbar_img, (uint32_t)T::IMG);
    tc::bulk_g2s(tc::smem_u32(sm), img, (uint32_t)T::IMG, mbar_img);
  }
  const bool img_ok = tc::mbar_wait_sleep(mbar_img, 0, kSplitWaitNs, kSplitSuspendNs);
  if (!img_ok) {
    for (int i = 0; i < T::SUBS; ++i) fail[i] = 1;
    atomicOr(err, kErrTimeout);
  }
  __syncthreads();
  const uint32_t tLane = (uint32_t)(quarter * 32) << 16;
  const uint32_t tD = tmem + tLane, tA = tD + (uint32_t)T::ND, aD = tmem + (uint32_t)T::ND;
  const uint32_t uB = tc::smem_u32(sm);
  const int *ex = reinterpret_cast<const int *>(sm + T::oEx);
  const double g1 = gamma - 1.0;
  uint32_t phase = 0;
  bool in_flight = false;

  auto sub_sync = [&]() -> bool {                            // false: a wait of this group expired
    bar_sync(1 + sub, kSubThreads);
    return fail[sub] == 0;
  };
  auto operands_ready = [&]() -> bool {
    tc::wait_st();
    tc::fence_before_sync();
    const bool ok = sub_sync();
    tc::fence_after_sync();
    return ok;
  };
  int waits = 0;
  auto mma_wait = [&]() -> bool {                            // false: expired, the accumulator is not to be used
    in_flight = true;
    const bool done = tc::mbar_wait_sleep(mbar, phase, kSplitWaitNs, kSplitSuspendNs) && !expire_wait(err, waits++);
    if (!done) {
      fail[sub] = 1;
      atomicOr(err, kErrTimeout);
    }
    phase ^= 1u;
    tc::fence_after_sync();
    return done;
  };
  // the larger of the two halves' values (a barrier of the row's two warps)
  auto pair_max = [&](uint32_t *s, uint32_t v) -> uint32_t {
    s[h * 128 + row] = v;
    bar_sync(1 + T::SUBS + sub * 4 + quarter, 64);
    return max(v, s[(h ^ 1) * 128 + row]);
  };
  // this half's NPH values -> A columns of GEMMs 1 and 3
  auto store_modes = [&](const double *v, int E) {
#pragma unroll
    for (int s = 0; s < T::K1H; s += 8) {
      double x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = s + i < NPH ? v[s + i] : 0.0;
      store_digits8(tA + (uint32_t)((h * T::K1H + s) / 2), T::CA, x, E);
    }
  };

  const int ntiles = (N + EB - 1) / EB;
  const bool need_u0 = mode == 1 && su.a0 != 0.0;
  auto load_modes = [&](int tile, double *v) {
    const int e0 = tile * EB;
    const bool on = e0 + rel < N;
    const size_t o = ((size_t)(e0 + rel) * M + rm) * NP + h * NPH;
#pragma unroll
    for (int i = 0; i < NPH; ++i) v[i] = on && h * NPH + i < NP ? c[o + i] : 0.0;
  };
  // With three groups (80 registers a thread) the edge fluxes are loaded beside the
  // flux of the points and the modes once more for the update; with two, both at the
  // start of the tile (p = 5: 0.476 against 0.502 ms; p = 3: 0.187 against 0.193).
  constexpr bool LATE = T::SUBS == 3;
  // a tile's edges and (a component per warp, the element across the lanes)
  // geometry, loaded ahead of it
  double geo_n = 0.0;
  int ef[3] = {0, 0, 0};
  auto edge_fluxes = [&](double *fl, bool live) {
    if (h == 0) load_edge_fluxes<NE, NFH, 0>(fhat, ef, rm, live, F, err, fl);
    else load_edge_fluxes<NE, NFH, 1>(fhat, ef, rm, live, F, err, fl);
  };
  auto load_inputs = [&](int tile) {
    const int e0 = tile * EB;
    const bool on = tile < ntiles && e0 + rel < N;
#pragma unroll
    for (int q = 0; q < 3; ++q) ef[q] = on ? elem_face[(size_t)(e0 + rel) * 3 + q] : 0;
    geo_n = warp < 5 && tile < ntiles && e0 + lane < N ? geo[(size_t)(e0 + lane) * GEO + warp] : 0.0;
  };
  constexpr int TV = (EB * M * NP + kSubThreads - 1) / kSubThreads;
  double tv[TRACES ? TV : 1];
  auto load_tile = [&](int tile) {
#pragma unroll
    for (int x = 0; x < TV; ++x) {
      const int i = tid + x * kSubThreads;
      tv[x] = tile < ntiles && i < min(EB, N - tile * EB) * M * NP ? c[(size_t)tile * EB * M * NP + i] : 0.0;
    }
  };
  auto tile_body = [&](int tile, int next) -> bool {
    const int e0 = tile * EB, ecount = min(EB, N - e0);
    bool live = rel < ecount;                                // (and, from the last GEMM 2 on, its wait did not expire)
    const size_t orow = ((size_t)(e0 + rel) * M + rm) * NP;
    double cv[NPH], fl[NFH];
    uint32_t left = 0u;                                      // bit q: this is edge q's left element
    if constexpr (TRACES) {
      // the tile through shared memory, whole rows of it in order (c may be host
      // memory), loaded a tile ahead
#pragma unroll
      for (int x = 0; x < TV; ++x) {
        const int i = tid + x * kSubThreads;
        if (copy && i < ecount * M * NP) copy[(size_t)e0 * M * NP + i] = tv[x];
        if (i < EB * M * NP) sU[i] = tv[x];
      }
      if (!sub_sync()) return false;
      load_tile(next);
#pragma unroll
      for (int i = 0; i < NPH; ++i) cv[i] = h * NPH + i < NP ? sU[row * NP + h * NPH + i] : 0.0;
    } else {
      if constexpr (!LATE) edge_fluxes(fl, live);
#pragma unroll
      for (int q = 0; q < 3; ++q) left |= (ef[q] & 1) ? 0u : 1u << q;
      load_modes(tile, cv);
    }
    uint32_t mx = 0;
#pragma unroll
    for (int i = 0; i < NPH; ++i) mx = max(mx, (uint32_t)__double2hiint(cv[i]) & 0x7FFFFFFFu);
    mx = pair_max(sMxA, mx);
    int E = row_exp(mx);
    uint32_t nan = row_nan(mx);
    if constexpr (!TRACES) {
      store_modes(cv, E);
      if (warp < 4) {
        sGeo[warp * 32 + lane] = geo_n;
        sGeo[(4 + warp) * 32 + lane] = g1 * geo_n;
      } else if (warp == 4) {
        sGeo[8 * 32 + lane] = mode == 0 ? geo_n : su.g * su.dt * geo_n;
        if (su.out2) sGeo[9 * 32 + lane] = su.w * su.dt * geo_n;
      } else if (warp == 5) {
#pragma unroll
        for (int m = 0; m < M; ++m) sMxG[m * 32 + lane] = 0u;
      }
      if (!operands_ready()) return false;
#pragma unroll
      for (int b = 0; b < T::NB1; ++b) {
        if (tid == 0) {
          gemm_digits<T::N1, T::K1>(tmem, aD, T::CA, uB + T::oB1 + b * T::B1B, true);
          tc::commit(mbar);
        }
        mma_wait();
        // ---- U at this half's points of the batch -> point layout ----
        const int xb = E + ex[0] + 5;
#pragma unroll
        for (int g = 0; g < T::N1 / 2; g += 4) {
          if (g >= T::QH) break;
          float d[4][kDigits];
          load_levels4(tD, T::N1, h * (T::N1 / 2) + g, d);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k = b * T::QB + h * T::QH + g + i;
            if (g + i < T::QH && h * T::QH + g + i < T::QB && k < NQ)
              sU[(k * M + rm) * LD + rel] = from_levels(d[i], xb, nan);
          }
        }
        tc::fence_before_sync();
        if (b == T::NB1 - 1) take_turn(turn, tid);
        if (!sub_sync()) return false;
        tc::fence_after_sync();
      }
      // ---- float64 flux, one point per warp and turn, the element across the lanes ----
      {
        if constexpr (LATE) edge_fluxes(fl, live);
        bool phys = true;
        uint32_t gm[M] = {0u, 0u, 0u, 0u};
        double g[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] = sGeo[i * 32 + lane];
        for (int k = warp; k < NQ; k += kSubThreads / 32) {
          double *pu = sU + k * M * LD + lane, *ps = sS + k * M * LD + lane;
          double U[M], Gr[M], Gs[M];
#pragma unroll
          for (int m = 0; m < M; ++m) U[m] = pu[m * LD];
          phys &= flux_dirs<(P >= 4)>(U, g[0], g[1], g[2], g[3], g[4], g[5], g[6], g[7], g1, Gr, Gs) || lane >= ecount;
#pragma unroll
          for (int m = 0; m < M; ++m) {
            if (lane >= ecount) { Gr[m] = 0.0; Gs[m] = 0.0; }
            pu[m * LD] = Gr[m];
            ps[m * LD] = Gs[m];
            gm[m] = max(gm[m], max((uint32_t)__double2hiint(Gr[m]) & 0x7FFFFFFFu,
                                   (uint32_t)__double2hiint(Gs[m]) & 0x7FFFFFFFu));
          }
        }
        if (!phys) atomicOr(err, kErrNonPhysical);
#pragma unroll
        for (int m = 0; m < M; ++m) atomicMax(&sMxG[m * 32 + lane], gm[m]);
        if (h == 0) orient_edge_fluxes<NE, NFH, 0>(left, fl);
        else orient_edge_fluxes<NE, NFH, 1>(left, fl);
        uint32_t fm = 0;
#pragma unroll
        for (int i = 0; i < NFH; ++i) fm = max(fm, (uint32_t)__double2hiint(fl[i]) & 0x7FFFFFFFu);
        atomicMax(&sMxG[rm * 32 + rel], fm);
      }
      if (!sub_sync()) return false;
      if (tid == 0) atomicExch(turn, 0);
      // ---- GEMM 2's operand: half 0 [G_r | fluxes], half 1 [G_s | fluxes] ----
      mx = sMxG[rm * 32 + rel];
      E = row_exp(mx);
      nan = row_nan(mx);
      const double *g = (h == 0 ? sU : sS) + rm * LD + rel;
      double uv[NPH];
#pragma unroll
      for (int b = 0; b < T::NB2; ++b) {
#pragma unroll
        for (int s = 0; s < T::KC; s += 8) {
          double x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int k = b * T::KC + s + i;
            x[i] = k < NQ ? g[k * M * LD] : (k < T::KH ? fl[k - NQ] : 0.0);
          }
          uint32_t w[kDigits][4];
          make_digits8(w, x, E);
          if (b > 0 && s == 0) mma_wait();                   // the previous batch has read its operand
#pragma unroll
          for (int i = 0; i < kDigits; ++i) tc::st4(tA + (uint32_t)((h * T::KC + s) / 2 + i * T::CA), w[i]);
        }
        if (!operands_ready()) return false;
        if (tid == 0) {
          gemm_digits<T::N2, T::K2>(tmem, aD, T::CA, uB + T::oB2 + b * T::B2B, b == 0);
          tc::commit(mbar);
        }
      }
#pragma unroll
      for (int i = 0; i < NPH; ++i) uv[i] = need_u0 && live && h * NPH + i < NP ? u0[orow + h * NPH + i] : 0.0;
      if constexpr (LATE)
        if (mode != 0) load_modes(tile, cv);
      live = mma_wait() && live;
      // ---- stage update ----
      {
        const int xb = E + ex[1] + 5;
        const double kap = sGeo[8 * 32 + rel];
#pragma unroll
        for (int gq = 0; gq < T::N2 / 2; gq += 4) {
          if (gq >= NPH) break;
          float d[4][kDigits];
          load_levels4(tD, T::N2, h * (T::N2 / 2) + gq, d);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int jj = gq + i, j = h * NPH + jj;
            if (jj < NPH && j < NP) {
              const double D = from_levels(d[i], xb, nan);
              double v;
              if (mode == 0) {
                v = D * kap;
              } else {
                // a0 u0 + b0 c + g dt R with R = D / det J
                const double cj = cv[jj < NPH ? jj : 0], uj = uv[jj < NPH ? jj : 0];
                double t;
                if (su.b0 == 0.0) t = su.a0 == 1.0 ? uj : su.a0 * uj;
                else t = su.b0 == 1.0 ? cj : su.b0 * cj;
                if (need_u0 && su.b0 != 0.0) t = fma(su.a0, uj, t);
                v = fma(kap, D, t);
                if (su.out2 && live) {
                  double t2 = su.y * v;
                  if (su.x != 0.0) t2 = fma(su.x, su.acc[orow + j], t2);
                  su.out2[orow + j] = fma(sGeo[9 * 32 + rel], D, t2);
                }
              }
              if (live) out[orow + j] = v;
              cv[jj < NPH ? jj : 0] = v;
            }
          }
        }
        tc::fence_before_sync();
      }
      load_inputs(next);
      if constexpr (P == 1) {
        // p = 1: the edge traces in float64, by the sums of every other kernel that
        // writes traces (the limiter recomputes those of limited elements)
        if (trace_out) {
          double *sN = sU + row * NP + h * NPH;
#pragma unroll
          for (int i = 0; i < NPH; ++i)
            if (h * NPH + i < NP) sN[i] = cv[i];
          if (!sub_sync()) return false;
          const double *cj = sU + row * NP;
          double z[P + 2], t0, t1, t2;
          face_sums<P>(cj, tab.EChiM1, tab.EChi[0], z);
          edge_traces_unit<P, NE>(cj, z, tab.EPa, tab.EChi, h, t0, t1, t2);
          if (live) {
            double *dst = trace_out + (size_t)(e0 + rel) * NF * M + rm;
            dst[h * M] = t0;
            dst[(NE + h) * M] = t1;
            dst[(3 * NE - 1 - h) * M] = t2;
          }
        }
        return sub_sync();
      }
      if (!trace_out) return sub_sync();       // the next tile overwrites the geometry read above
      // ---- the new state's row exponents ----
      mx = 0;
#pragma unroll
      for (int i = 0; i < NPH; ++i)
        if (h * NPH + i < NP) mx = max(mx, (uint32_t)__double2hiint(cv[i]) & 0x7FFFFFFFu);
      mx = pair_max(sMxB, mx);
      E = row_exp(mx);
      nan = row_nan(mx);
    }
    // ---- GEMM 3: edge traces of the state in cv ----
    store_modes(cv, E);
    if (!operands_ready()) return false;
    if (tid == 0) {
      gemm_digits<T::N3, T::K1>(tmem, aD, T::CA, uB + T::oB3, true);
      tc::commit(mbar);
    }
    live = mma_wait() && live;
    {
      const int xb = E + ex[2] + 5;
      double *dst = trace_out + (size_t)(e0 + rel) * NF * M + rm;
#pragma unroll
      for (int gq = 0; gq < T::N3 / 2; gq += 4) {
        if (gq >= NFH) break;
        float d[4][kDigits];
        load_levels4(tD, T::N3, h * (T::N3 / 2) + gq, d);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int qk = h * NFH + gq + i;
          if (gq + i < NFH && qk < NF && live) dst[qk * M] = from_levels(d[i], xb, nan);
        }
      }
      tc::fence_before_sync();
    }
    return true;
  };

  bool ok = img_ok && fail[sub] == 0;
  const int first = sub * (int)gridDim.x + (int)blockIdx.x, step = T::SUBS * (int)gridDim.x;
  if constexpr (TRACES) load_tile(first);
  else load_inputs(first);
  for (int tile = first; ok && tile < ntiles; tile += step) ok = tile_body(tile, tile + step);
  // a wait expired: wait (bounded again) for that batch, so that no MMA writes the
  // columns freed below, and for the image's copy
  if (fail[sub] && in_flight) tc::mbar_wait_sleep(mbar, phase ^ 1u, kSplitWaitNs, kSplitSuspendNs);
  if (!img_ok) tc::mbar_wait_sleep(mbar_img, 0, kSplitWaitNs, kSplitSuspendNs);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x < 32) tc::tmem_dealloc(*slot, T::COLS);
}

// ---- the table image ------------------------------------------------------

// digit i (0 = leading) of b 2^(59 - eb), |b| < 2^eb, rounded to an integer
__device__ __forceinline__ float table_digit(double b, int eb, int i) {
  constexpr long long BIAS = 512ll * ((1ll << 50) + (1ll << 40) + (1ll << 30) + (1ll << 20) + (1ll << 10) + 1ll);
  const long long t = llrint(ldexp(b, 59 - eb)) + BIAS;
  const long long u = t >> (10 * (kDigits - 1 - i));
  return (float)((i == 0 ? u : (u & 1023)) - 512);
}

// The largest magnitude of each table (every block for itself), then the digit
// blocks of the three GEMMs in the layout the MMAs read (rows digit * n + output
// slot, K-major), spread over the grid.
template <int P, int NE, int Q>
__global__ void __launch_bounds__(256) k_split_tables(DevTables tab, unsigned char *img) {
  using T = Sp<P, NE, Q>;
  constexpr int NP = T::NP, NQ = T::NQ, NF = T::NF;
  __shared__ unsigned long long mx[3];
  __shared__ int ex[3];
  if (threadIdx.x < 3) mx[threadIdx.x] = 0ull;
  __syncthreads();
  double big[3] = {0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < NP * NQ; i += blockDim.x) {
    big[0] = fmax(big[0], fabs(tab.BvT[i]));
    big[1] = fmax(big[1], fmax(fabs(tab.Dr[i]), fabs(tab.Ds[i])));
  }
  for (int i = threadIdx.x; i < NP * NF; i += blockDim.x) {
    big[1] = fmax(big[1], fabs(tab.Lf[i]));
    big[2] = fmax(big[2], fabs(tab.BfT[i]));
  }
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    for (int o = 16; o > 0; o >>= 1) big[t] = fmax(big[t], __shfl_down_sync(0xFFFFFFFFu, big[t], o));
    if ((threadIdx.x & 31) == 0) atomicMax(&mx[t], (unsigned long long)__double_as_longlong(big[t]));
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    int e;
    frexp(__longlong_as_double((long long)mx[threadIdx.x]), &e);
    ex[threadIdx.x] = e;                                      // |b| < 2^e
    if (blockIdx.x == 0) {
      reinterpret_cast<int *>(img + T::oEx)[threadIdx.x] = e;
      if (threadIdx.x == 0) reinterpret_cast<int *>(img + T::oEx)[3] = 0;
    }
  }
  __syncthreads();
  // K slot of GEMMs 1 and 3 -> mode
  auto mode_of = [](int s) { const int hh = s / T::K1H, i = s % T::K1H; return i < T::NPH && hh * T::NPH + i < NP ? hh * T::NPH + i : -1; };
  auto put = [&](int off, int r, int k, int ktot, double v, int t, int digit) {
    *reinterpret_cast<__half *>(img + off + tc::kmaj16(r, k, ktot)) = __float2half_rn(table_digit(v, ex[t], digit));
  };
  const int at = blockIdx.x * blockDim.x + threadIdx.x, all = gridDim.x * blockDim.x;
  for (int b = 0; b < T::NB1; ++b)
    for (int i = at; i < kDigits * T::N1 * T::K1; i += all) {
      const int r = i / T::K1, k = i % T::K1, digit = r / T::N1, s = r % T::N1;
      const int hh = s / (T::N1 / 2), x = s % (T::N1 / 2), pt = b * T::QB + hh * T::QH + x, j = mode_of(k);
      const bool on = x < T::QH && hh * T::QH + x < T::QB && pt < NQ && j >= 0;
      put(T::oB1 + b * T::B1B, r, k, T::K1, on ? tab.BvT[j * NQ + pt] : 0.0, 0, digit);
    }
  for (int b = 0; b < T::NB2; ++b)
    for (int i = at; i < kDigits * T::N2 * T::K2; i += all) {
      const int r = i / T::K2, k = i % T::K2, digit = r / T::N2, s = r % T::N2;
      const int hn = s / (T::N2 / 2), x = s % (T::N2 / 2), j = hn * T::NPH + x;
      const int hk = k / T::KC, sl = b * T::KC + k % T::KC;
      double v = 0.0;
      if (x < T::NPH && j < NP) {
        if (sl < NQ) v = (hk ? tab.Ds : tab.Dr)[sl * NP + j];
        else if (sl < T::KH && hk * T::NFH + sl - NQ < NF) v = tab.Lf[(hk * T::NFH + sl - NQ) * NP + j];
      }
      put(T::oB2 + b * T::B2B, r, k, T::K2, v, 1, digit);
    }
  for (int i = at; i < kDigits * T::N3 * T::K1; i += all) {
    const int r = i / T::K1, k = i % T::K1, digit = r / T::N3, s = r % T::N3;
    const int hn = s / (T::N3 / 2), x = s % (T::N3 / 2), qk = hn * T::NFH + x, j = mode_of(k);
    put(T::oB3, r, k, T::K1, x < T::NFH && qk < NF && j >= 0 ? tab.BfT[j * NF + qk] : 0.0, 2, digit);
  }
}

template <int P, int NE, int Q>
int split_tables_pq(dg_mesh *m) {
  using T = Sp<P, NE, Q>;
  cudaError_t e = cudaMalloc((void **)&m->split_img, T::IMG);
  if (e != cudaSuccess) return (int)e;
  k_split_tables<P, NE, Q><<<64, 256>>>(m->tab, m->split_img);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return (int)e;
}

// Elements [e0, e1) of the mesh (e1 < 0: all), as run_element_sf: a row's
// arithmetic does not depend on its tile, so a range launch gives the same bits.
template <int P, int NE, int Q>
int run_split(const dg_mesh *m, const double *c, const double *u0, double *out, double *trace_out, const double *fhat,
              const StageUpdate &su0, int mode, double *copy, cudaStream_t s, int64_t e0, int64_t e1) {
  using T = Sp<P, NE, Q>;
  static PerDevice attr_set;
  auto stage = k_element_split<P, NE, Q, false>, traces = k_element_split<P, NE, Q, (P > 1)>;   // p = 1: k_traces
  if (!attr_set.test(m->device)) {
    cudaError_t e = cudaFuncSetAttribute(stage, cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(traces, cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEM);
    if (e != cudaSuccess) return (int)e;
    attr_set.set(m->device);
  }
  if (e1 < 0) e1 = m->N;
  const int64_t n = e1 - e0;
  if (n <= 0) return (int)cudaSuccess;
  const size_t so = (size_t)e0 * M * T::NP;
  StageUpdate su = su0;
  if (su.acc) su.acc += so;
  if (su.out2) su.out2 += so;
  const int64_t ntiles = (n + T::EB - 1) / T::EB;
  const int grid = (int)(ntiles < m->num_sms ? ntiles : m->num_sms);
  (mode == 2 ? traces : stage)<<<grid, T::THREADS, T::SMEM, s>>>(
      c + so, u0 ? u0 + so : nullptr, out ? out + so : nullptr,
      trace_out ? trace_out + (size_t)e0 * T::NF * M : nullptr, fhat, m->geo + (size_t)e0 * GEO,
      m->elem_face + (size_t)e0 * 3, m->split_img, m->tab, (int)n, m->F, su, mode, m->gamma, copy ? copy + so : nullptr,
      m->err_flag);
  return (int)cudaGetLastError();
}

}  // namespace
}  // namespace dg
