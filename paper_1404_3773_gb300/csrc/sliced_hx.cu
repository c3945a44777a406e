// H.X in FP64 from exact integer-slice products on the tensor cores (Sec. 2.2.4 eq.
// matvec_final): every contraction of the radial, Legendre and phi transforms as products of
// 8-bit digits (the error-free splitting of Ozaki, Ogita, Oishi and Rump 2012), because GB300's
// FP64 pipe runs at 1/64 of the FP32 rate and bounds the FMA kernels.
//
// A row of 128 operand rows is scaled to 54-bit integers below its power of two and cut into 7
// signed digits of 8 bits, exact in BF16. The table side is cut the same way at set-up. Digit i
// of the rows times digits j of the table goes to the FP32 accumulator of diagonal t = i + j
// in tensor memory, t = 0 .. 7 (34 of the 49 pairs; the first dropped diagonal is 2^-60 of the
// row's bound). A diagonal adds at most 7 products of 2^14 per k, so sums over 64 k are
// integers below 2^24: exact in any order. A drain joins the eight diagonals into one 64-bit
// integer.
//
// Between the contractions the values stay 64-bit integers with one power of two per row, so
// the pointwise product with W V and every sum of mirror images run on the integer pipe:
//   R1  G[k][lm][s]        = sum_n R_ln(r_k) X                per l; FP64 in and out
//   L1  FA[k][par][t][kap] = sum_l Theta_lm(t) G              per |m| and parity of l - |m|
//   P1  W[k][j][class][q]  = sum_m T_class(m, q) F            per class (cos / sin, m even / odd)
//                            at the quarter angles, F(t) = E + O, F(pi - t) = E - O
//   PW  the four mirror angles of q from the class sums, times W V, folded back
//   P2  AP[k][j][kap]      = sum_q T_class(m, q) W            phi quadrature
//   L2  G'[k][lm][s]       = sum_t Theta_lm(t) (AP_j +- AP_jb)  Legendre quadrature
//   R2  Z = sum_k R_ln(r_k) G', with the epilogue of the H.X and the Chebyshev recurrence
// L1 .. L2 run over chunks of radial nodes so that the intermediates stay in the workspace slot.
//
// The kernels are bound by the instructions of splitting (about 40 per value with its load) and
// joining (about 25): 0.75 G warp instructions for 80 states at lmax 30, issued at 35 % (radial) to
// 60 % of the peak rate; the tensor cores are idle most of the time. That H.X takes 1.48 ms against
// 7.13 on the FP64 pipe (whose peak would need 2.9 ms) and 2.41 in double-float. Two to four CTAs
// of 256 threads run per SM, so one CTA's loads and drains cover the others' waits. A thread owns the same
// operand row when it loads and when it drains, so its row's scale never leaves its registers.
// Every mbarrier wait is bounded: on expiry the kernel records an error code in *err, frees its
// tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <vector>

#include "cs_internal.h"
#include "hx_device.cuh"
#include "hx_kernels.cuh"
#include "image_ring.cuh"
#include "ozaki_split.cuh"
#include "sliced_hx.h"
#include "tc_common.cuh"

namespace cs {

namespace {

using namespace tcx;

constexpr int kSlThreads = 256;
constexpr int kDig = 7;        // digits of 8 bits per value
constexpr int kDiag = 8;       // diagonals kept
constexpr int kRows = 128;     // operand rows per tile (MMA M)
constexpr int kFix = 54;       // |value| <= 2^E is held as an integer in units of 2^(E - 54)
constexpr int kADigit = kRows / 8 * 256;           // bytes of one (K step, digit): 4 KB
constexpr int kBig = 1 << 20;
constexpr int kNoUnit = (int)0x80808080;  // below every unit (a memset of 0x80)

enum { OP_R1, OP_L1, OP_P1, OP_P2, OP_L2, OP_R2 };

// Programmatic dependent launch (SlPlan says when): a kernel of the chain lets the next one start its prologue
// (barriers, tensor memory, table images) at once, and touches the chain's data only when the
// kernel before it has completed and its writes are visible. A kernel that is resident early runs
// while its predecessor still writes, so __ldg and __restrict__ are for what no kernel of a chain
// writes (the set-up tables, W V, the weights and occupations): the read-only path needs data that
// does not change while the kernel runs, and either lets the compiler move a load above the wait.
// Blocks, grid functions and intermediates are read with ordinary loads through plain pointers.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// One word of a chain's data. Volatile, so that it stays behind pdl_wait, and stated as an
// instruction, because plain C++ loads here cost 1.0 % of an 80-state H.X at lmax 30 (1496 -> 1512
// us) and 8 % of two states at lmax 62 (199 -> 216 us); this form takes the time of __ldg.
__device__ __forceinline__ long long ld_chain(const long long* p) {
  long long v;
  asm volatile("ld.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_chain(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// bytes of one table image: `ks` K steps, nb table rows
__host__ __device__ inline size_t img_bytes(int ks, int nb) {
  return (size_t)ks * kDig * (nb / 8) * 256;
}

// ---------------------------------------------------------------- integers
// bits of a two's complement value's magnitude, from v ^ (v >> 63)
__device__ __forceinline__ int bit_len(unsigned long long a) { return 64 - __clzll((long long)a); }
// A row's shift sh to 54 bits (-9 .. 31): left by l, then right by r with rounding
struct RowShift {
  int l, r;
  uint32_t rnd;
};
__device__ __forceinline__ RowShift row_shift(int sh) {
  RowShift w;
  w.l = sh > 0 ? sh : 0;
  w.r = sh < 0 ? -sh : 0;
  w.rnd = (1u << w.r) >> 1;
  return w;
}
__device__ __forceinline__ int clamp_shift(int bits) { return min(31, kFix - bits); }
__device__ __forceinline__ long long scale_i64(long long v, const RowShift& w) {
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)((unsigned long long)v >> 32);
  const uint32_t lo1 = lo << w.l, hi1 = __funnelshift_l(lo, hi, w.l);
  const unsigned long long x = (((unsigned long long)hi1 << 32) | lo1) + w.rnd;
  const uint32_t xl = (uint32_t)x, xh = (uint32_t)(x >> 32);
  return (long long)(((unsigned long long)(uint32_t)((int)xh >> w.r) << 32) |
                     __funnelshift_r(xl, xh, w.r));
}
// the double x (|x| < 2^E) as an integer in units of 2^(E - kFix), rounded to nearest
__device__ __forceinline__ long long fix_f64(unsigned long long b, int E) {
  const int e = (int)((b >> 52) & 0x7FF);
  const int r = E + 1022 - e;  // >= 0: 2^(e - 1022) is the next power of two above |x|
  if (e == 0 || r > 60) return 0;
  long long v = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 1;
  v = r == 0 ? v : ((v >> (r - 1)) + 1) >> 1;
  return (long long)b < 0 ? -v : v;
}
// Exponent 2^E above every value of a row whose largest biased exponent is mx. A row with an
// infinity or a NaN gets kNonFinite, which every unit derived from it keeps above kNonFinite / 2,
// so that all it feeds becomes NaN.
constexpr int kNonFinite = 1 << 20;
__device__ __forceinline__ int exp_above_bits(int mx) {
  return mx == 0 ? -900 : (mx == 0x7FF ? kNonFinite : mx - 1022);
}
// v 2^u as a double
__device__ __forceinline__ double to_f64(long long v, int u) {
  if (u > kNonFinite / 2) return __longlong_as_double(0x7FF8000000000000ll);
  double x = (double)v;
  if (u < -960) {  // towards underflow: in two steps
    x *= oz_pow2(-960);
    u = max(u + 960, -1022);
  }
  return x * oz_pow2(min(u, 1023));
}

// The 7 digits of two neighbouring values of an octet, as BF16 pairs: byte k of v + bias is
// digit k + 128; 128 + (b & 127) minus 128 or 256 is the digit, exactly.
__device__ __forceinline__ void pack_pair(long long v0, long long v1, uint32_t* p) {
  const unsigned long long bias = 0x0080808080808080ull;
  const unsigned long long a = (unsigned long long)v0 + bias, b = (unsigned long long)v1 + bias;
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
  const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
#pragma unroll
  for (int k = 0; k < kDig; ++k) {  // k = 0: lowest byte; stored last (digit 0 = leading)
    const int by = k & 3;
    const uint32_t x = __byte_perm(k < 4 ? al : ah, k < 4 ? bl : bh,
                                   (uint32_t)(by | (by << 4) | ((4 + by) << 8) | ((4 + by) << 12)));
    const uint32_t m = (x & 0x007F007Fu) | 0x43004300u;
    const uint32_t c = (~x & 0x00800080u) | 0xC300C300u;
    const __nv_bfloat162 d = __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&m),
                                     *reinterpret_cast<const __nv_bfloat162*>(&c));
    p[kDig - 1 - k] = *reinterpret_cast<const uint32_t*>(&d);
  }
}

// The eight diagonal sums (exact integers in FP32) as one integer in units of 2^-56 of the row's
// bound times the table's: diagonal t carries 2^(-12 - 8 t). SMALL (K <= 32): every sum is below
// 2^22, so adding 1.5 2^23 leaves it in the low bits of the float; the constant's bits are taken
// off pairs of terms, modulo 2^32 (a conversion runs at a quarter of the rate of an addition).
template <bool SMALL, bool WIDE = false>
__device__ __forceinline__ long long join_diags(const float* d, int c4, int c20) {
  if constexpr (SMALL) {
    uint32_t b[kDiag];
#pragma unroll
    for (int t = 0; t < kDiag; ++t) b[t] = __float_as_uint(d[t] + 12582912.f);
    constexpr uint32_t kB = 0x4B400000u * 257u;  // the bits of 1.5 2^23, for pairs 256 b + b'
    const int p = (int)((b[0] << 8) + (b[1] - kB)), q = (int)((b[2] << 8) + (b[3] - kB));
    const int r = (int)((b[4] << 8) + (b[5] - kB)), t = (int)((b[6] << 8) + (b[7] - (kB - 2048u)));
    // c4 = 2^4 and c20 = 2^20 come as kernel arguments, so that the products stay multiply-adds
    const long long v = (long long)q * c20 + ((long long)r * c4 + (t >> 12));
    return v + ((long long)(p << 4) << 32);
  } else {
    int i[kDiag];
#pragma unroll
    for (int t = 0; t < kDiag; ++t) i[t] = __float2int_rn(d[t]);
    if constexpr (WIDE) {  // up to 128 k: sums below 2^24, 2 bits less kept
      const long long h = (long long)i[0] * 65536 + ((long long)i[1] * 256 + i[2]);
      const long long m = (long long)i[3] * 65536 + ((long long)i[4] * 256 + i[5]);
      const int lo = (int)(((long long)i[6] * 256 + (i[7] + 8192)) >> 14);
      return (h << 26) + (m << 2) + lo;
    }
    const long long h = (long long)i[0] * 65536 + (i[1] * 256 + i[2]);
    const long long m = (long long)i[3] * 65536 + (i[4] * 256 + i[5]);
    const int lo = (i[6] * 256 + i[7] + 2048) >> 12;
    return (h << 28) + (m << 4) + lo;
  }
}

// ---------------------------------------------------------------- the contraction kernel
struct SlArgs {
  int L, N, n_r, Nt, NP, M2, Q, S;  // S: states of the whole block
  int k0, kc, s0, SB;               // chunk: radial nodes k0 .. k0 + kc - 1, states s0 .. s0+SB-1
  int F1;                           // exponent of the Legendre table of L1
  int ks;                           // K steps of one mode class (L1, P1)
  int nb2;                          // table rows per class, padded (P2, L2): 16 or 32
  const unsigned char* tab;         // this operation's table images
  const int* fexp;                  // per table row exponents (R1, R2, L2)
  const int* rexp;                  // R2: exponent e_k of the radial scaling
  const double* X;                  // R1
  long long ld;
  double* G;
  const int* EG;                    // [k][S]
  long long* FA;                    // also AP
  long long* W;
  int* eW;                          // P1: unit of W's row, [k'][j][SB]
  const int* shP;                   // P2: shift of W's row
  const int* uP;                    // unit of AP's row
  const int* U;                     // [k'][SB] largest uP of the node
  int* Uw;                          // the same, to be written
  long long ntiles;
  bool early;                       // host: launch with programmatic dependence
  int c4 = 1 << 4, c20 = 1 << 20;  // see join_diags
  int* err;
  Epilogue<double> ep;              // R2
};

// Tile -> (table, rows) of one operation, and what a thread knows of its row.
struct SlRow {
  bool live;
  int kp, j, s;        // chunk node, theta row, state of the block
  int l, mi, m, par, cls;
};

template <int OP>
__device__ __forceinline__ void sl_locate(const SlArgs& a, long long tile, int r, SlRow& w,
                                          int& table) {
  w.l = w.mi = w.m = w.par = w.cls = w.kp = w.j = w.s = 0;
  table = 0;
  if constexpr (OP == OP_R1 || OP == OP_R2) {
    int l = 0;
    for (;; ++l) {
      const long long ct = ((long long)(2 * l + 1) * a.S + kRows - 1) / kRows;
      if (tile < ct) break;
      tile -= ct;
    }
    const long long c = tile * kRows + r;
    w.live = c < (long long)(2 * l + 1) * a.S;
    w.l = l;
    w.mi = (int)(c / a.S);
    w.s = (int)(c - (long long)w.mi * a.S);
    table = l;
  } else if constexpr (OP == OP_L1 || OP == OP_L2) {
    const int rows1 = a.kc * a.SB;
    const int t0 = (rows1 + kRows - 1) / kRows, t1 = (2 * rows1 + kRows - 1) / kRows;
    int am, c;
    if (tile < 2 * t0) {
      am = 0;
      w.par = (int)(tile / t0);
      c = (int)(tile - (long long)w.par * t0) * kRows + r;
    } else {
      tile -= 2 * t0;
      const int g = (int)(tile / t1);
      am = 1 + (g >> 1);
      w.par = g & 1;
      c = (int)(tile - (long long)g * t1) * kRows + r;
    }
    const int nrows = am ? 2 * rows1 : rows1;
    w.live = c < nrows;
    const int neg = c >= rows1;
    c -= neg ? rows1 : 0;
    w.m = neg ? -am : am;
    w.kp = c / a.SB;
    w.s = c - w.kp * a.SB;
    table = am * 2 + w.par;
  } else {
    const int rows = a.kc * a.Nt * a.SB;
    const int tr = (rows + kRows - 1) / kRows;
    if constexpr (OP == OP_P2) {
      w.cls = (int)(tile / tr);
      tile -= (long long)w.cls * tr;
      table = w.cls;
    }
    const int c = (int)tile * kRows + r;
    w.live = c < rows;
    const int kj = c / a.SB;
    w.s = c - kj * a.SB;
    w.kp = kj / a.Nt;
    w.j = kj - w.kp * a.Nt;
  }
}

// Geometry: column blocks per table, K chunks of 32, table rows per block
template <int OP, int NB>
__device__ __forceinline__ void sl_geom(const SlArgs& a, int& nsteps, int& nch, int& lastks) {
  int K = 0, Nn = 0;
  if constexpr (OP == OP_R1) { K = a.N; Nn = a.n_r; }
  if constexpr (OP == OP_R2) { K = a.n_r; Nn = a.N; }
  if constexpr (OP == OP_L1) { K = a.ks * 16; Nn = a.NP; }
  if constexpr (OP == OP_P1) { K = a.ks * 16; Nn = a.Q; }
  if constexpr (OP == OP_P2) { K = a.Q; Nn = 1; }
  if constexpr (OP == OP_L2) { K = a.NP; Nn = 1; }
  nsteps = (Nn + NB - 1) / NB;
  if constexpr (OP == OP_P1) nsteps *= 4;  // the four classes of a row tile
  nch = (K + 31) / 32;
  lastks = (K - 32 * (nch - 1) + 15) / 16;
}

// eight operand values k = kb .. kb + 7 of a row as integers in the row's common unit
// (L1: doubles' bits; R1, R2: doubles' bits)
template <int OP>
__device__ __forceinline__ void sl_load8(const SlArgs& a, const SlRow& w, int cls, int kb,
                                         long long* v) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0;
  if (!w.live) return;
  if constexpr (OP == OP_R1) {
    const double* x = a.X + (size_t)(w.l * w.l + w.mi) * a.N + (size_t)w.s * a.ld;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (kb + i < a.N) v[i] = __double_as_longlong(ld_chain(x + kb + i));
  } else if constexpr (OP == OP_R2) {
    const size_t st = (size_t)a.L * a.L * a.S;
    const double* g = a.G + (size_t)(w.l * w.l + w.mi) * a.S + w.s;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (kb + i < a.n_r) v[i] = __double_as_longlong(ld_chain(g + (size_t)(kb + i) * st));
  } else if constexpr (OP == OP_L1) {
    const int am = w.m < 0 ? -w.m : w.m;
    const double* g = a.G + (size_t)(a.k0 + w.kp) * a.L * a.L * a.S + a.s0 + w.s;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int l = am + w.par + 2 * (kb + i);
      if (l < a.L) v[i] = __double_as_longlong(ld_chain(g + (size_t)(l * l + l + w.m) * a.S));
    }
  } else if constexpr (OP == OP_P1) {
    const int t = w.j < a.NP ? w.j : a.Nt - 1 - w.j;
    const long long* e = a.FA + ((size_t)(w.kp * 2) * a.NP + t) * a.M2 * a.SB + w.s;
    const long long* o = e + (size_t)a.NP * a.M2 * a.SB;
    const long long mir = w.j >= a.NP ? -1 : 0;
    const int lmax = a.L - 1;
    const int m0 = 2 * kb + (cls & 1), sg = cls < 2 ? 1 : -1;
    const int off = (lmax + sg * m0) * a.SB, st = 2 * sg * a.SB;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = m0 + 2 * i <= lmax && (cls < 2 || m0 + 2 * i > 0);
      const long long ev = in ? ld_chain(e + off + i * st) : 0, ov = in ? ld_chain(o + off + i * st) : 0;
      v[i] = ev + (ov ^ mir) - mir;
    }
  } else if constexpr (OP == OP_P2) {
    const long long* x =
        a.W + (((size_t)(w.kp * a.Nt + w.j) * 4 + cls) * a.Q + kb) * a.SB + w.s;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (kb + i < a.Q) v[i] = ld_chain(x + i * a.SB);
  } else {
    const int rs = a.M2 * a.SB;
    const long long odd = w.par ? -1 : 0;
    const long long* x = a.FA + (size_t)w.kp * a.Nt * rs + (a.L - 1 + w.m) * a.SB + w.s;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int t = kb + i, jb = a.Nt - 1 - t;
      const long long y = t < a.NP ? ld_chain(x + t * rs) : 0;
      const long long z = t < a.NP && jb != t ? ld_chain(x + jb * rs) : 0;
      v[i] = y + (z ^ odd) - odd;
    }
  }
}

// CTAs per SM: 16-column blocks take 128 of the 512 columns of tensor memory, and the syntheses
// fit 64 registers; P2 and L2 hold K = 32 in shared memory (70 KB)
constexpr int sl_ctas(int op, int nb) {
  return nb != 16 ? 2 : (op == OP_L1 || op == OP_P1 ? 4 : 3);
}

// SMALL: at most 32 k per accumulation (join_diags)
template <int OP, int NB, bool SMALL>
__global__ void __launch_bounds__(kSlThreads, sl_ctas(OP, NB)) k_sl(SlArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar_b[2], bar_mma;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int red[2][kRows];
  constexpr bool F64 = OP == OP_R1 || OP == OP_R2 || OP == OP_L1;  // double operands
  constexpr bool RAD = OP == OP_R1 || OP == OP_R2;
  constexpr int kBStep = kDig * (NB / 8) * 256;  // bytes of a K step of a table image
  constexpr uint32_t kCols = kDiag * NB;
  constexpr int HC = NB / 2;  // columns a thread drains
  constexpr int kGrp = RAD ? 3 : 1;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int r = tid & (kRows - 1), half = tid >> 7;
  int nsteps, nch, lastks;
  sl_geom<OP, NB>(a, nsteps, nch, lastks);
  const int ksmax = nch > 1 ? 2 : lastks;
  if (tid == 0) {
    mbar_init(smem_u32(&bar_b[0]), 1);
    mbar_init(smem_u32(&bar_b[1]), 1);
    mbar_init(smem_u32(&bar_mma), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(&tmem_base_sh), kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  // only now: a kernel further down the chain must not take the tensor memory that this one,
  // which it waits for, still asks for
  pdl_trigger();
  const uint32_t sA = smem_u32(smem), sB = sA + (uint32_t)(ksmax * kDig * kADigit);
  const uint32_t bslot = (uint32_t)(ksmax * kBStep);

  // this CTA's tiles: a contiguous range, so that tables and cached rows are shared
  const long long t0 = a.ntiles * blockIdx.x / gridDim.x;
  const long long t1 = a.ntiles * (blockIdx.x + 1) / gridDim.x;
  auto ks_of = [&](int ch) { return ch == nch - 1 ? lastks : 2; };
  // table images: [table][column block][K chunk]
  const size_t img_full = (size_t)2 * kBStep;
  const size_t tab_block = img_full * (nch - 1) + (size_t)lastks * kBStep;
  int step = 0, issued = 0;     // steps begun; images requested (thread 0); see image_ring.cuh
  auto issue_b = [&](int table, int st, int ch) {
    const int sl = image_slot(issued);
    const uint32_t bytes = (uint32_t)(ks_of(ch) * kBStep);
    const uint32_t b = smem_u32(&bar_b[sl]);
    mbar_expect_tx(b, bytes);
    bulk_g2s(sB + (uint32_t)sl * bslot,
             a.tab + ((size_t)table * nsteps + st) * tab_block + (size_t)ch * img_full, bytes, b);
    ++issued;
  };
  SlRow w;
  int table;
  sl_locate<OP>(a, t0, r, w, table);
  if (tid == 0 && t0 < t1) issue_b(table, 0, 0);
  pdl_wait();
  if constexpr (OP == OP_L1)  // the units' maxima of the chunk start from nothing
    for (int i = blockIdx.x * kSlThreads + tid; i < a.kc * a.SB; i += gridDim.x * kSlThreads)
      a.Uw[i] = kNoUnit;

  bool ok = true;    // block-uniform
  bool good = true;  // this thread's waits
  for (long long tile = t0; ok && tile < t1; ++tile) {
    if (tile != t0) sl_locate<OP>(a, tile, r, w, table);
    int rowsc = 0;  // F64: exponent E of the row; else: shift to 54 bits
    // ---- scale of the row
    if constexpr (OP == OP_L1) {
      if (w.live) rowsc = a.EG[(size_t)(a.k0 + w.kp) * a.S + a.s0 + w.s];
    } else if constexpr (OP == OP_P2) {
      if (w.live) rowsc = a.shP[(size_t)(w.kp * a.Nt + w.j) * a.SB + w.s];
    } else {
      int mx = -kBig;
      if constexpr (OP == OP_P1) {
        unsigned long long acc = 0;
        if (w.live) {
          const int t = w.j < a.NP ? w.j : a.Nt - 1 - w.j;
          const long long* e =
              a.FA + (((size_t)(w.kp * 2) * a.NP + t) * a.M2 + half) * a.SB + w.s;
          const size_t od = (size_t)a.NP * a.M2 * a.SB, st = (size_t)2 * a.SB;
          const long long mir = w.j >= a.NP ? -1 : 0;
#pragma unroll 8
          for (int kap = half; kap < a.M2; kap += 2, e += st) {
            const long long ev = ld_chain(e), ov = ld_chain(e + od);
            const long long v = ev + (ov ^ mir) - mir;
            acc |= (unsigned long long)(v ^ (v >> 63));
          }
        }
        mx = bit_len(acc);
      } else {
        unsigned long long acc = 0;
        for (int ch = 0; ch < nch; ++ch)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int oct = half + 2 * u;
            if (oct >= 2 * ks_of(ch)) continue;
            long long v[8];
            sl_load8<OP>(a, w, 0, 32 * ch + 8 * oct, v);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if constexpr (F64) {
                mx = max(mx, (int)((v[i] >> 52) & 0x7FF));
              } else {
                acc |= (unsigned long long)(v[i] ^ (v[i] >> 63));
              }
            }
          }
        if constexpr (!F64) mx = bit_len(acc);
      }
      red[half][r] = mx;
      __syncthreads();
      mx = max(red[0][r], red[1][r]);
      rowsc = F64 ? exp_above_bits(max(mx, 0)) : clamp_shift(mx);
    }
    const RowShift rsh = row_shift(F64 ? 0 : rowsc);
    // ---- where the row's results go: base, stride and range of the column index n
    long long* out = nullptr;
    int ost = 0;
    int nlo = 0, nhi = 0, ush = 0;
    if constexpr (OP == OP_L1) {
      out = a.FA + (((size_t)(w.kp * 2 + w.par) * a.NP) * a.M2 + (a.L - 1 + w.m)) * a.SB + w.s;
      ost = a.M2 * a.SB;
      nhi = w.live ? a.NP : 0;
    } else if constexpr (OP == OP_P2) {
      const int sg = w.cls < 2 ? 1 : -1, m0 = w.cls & 1;
      out = a.FA + ((ptrdiff_t)(w.kp * a.Nt + w.j) * a.M2 + (a.L - 1 + sg * m0)) * a.SB + w.s;
      ost = 2 * sg * a.SB;
      nlo = w.cls == 2 ? 1 : 0;
      nhi = w.live ? (a.L - m0 + 1) / 2 : 0;
      // results in the unit of the node's largest row (rows of zeros: no shift)
      if (w.live)
        ush = max(0, min(63, a.U[w.kp * a.SB + w.s] -
                                 a.uP[(size_t)(w.kp * a.Nt + w.j) * a.SB + w.s]));
    } else if constexpr (OP == OP_L2) {
      // unit of G', which is left scaled by the radial table's power of two of its node
      if (w.live)
        ush = a.U[w.kp * a.SB + w.s] - rowsc + kFix - 56 - __ldg(a.rexp + a.k0 + w.kp);
    } else if constexpr (OP == OP_P1) {
      out = a.W + (size_t)(w.kp * a.Nt + w.j) * 4 * a.Q * a.SB + w.s;
      ost = a.SB;
      nhi = w.live ? a.Q : 0;
    }
    long long acc[RAD ? HC : 1];
    for (int st = 0; ok && st < nsteps; ++st) {
      const int qb = OP == OP_P1 ? nsteps / 4 : 1;
      const int cls = OP == OP_P1 ? st / qb : w.cls;
      const bool new_rows = OP == OP_P1 ? st == cls * qb : (st == 0 || nch > 1);
      if constexpr (RAD) {
#pragma unroll
        for (int c = 0; c < HC; ++c) acc[c] = 0;
      }
      for (int ch = 0; ok && ch < nch; ++ch) {
        const int ks = ks_of(ch);
        // ---- operand rows -> digits
        if (new_rows) {
#pragma unroll 1
          for (int u = 0; u < 2; ++u) {
            const int oct = half + 2 * u;
            if (oct >= 2 * ks) break;
            long long v[8];
            sl_load8<OP>(a, w, cls, 32 * ch + 8 * oct, v);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if constexpr (F64) {
                v[i] = fix_f64((unsigned long long)v[i], rowsc);
              } else {
                v[i] = scale_i64(v[i], rsh);
              }
            }
            uint32_t p[4][kDig];
#pragma unroll
            for (int i = 0; i < 4; ++i) pack_pair(v[2 * i], v[2 * i + 1], p[i]);
            unsigned char* dst = smem + (size_t)(oct >> 1) * kDig * kADigit + (r >> 3) * 256 +
                                 (oct & 1) * 128 + (r & 7) * 16;
#pragma unroll
            for (int k = 0; k < kDig; ++k)
              *reinterpret_cast<uint4*>(dst + k * kADigit) =
                  make_uint4(p[0][k], p[1][k], p[2][k], p[3][k]);
          }
        }
        fence_async_smem();
        tc_fence_before();
        ok = __syncthreads_and(good ? 1 : 0) != 0;
        if (!ok) break;
        // sums over groups of 64 k (the radial products: 128) start and end here
        const bool fresh = (ch & kGrp) == 0, drain = (ch & kGrp) == kGrp || ch == nch - 1;
        if (tid == 0) {
          // the next step's image: the MMAs that read that slot have completed
          if (ch + 1 < nch) {
            issue_b(table, st, ch + 1);
          } else if (st + 1 < nsteps) {
            issue_b(table, st + 1, 0);
          } else if (tile + 1 < t1) {
            SlRow wn;
            int tn;
            sl_locate<OP>(a, tile + 1, 0, wn, tn);
            issue_b(tn, 0, 0);
          }
          tc_fence_after();
          if (!mbar_wait(smem_u32(&bar_b[image_slot(step)]), image_parity(step))) {
            atomicCAS(a.err, 0, 41);
            good = false;
          } else {
            const uint32_t b0 = sB + (uint32_t)image_slot(step) * bslot;
            for (int s = 0; s < ks; ++s) {
              const uint32_t ab = sA + s * kDig * kADigit, bb = b0 + s * kBStep;
              auto mma = [&](int i, int j, int cnt, uint32_t accum) {
                mma_bf16(tmem + (uint32_t)((i + j) * NB), make_desc(ab + i * kADigit, 128, 256),
                         make_desc(bb + j * (NB / 8) * 256, 128, 256),
                         make_idesc(kRows, cnt * NB), accum);
              };
              // the first K step of a group starts the accumulators: digit 0 x 0 starts
              // diagonal 0, digit 1 x 0 .. 6 diagonals 1 .. 7
              const uint32_t go = (fresh && s == 0) ? 0u : 1u;
              mma(0, 0, 1, go);
              mma(1, 0, 7, go);
              mma(0, 1, 6, 1u);
#pragma unroll
              for (int i = 2; i < kDig; ++i) mma(i, 0, kDiag - i, 1u);
            }
          }
          mma_commit(smem_u32(&bar_mma));
        }
        if (!mbar_wait(smem_u32(&bar_mma), mma_parity(step))) {
          atomicCAS(a.err, 0, 42);
          good = false;
        }
        ++step;
        tc_fence_after();
        if (!drain) continue;
        // ---- drain: 4 columns at a time
        const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(half * HC);
        [[maybe_unused]] long long* const o =
            out + (ptrdiff_t)((OP == OP_P1 ? cls * a.Q + NB * (st - cls * qb) : NB * st) +
                              half * HC) * ost;
#pragma unroll
        for (int c0 = 0; c0 < HC; c0 += 4) {
          float d[kDiag][4];
#pragma unroll
          for (int t = 0; t < kDiag; ++t) tmem_ld4_issue(ta + (uint32_t)(t * NB + c0), d[t]);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float x[kDiag];
#pragma unroll
            for (int t = 0; t < kDiag; ++t) x[t] = d[t][c];
            const long long v = join_diags<SMALL, RAD>(x, a.c4, a.c20);
            const int n = half * HC + c0 + c;  // column of the block
            if constexpr (RAD) {
              acc[c0 + c] += v;  // units of 2^-54: room for 448 k
            } else if constexpr (OP == OP_L1) {
              if (NB * st + n < nhi) o[(c0 + c) * ost] = v;
            } else if constexpr (OP == OP_P1) {
              if (NB * (st - cls * qb) + n < nhi) o[(c0 + c) * ost] = v;
            } else if constexpr (OP == OP_P2) {
              if (n >= nlo && n < nhi) o[(c0 + c) * ost] = v >> ush;
            } else {
              const int am = w.m < 0 ? -w.m : w.m;
              const int l = am + w.par + 2 * n;
              if (w.live && l < a.L) {
                const int u = ush + __ldg(a.fexp + table * a.nb2 + n);
                a.G[((size_t)(a.k0 + w.kp) * a.L * a.L + l * l + l + w.m) * a.S + a.s0 + w.s] =
                    to_f64(v, u);
              }
            }
          }
        }
      }
      if constexpr (OP == OP_R1) {
        if (ok && w.live) {
#pragma unroll
          for (int c = 0; c < HC; ++c) {
            const int k = NB * st + half * HC + c;
            if (k < a.n_r)
              a.G[((size_t)k * a.L * a.L + w.l * w.l + w.mi) * a.S + w.s] =
                  to_f64(acc[c], rowsc + __ldg(a.fexp + w.l * a.n_r + k) - 54);
          }
        }
      }
      if constexpr (OP == OP_R2) {
        if (ok && w.live) {
#pragma unroll
          for (int c = 0; c < HC; ++c) {
            const int n = NB * st + half * HC + c;
            if (n >= a.N) continue;
            const double z = to_f64(acc[c], rowsc + __ldg(a.fexp + w.l * a.N + n) - 54);
            const size_t al = (size_t)(w.l * w.l + w.mi) * a.N + n;
            radial_epilogue(a.ep, al, w.s, z);
          }
        }
      }
    }
    if constexpr (OP == OP_P1) {
      // unit of the row's class sums: the operand's unit 2^(E_G + F1 - 56 - shift), less 2 bits
      if (w.live && half == 0)
        a.eW[(size_t)(w.kp * a.Nt + w.j) * a.SB + w.s] =
            a.EG[(size_t)(a.k0 + w.kp) * a.S + a.s0 + w.s] + a.F1 - 56 - rowsc +
            kFix - 56;
    }
  }
  // after an expired wait: what is still on its way into this CTA's memory lands before the exit
  if (tid == 0 && (!good || issued != step))
    settle_images(
        step, issued,
        [&](int sl, uint32_t parity) { mbar_wait(smem_u32(&bar_b[sl]), parity); },
        [&](uint32_t parity) { mbar_wait(smem_u32(&bar_mma), parity); });
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------- pointwise pass
// f w / 2^64 without the product of the low halves (less than one unit); w is stored with its
// low half signed (k_sl_wv), f is split the same way
__device__ __forceinline__ long long mul_hi(long long f, long long w) {
  const int fl = (int)f, fh = (int)((unsigned long long)f >> 32) - (fl >> 31);
  const int wl = (int)w, wh = (int)((unsigned long long)w >> 32);
  const long long mid = (long long)fl * wh + (long long)fh * wl;
  return (long long)fh * wh + (mid >> 32);
}

// Per (grid row, state): the four mirror angles of each quarter angle from the class
// sums, times W V (integer of 62 bits below the row's power of two), folded back into the four
// classes in place; then the row's shift to 54 bits, its unit after P2 and the node's largest.
// A CTA holds 32 (row, state) pairs; its 8 warps take the quarter angles q = warp, warp + 8, ...
__global__ void __launch_bounds__(256) k_sl_pointwise(long long* W, const int* eW,
                                                      const long long* __restrict__ wv,
                                                      const int* __restrict__ ewv, int rows,
                                                      int SB, int Nt, int Np, int Q, int k0,
                                                      int* shP, int* uP, int* U) {
  pdl_trigger();
  pdl_wait();
  __shared__ int red[8][32];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const long long i = (long long)blockIdx.x * 32 + lane;
  const bool live = i < (long long)rows * SB;
  const int row = live ? (int)(i / SB) : 0, s = live ? (int)(i - (long long)row * SB) : 0;
  const long long gr = (long long)k0 * Nt + row;  // grid row of the whole grid
  const long long* w = wv + gr * Np;
  const size_t cs = (size_t)Q * SB;
  const int h = Np / 2;
  unsigned long long acc = 0;
  long long* p = W + (size_t)row * 4 * cs + (size_t)wp * SB + s;
  if (live) {
#pragma unroll 2
    for (int q = wp; q < Q; q += 8, p += (size_t)8 * SB) {
      const long long c0 = p[0], c1 = p[cs], c2 = p[2 * cs], c3 = p[3 * cs];
      const long long ep = c0 + c1, em = c0 - c1, op = c2 + c3, om = c2 - c3;
      const long long g0 = mul_hi(ep + op, __ldg(w + q));
      const long long g1 = mul_hi(ep - op, __ldg(w + (q == 0 ? 0 : Np - q)));
      const long long g2 = mul_hi(em - om, __ldg(w + h - q));
      const long long g3 = mul_hi(em + om, __ldg(w + h + q));
      long long P = g0 + g1, M = g0 - g1, P2 = g2 + g3, N2 = g2 - g3;
      if (q == 0 || 2 * q == h) {  // mirror angles that coincide count once
        P >>= 1;
        M >>= 1;
        P2 >>= 1;
        N2 >>= 1;
      }
      const long long r0 = P + P2, r1 = P - P2, r2 = M - N2, r3 = M + N2;
      p[0] = r0;
      p[cs] = r1;
      p[2 * cs] = r2;
      p[3 * cs] = r3;
      acc |= (unsigned long long)(r0 ^ (r0 >> 63)) | (unsigned long long)(r1 ^ (r1 >> 63)) |
             (unsigned long long)(r2 ^ (r2 >> 63)) | (unsigned long long)(r3 ^ (r3 >> 63));
    }
  }
  red[wp][lane] = bit_len(acc);
  __syncthreads();
  if (wp == 0 && live) {
    int b = red[0][lane];
#pragma unroll
    for (int g = 1; g < 8; ++g) b = max(b, red[g][lane]);
    const int sh = clamp_shift(b);
    const int u = eW[i] + ewv[gr] + 2 - sh + kFix - 56;  // unit of AP's row
    shP[i] = sh;
    uP[i] = u;
    if (b || u > kNonFinite / 2) atomicMax(U + (row / Nt) * SB + s, u);
  }
}

// The folded classes of grid functions g[s][k][j][q] times the row's quadrature weight, as the
// pointwise pass leaves them: one warp per (grid row, state), lanes over the quarter angles.
__global__ void __launch_bounds__(256) k_sl_fold(const double* g,
                                                 const double* __restrict__ wkj, int rows, int SB,
                                                 int s0, int k0, int Nt, int Np, int Q, int n_r,
                                                 long long* W, int* shP, int* uP, int* U) {
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= (long long)rows * SB) return;
  const int row = (int)(i / SB), s = (int)(i - (long long)row * SB);
  const long long gr = (long long)k0 * Nt + row;
  const double* x = g + ((long long)(s0 + s) * n_r * Nt + gr) * Np;
  const double wt = __ldg(wkj + gr);
  const int h = Np / 2;
  double v[2][4];
  int mx = 0;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int q = lane + 32 * u;
    const int at[4] = {q, q == 0 ? 0 : Np - q, h - q, h + q};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[u][c] = q < Q ? ld_chain(x + at[c]) * wt : 0.0;
      mx = max(mx, (int)((__double_as_longlong(v[u][c]) >> 52) & 0x7FF));
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  const int E = exp_above_bits(mx);
  unsigned long long acc = 0;
  long long* o = W + (size_t)row * 4 * Q * SB + s;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int q = lane + 32 * u;
    if (q >= Q) continue;
    long long f[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      f[c] = fix_f64((unsigned long long)__double_as_longlong(v[u][c]), E) * 2;
    const int hf = (q == 0 || 2 * q == h) ? 1 : 0;
    const long long P = (f[0] + f[1]) >> hf, M = (f[0] - f[1]) >> hf;
    const long long P2 = (f[2] + f[3]) >> hf, N2 = (f[2] - f[3]) >> hf;
    const long long r[4] = {P + P2, P - P2, M - N2, M + N2};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      o[(size_t)(c * Q + q) * SB] = r[c];
      acc |= (unsigned long long)(r[c] ^ (r[c] >> 63));
    }
  }
  const int bits = __reduce_max_sync(0xffffffffu, bit_len(acc));
  if (lane == 0) {
    const int sh = clamp_shift(bits);
    const int u = E - kFix - 1 - sh + kFix - 56;
    shP[i] = sh;
    uP[i] = u;
    if (bits || u > kNonFinite / 2) atomicMax(U + (row / Nt) * SB + s, u);
  }
}

// Grid values f[s][k][j][q] from the class sums: one warp per (grid row, state), the CTA's warps
// on consecutive states so that they share the sectors of W.
__global__ void __launch_bounds__(256) k_sl_grid(const long long* W, const int* eW, int rows,
                                                 int SB, int s0, int k0, int Nt, int Np, int Q,
                                                 int n_r, double* f) {
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= (long long)rows * SB) return;
  const int row = (int)(i / SB), s = (int)(i - (long long)row * SB);
  double* y = f + ((long long)(s0 + s) * n_r * Nt + (long long)k0 * Nt + row) * Np;
  const long long* x = W + (size_t)row * 4 * Q * SB + s;
  const size_t cs = (size_t)Q * SB;
  const int h = Np / 2, u = eW[i];
  for (int q = lane; q < Q; q += 32) {
    const long long* p = x + (size_t)q * SB;
    const long long c0 = ld_chain(p), c1 = ld_chain(p + cs), c2 = ld_chain(p + 2 * cs), c3 = ld_chain(p + 3 * cs);
    const long long ep = c0 + c1, em = c0 - c1, op = c2 + c3, om = c2 - c3;
    y[q] = to_f64(ep + op, u);
    if (q > 0) y[Np - q] = to_f64(ep - op, u);
    if (2 * q != h) {
      y[h - q] = to_f64(em - om, u);
      if (q > 0) y[h + q] = to_f64(em + om, u);
    }
  }
}

// rho (+)= 2 sum_s occ[s] f[s]^2 over the block's states, in state order. One CTA per grid row:
// the four mirror angles of every quarter angle for 32 states at a time (lanes over the states),
// through shared memory to one thread per angle. A state's power of two goes into its weight, so
// that the squares need three FP64 operations per value; the FP64 pipe is what bounds this pass.
__global__ void __launch_bounds__(256) k_sl_density(const long long* W, const int* eW, int SB,
                                                    int Nt, int Np, int Q, int k0,
                                                    const double* __restrict__ occ, double* rho,
                                                    int accumulate) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ double dsm[];  // [4 Q][33], then weights [32]
  double* wt = dsm + 4 * Q * 33;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int row = blockIdx.x, h = Np / 2;
  const long long* x = W + (size_t)row * 4 * Q * SB;
  const size_t cs = (size_t)Q * SB;
  double acc = 0.0;  // the angle 4 q + c of this thread: at most 4 Q <= 256
  for (int b = 0; b < SB; b += 32) {
    const int s = b + lane;
    const bool live = s < SB;
    const int u = live ? eW[(size_t)row * SB + s] : 0;
    const bool plain = u > -400 && u < 400;  // the square of the unit stays in range
    __syncthreads();
    if (wp == 0) {
      const double o = live ? __ldg(occ + s) : 0.0;
      wt[lane] = plain ? o * oz_pow2(2 * u) : o;
    }
    for (int q = wp; q < Q; q += 8) {
      long long c0 = 0, c1 = 0, c2 = 0, c3 = 0;
      if (live) {
        const long long* p = x + (size_t)q * SB + s;
        c0 = ld_chain(p);
        c1 = ld_chain(p + cs);
        c2 = ld_chain(p + 2 * cs);
        c3 = ld_chain(p + 3 * cs);
      }
      const long long ep = c0 + c1, em = c0 - c1, op = c2 + c3, om = c2 - c3;
      const long long f[4] = {ep + op, ep - op, em - om, em + om};
#pragma unroll
      for (int c = 0; c < 4; ++c)
        dsm[(4 * q + c) * 33 + lane] = plain ? (double)f[c] : to_f64(f[c], u);
    }
    __syncthreads();
    if (tid < 4 * Q) {
      const int n = min(32, SB - b);
      for (int i = 0; i < n; ++i) {
        const double v = dsm[tid * 33 + i];
        acc = fma(wt[i] * v, v, acc);
      }
    }
  }
  if (tid < 4 * Q) {
    const int q = tid >> 2, c = tid & 3;
    const int p = c == 0 ? q : c == 1 ? Np - q : c == 2 ? h - q : h + q;
    // mirror angles that coincide are written once
    const bool own = c == 0 || (c == 1 && q > 0) || (c >= 2 && 2 * q != h && (c == 2 || q > 0));
    if (own) {
      double* o = rho + ((long long)k0 * Nt + row) * Np + p;
      *o = (accumulate ? *o : 0.0) + 2.0 * acc;
    }
  }
}

// E_G[k][s]: 2^E above every |G[k][lm][s]|
__global__ void __launch_bounds__(256) k_sl_gexp(const double* G, int L2, int S, int* EG) {
  pdl_trigger();
  pdl_wait();
  __shared__ int red[8][32];
  const int s = blockIdx.x * 32 + (threadIdx.x & 31), k = blockIdx.y, wp = threadIdx.x >> 5;
  int mx = 0;
  if (s < S) {
    const double* g = G + (size_t)k * L2 * S + s;
    for (int lm = wp; lm < L2; lm += 8)
      mx = max(mx, (int)((__double_as_longlong(ld_chain(g + (size_t)lm * S)) >> 52) & 0x7FF));
  }
  red[wp][threadIdx.x & 31] = mx;
  __syncthreads();
  if (wp == 0 && s < S) {
#pragma unroll
    for (int i = 1; i < 8; ++i) mx = max(mx, red[i][threadIdx.x]);
    EG[(size_t)k * S + s] = exp_above_bits(mx);
  }
}

// W V of one grid row as 62-bit integers below the row's power of two
__global__ void __launch_bounds__(128) k_sl_wv(const double* __restrict__ wv, int Np,
                                               long long* __restrict__ out,
                                               int* __restrict__ ewv) {
  __shared__ int red[4];
  const size_t row = blockIdx.x;
  int mx = 0;
  for (int q = threadIdx.x; q < Np; q += 128)
    mx = max(mx, (int)((__double_as_longlong(wv[row * Np + q]) >> 52) & 0x7FF));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = max(max(red[0], red[1]), max(red[2], red[3]));
  const int E = exp_above_bits(mx);
  for (int q = threadIdx.x; q < Np; q += 128) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(wv[row * Np + q]);
    const int e = (int)((b >> 52) & 0x7FF), r = E + 1022 - e;
    long long v = 0;
    if (e && r <= 60) {
      v = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 9;
      v = r == 0 ? v : ((v >> (r - 1)) + 1) >> 1;
    }
    if ((long long)b < 0) v = -v;
    // low half as a signed 32-bit integer, the high half raised by what that takes off
    out[row * Np + q] = v + (long long)((unsigned long long)((uint32_t)v >> 31) << 32);
  }
  if (threadIdx.x == 0) ewv[row] = E;
}

// ---------------------------------------------------------------- table images
struct TabArgs {
  int op, L, N, n_r, NP, Q, Np, nb, nblk, nch, lastks, ntab;
  const double* src;   // rad, or the packed Legendre rows [t][(m, l)]
  const int* fexp;     // per row exponents, or null: fglob
  const int* rexp;
  int fglob;
  unsigned char* out;
};

__global__ void k_sl_table(TabArgs a) {
  const int kpad = 32 * (a.nch - 1) + 16 * a.lastks;
  const long long per = (long long)a.nblk * a.nb * kpad;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= per * a.ntab) return;
  const int table = (int)(i / per);
  int rem = (int)(i - per * table);
  const int blk = rem / (a.nb * kpad);
  rem -= blk * a.nb * kpad;
  const int row = rem / kpad, k = rem - row * kpad;  // row in the block, K index
  const int n = blk * a.nb + row;
  double v = 0.0;
  int F = a.fglob;
  const int L = a.L;
  if (a.op == OP_R1) {
    if (n < a.n_r && k < a.N) {
      v = a.src[((size_t)table * a.n_r + n) * a.N + k];
      F = a.fexp[table * a.n_r + n];
    }
  } else if (a.op == OP_R2) {
    if (n < a.N && k < a.n_r) {
      v = a.src[((size_t)table * a.n_r + k) * a.N + n] * oz_pow2(a.rexp[k]);
      F = a.fexp[table * a.N + n];
    }
  } else if (a.op == OP_L1 || a.op == OP_L2) {
    const int am = table >> 1, par = table & 1;
    const int t = a.op == OP_L1 ? n : k, l = am + par + 2 * (a.op == OP_L1 ? k : n);
    if (t < a.NP && l < L) {
      v = a.src[(size_t)t * theta_row_len(L) + theta_off(L, am) + l - am];
      if (a.op == OP_L2) F = a.fexp[table * a.nb + n];
    }
  } else {
    // P1: blocks = class x blocks of angles, rows q, K = mode; P2: rows = mode, K = q
    const int qb = a.op == OP_P1 ? a.nblk / 4 : 1;
    const int cls = a.op == OP_P1 ? blk / qb : table;
    const int q = a.op == OP_P1 ? (blk % qb) * a.nb + row : k;
    const int m = 2 * (a.op == OP_P1 ? k : row) + (cls & 1);
    if (q < a.Q && m < L && (cls < 2 || m > 0)) {
      const double x = 2.0 * (double)((long long)m * q % a.Np) / a.Np;
      v = cls < 2 ? cospi(x) : sinpi(x);
      if (fabs(v) < 1e-12) v = 0.0;
    }
  }
  const int ch = k >> 5, kk = k & 31;
  const size_t img = img_bytes(2, a.nb);
  unsigned char* o = a.out + ((size_t)table * a.nblk + blk) *
                                 (img * (a.nch - 1) + img_bytes(a.lastks, a.nb)) + ch * img +
                     (size_t)(kk >> 4) * kDig * (a.nb / 8) * 256 + (row >> 3) * 256 +
                     ((kk >> 3) & 1) * 128 + (row & 7) * 16 + (kk & 7) * 2;
  // |v| <= 2^F (a cosine of 1 is 2^54 exactly): round(v 2^(54 - F)) is exact in FP64's range
  const long long iv = (long long)rint(v * oz_pow2(kFix - F));
  const unsigned long long u = (unsigned long long)iv + 0x0080808080808080ull;
#pragma unroll
  for (int d = 0; d < kDig; ++d) {
    const int dig = (int)((u >> (8 * d)) & 255) - 128;
    *reinterpret_cast<__nv_bfloat16*>(o + (size_t)(kDig - 1 - d) * (a.nb / 8) * 256) =
        __float2bfloat16_rn((float)dig);
  }
}

struct Geo {
  int K, Nn, nb, nblk, nch, lastks, ntab;
  size_t bytes;
};

Geo geo(int op, int L, int N, int n_r, int n_theta, int n_phi) {
  const int NP = (n_theta + 1) / 2, Q = n_phi / 4 + 1, half = (L + 1) / 2;
  const int ks = (half + 15) / 16, nb2 = half <= 16 ? 16 : 32;
  Geo g{};
  switch (op) {
    case OP_R1: g = {N, n_r, 32, 0, 0, 0, L, 0}; break;
    case OP_R2: g = {n_r, N, 32, 0, 0, 0, L, 0}; break;
    case OP_L1: g = {16 * ks, NP, 16, 0, 0, 0, 2 * L, 0}; break;
    case OP_P1: g = {16 * ks, Q, 16, 0, 0, 0, 1, 0}; break;
    case OP_P2: g = {Q, 1, nb2, 0, 0, 0, 4, 0}; break;
    default: g = {NP, 1, nb2, 0, 0, 0, 2 * L, 0}; break;
  }
  g.nblk = (g.Nn + g.nb - 1) / g.nb * (op == OP_P1 ? 4 : 1);
  g.nch = (g.K + 31) / 32;
  g.lastks = (g.K - 32 * (g.nch - 1) + 15) / 16;
  g.bytes = (size_t)g.ntab * g.nblk * (img_bytes(2, g.nb) * (g.nch - 1) + img_bytes(g.lastks, g.nb));
  return g;
}

int exp_above(double m) {  // 2^e >= m
  int e = 0;
  if (m <= 0.0) return 0;
  std::frexp(m, &e);
  return e;
}

// Intermediates of one chunk of radial nodes. Larger chunks fill the last wave of each launch
// better than smaller ones keep the intermediates in the 129 MB L2: 80-state H.X at lmax 30
// 1.53 ms at 512 MB, 1.59 at 256, 1.74 at 128, 1.85 at 64.
constexpr size_t kChunkBytes = kSlChunkBytes;
constexpr int kMaxSB = 128;

size_t al(size_t x) { return (x + 255) & ~size_t(255); }

size_t node_bytes(int L, int n_theta, int n_phi, int SB) {
  const size_t NP = (n_theta + 1) / 2, M2 = 2 * L - 1, Q = n_phi / 4 + 1;
  return (2 * NP * M2 + (size_t)n_theta * 4 * Q) * SB * 8 + (size_t)n_theta * SB * 12 + SB * 4;
}

void chunking(int L, int n_r, int n_theta, int n_phi, int S, size_t bytes, int& SB, int& kc) {
  const int nblk = (S + kMaxSB - 1) / kMaxSB;
  SB = (S + nblk - 1) / nblk;
  const size_t nb = node_bytes(L, n_theta, n_phi, SB);
  int most = (int)std::max<size_t>(1, bytes / nb);
  const int nchunks = (n_r + most - 1) / most;
  kc = (n_r + nchunks - 1) / nchunks;
}

template <class... P, class... A>
cudaError_t launch_chain(bool early, void (*kernel)(P...), unsigned grid_x, unsigned grid_y,
                         int threads, int smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid_x, grid_y);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int OP, int NB, bool SMALL>
cudaError_t launch_sl(const SlArgs& a, const Geo& g, cudaStream_t st) {
  const int ks = g.nch > 1 ? 2 : g.lastks;
  const int smem = ks * (kDig * kADigit + 2 * kDig * (NB / 8) * 256);
  cudaError_t e =
      cudaFuncSetAttribute(k_sl<OP, NB, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  const int fit = std::min(sl_ctas(OP, NB), 227 * 1024 / (smem + 3 * 1024));
  const unsigned grid = (unsigned)std::min<long long>(a.ntiles, (long long)fit * nsm);
  return launch_chain(a.early, k_sl<OP, NB, SMALL>, grid, 1, kSlThreads, smem, st, a);
}
// P2, L2: up to 16 or 32 modes per class, up to 32 or 64 k
template <int OP>
cudaError_t launch_sl2(const SlArgs& a, const Geo& g, cudaStream_t st) {
  if (g.nb == 32) return launch_sl<OP, 32, false>(a, g, st);
  return g.nch == 1 ? launch_sl<OP, 16, true>(a, g, st) : launch_sl<OP, 16, false>(a, g, st);
}

}  // namespace

bool sliced_hx_eligible(int L, int N, int n_r, int n_theta, int n_phi) {
  return L <= 63 && N <= 448 && n_r <= 448 && (n_theta + 1) / 2 <= 64 && n_phi / 4 + 1 <= 64;
}

// CS_ANGULAR_KERNEL keeps the FMA kernels where it names one of them: stream, rp.. or fma; wide
// names the three-pass blocks, of which FP64 has none. gm and tc choose among FP32 and mixed
// kernels and, like the empty string, leave these calls alone.
bool sliced_hx_enabled(bool df) {
  const char* e = getenv("CS_ANGULAR_KERNEL");
  if (!e) return true;
  const bool fma = e[0] == 's' || (e[0] == 'r' && e[1] == 'p') || e[0] == 'f';
  return !fma && !(df && e[0] == 'w');
}

// What SlPlan takes beside the intermediates, and one node of them: the least it runs in.
size_t sliced_hx_fixed_bytes(int n_r, int S) { return (size_t)n_r * S * 4 + 7 * 256; }
size_t sliced_hx_node_bytes(int L, int n_theta, int n_phi, int S) {
  return node_bytes(L, n_theta, n_phi, std::min(S, kMaxSB));
}

// An upper bound of what SlPlan takes that grows with S, so that a workspace sized for S states
// serves every smaller block: at most n_r nodes, and at most kChunkBytes or one node.
size_t sliced_hx_work_bytes(int L, int n_r, int n_theta, int n_phi, int S) {
  const size_t node = node_bytes(L, n_theta, n_phi, std::min(S, kMaxSB));
  return std::min((size_t)n_r * node, kChunkBytes + node) + sliced_hx_fixed_bytes(n_r, S);
}

void free_sliced_tables(SlicedTables& T) {
  for (int i = 0; i < 6; ++i) {
    if (T.tab[i]) cudaFree(T.tab[i]);
    T.tab[i] = nullptr;
  }
  for (void** p : {(void**)&T.exps, (void**)&T.wv, (void**)&T.ewv}) {
    if (*p) cudaFree(*p);
    *p = nullptr;
  }
}

cudaError_t build_sliced_tables(const HostTables& H, const double* rad, const double* theta,
                                SlicedTables& T) {
  const int L = H.L, N = H.N, NP = (H.n_theta + 1) / 2, RL = theta_row_len(L);
  const int nb2 = (L + 1) / 2 <= 16 ? 16 : 32;
  // exponents: R1 rows [l][k], R2 rows [l][n], L2 rows [am][par][i], radial scaling [k]
  std::vector<int> ex((size_t)L * H.n_r + (size_t)L * N + (size_t)2 * L * nb2 + H.n_r, 0);
  int* f1 = ex.data();
  int* f2 = f1 + (size_t)L * H.n_r;
  int* fl = f2 + (size_t)L * N;
  int* re = fl + (size_t)2 * L * nb2;
  for (int k = 0; k < H.n_r; ++k) re[k] = exp_above(H.r[k]);
  std::vector<double> mx(N);
  for (int l = 0; l < L; ++l) {
    std::fill(mx.begin(), mx.end(), 0.0);
    for (int k = 0; k < H.n_r; ++k) {
      const double* row = H.rad.data() + ((size_t)l * H.n_r + k) * N;
      double m = 0.0;
      const double sc = std::ldexp(1.0, re[k]);
      for (int n = 0; n < N; ++n) {
        m = std::max(m, std::fabs(row[n]));
        mx[n] = std::max(mx[n], std::fabs(row[n]) * sc);
      }
      f1[(size_t)l * H.n_r + k] = exp_above(m);
    }
    for (int n = 0; n < N; ++n) f2[(size_t)l * N + n] = exp_above(mx[n]);
  }
  double tmax = 0.0;
  for (int am = 0; am < L; ++am)
    for (int l = am; l < L; ++l) {
      double m = 0.0;
      for (int t = 0; t < NP; ++t)
        m = std::max(m, std::fabs(H.theta[(size_t)t * RL + theta_off(L, am) + l - am]));
      tmax = std::max(tmax, m);
      fl[(size_t)(am * 2 + ((l - am) & 1)) * nb2 + (l - am) / 2] = exp_above(m);
    }
  T.F1 = exp_above(tmax);
  T.off_f2 = (size_t)L * H.n_r;
  T.off_fl = T.off_f2 + (size_t)L * N;
  T.off_re = T.off_fl + (size_t)2 * L * nb2;
  cudaError_t e;
  if ((e = cudaMalloc((void**)&T.exps, ex.size() * sizeof(int))) != cudaSuccess) return e;
  if ((e = cudaMemcpy(T.exps, ex.data(), ex.size() * sizeof(int), cudaMemcpyHostToDevice)) !=
      cudaSuccess)
    return e;
  const size_t rows = (size_t)H.n_r * H.n_theta;
  if ((e = cudaMalloc((void**)&T.wv, rows * H.n_phi * 8)) != cudaSuccess) return e;
  if ((e = cudaMalloc((void**)&T.ewv, rows * sizeof(int))) != cudaSuccess) return e;
  for (int op = 0; op < 6; ++op) {
    const Geo g = geo(op, L, N, H.n_r, H.n_theta, H.n_phi);
    if ((e = cudaMalloc((void**)&T.tab[op], g.bytes)) != cudaSuccess) return e;
    TabArgs a{op, L, N, H.n_r, NP, H.n_phi / 4 + 1, H.n_phi, g.nb, g.nblk, g.nch, g.lastks, g.ntab};
    a.src = (op == OP_R1 || op == OP_R2) ? rad : theta;
    a.fexp = op == OP_R1 ? T.exps : op == OP_R2 ? T.exps + T.off_f2 : T.exps + T.off_fl;
    a.rexp = T.exps + T.off_re;
    a.fglob = op == OP_L1 ? T.F1 : 0;
    a.out = T.tab[op];
    const long long tot = (long long)g.ntab * g.nblk * g.nb * (32 * (g.nch - 1) + 16 * g.lastks);
    k_sl_table<<<(unsigned)((tot + 255) / 256), 256>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaDeviceSynchronize();
}

cudaError_t launch_sliced_wv(const SlicedTables& T, const double* wv, int rows, int n_phi,
                             cudaStream_t st) {
  k_sl_wv<<<(unsigned)rows, 128, 0, st>>>(wv, n_phi, T.wv, T.ewv);
  return cudaGetLastError();
}

namespace {

// One block's launches: the arguments shared by all operations and the workspace's parts.
struct SlPlan {
  const HostTables& H;
  const SlicedTables& T;
  cudaStream_t st;
  SlArgs a{};
  int L2, Np, SBm, kcm, n = 0;  // n: kernels launched
  int *shP, *uP, *U, *EG;
  long long rad_tiles = 0;
  Geo g[6];

  SlPlan(const HostTables& H_, const SlicedTables& T_, int S, double* G, void* work, int* err,
         cudaStream_t st_, size_t bytes = kChunkBytes)
      : H(H_), T(T_), st(st_), L2(H_.L * H_.L), Np(H_.n_phi) {
    const int L = H.L, NP = (H.n_theta + 1) / 2, half = (L + 1) / 2;
    for (int op = 0; op < 6; ++op) g[op] = geo(op, L, H.N, H.n_r, H.n_theta, H.n_phi);
    chunking(L, H.n_r, H.n_theta, H.n_phi, S, bytes, SBm, kcm);
    for (int l = 0; l < L; ++l) rad_tiles += ((long long)(2 * l + 1) * S + kRows - 1) / kRows;
    char* p = static_cast<char*>(work);
    auto take = [&](size_t b) {
      char* at = p;
      p += al(b);
      return at;
    };
    const size_t mrows = (size_t)kcm * H.n_theta * SBm;
    a.L = L;
    a.N = H.N;
    a.n_r = H.n_r;
    a.Nt = H.n_theta;
    a.NP = NP;
    a.M2 = 2 * L - 1;
    a.Q = Np / 4 + 1;
    a.S = S;
    // An early launch hides a few microseconds per kernel, which counts in small problems: lmax 10,
    // 16 states 88 -> 76 us, 64 states 129 -> 114. In larger ones the next kernel's CTAs take the
    // room of the running one's unevenly: lmax 30, one state 221 -> 324 us; lmax 23, 4 states 160
    // -> 167; the two meet near rows L^2 = 7M at lmax 16 (16 states: 130 us both).
    a.early = L <= 17 && (long long)H.n_r * H.n_theta * S * L2 < 6000000;
    a.F1 = T.F1;
    a.ks = (half + 15) / 16;
    a.nb2 = half <= 16 ? 16 : 32;
    a.rexp = T.exps + T.off_re;
    a.G = G;
    a.FA = reinterpret_cast<long long*>(take((size_t)kcm * 2 * NP * a.M2 * SBm * 8));
    a.W = reinterpret_cast<long long*>(take(mrows * 4 * a.Q * 8));
    a.eW = reinterpret_cast<int*>(take(mrows * 4));
    shP = reinterpret_cast<int*>(take(mrows * 4));
    uP = reinterpret_cast<int*>(take(mrows * 4));
    U = reinterpret_cast<int*>(take((size_t)kcm * SBm * 4));
    EG = reinterpret_cast<int*>(take((size_t)H.n_r * S * 4));
    a.shP = shP;
    a.uP = uP;
    a.U = U;
    a.Uw = U;
    a.EG = EG;
    a.err = err;
  }
  int rows() const { return a.kc * a.Nt; }  // grid rows of the chunk
  long long row_tiles() const { return ((long long)rows() * a.SB + kRows - 1) / kRows; }
  cudaError_t radial_synth(const double* X, long long ld) {
    a.X = X;
    a.ld = ld;
    a.tab = T.tab[OP_R1];
    a.fexp = T.exps;
    a.ntiles = rad_tiles;
    ++n;
    return launch_sl<OP_R1, 32, false>(a, g[OP_R1], st);
  }
  cudaError_t radial_anal(const Epilogue<double>& ep) {
    a.ep = ep;
    a.tab = T.tab[OP_R2];
    a.fexp = T.exps + T.off_f2;
    a.ntiles = rad_tiles;
    ++n;
    return launch_sl<OP_R2, 32, false>(a, g[OP_R2], st);
  }
  cudaError_t scales() {
    ++n;
    return launch_chain(a.early, k_sl_gexp, (a.S + 31) / 32, H.n_r, 256, 0, st, a.G, L2, a.S, EG);
  }
  void legendre_tiles() {
    const int nodes = a.kc * a.SB;
    a.ntiles = 2ll * ((nodes + kRows - 1) / kRows) +
               2ll * (a.L - 1) * ((2 * nodes + kRows - 1) / kRows);
  }
  // L1 and P1 of the chunk: the class sums of its grid rows in W
  cudaError_t synth() {
    legendre_tiles();
    a.tab = T.tab[OP_L1];
    n += 2;
    cudaError_t e = launch_sl<OP_L1, 16, true>(a, g[OP_L1], st);
    if (e != cudaSuccess) return e;
    a.tab = T.tab[OP_P1];
    a.ntiles = row_tiles();
    return launch_sl<OP_P1, 16, true>(a, g[OP_P1], st);
  }
  // P2 and L2: from the folded W, its shifts and units to G'
  cudaError_t anal() {
    a.tab = T.tab[OP_P2];
    a.ntiles = 4 * row_tiles();
    n += 2;
    cudaError_t e = launch_sl2<OP_P2>(a, g[OP_P2], st);
    if (e != cudaSuccess) return e;
    legendre_tiles();
    a.tab = T.tab[OP_L2];
    a.fexp = T.exps + T.off_fl;
    return launch_sl2<OP_L2>(a, g[OP_L2], st);
  }
  cudaError_t clear_units() {
    return cudaMemsetAsync(U, 0x80, (size_t)a.kc * a.SB * sizeof(int), st);
  }
  // body() for every block of states and chunk of radial nodes
  template <class F>
  cudaError_t chunks(F body) {
    for (a.s0 = 0; a.s0 < a.S; a.s0 += SBm)
      for (a.k0 = 0; a.k0 < H.n_r; a.k0 += kcm) {
        a.SB = std::min(SBm, a.S - a.s0);
        a.kc = std::min(kcm, H.n_r - a.k0);
        const cudaError_t e = body();
        if (e != cudaSuccess) return e;
      }
    return cudaSuccess;
  }
};

unsigned warp_grid(long long items) { return (unsigned)((items + 7) / 8); }

#define SL_TRY(expr)                          \
  do {                                        \
    const cudaError_t e_ = (expr);            \
    if (e_ != cudaSuccess) return e_;         \
  } while (0)

}  // namespace

cudaError_t launch_sliced_hx(const HostTables& H, const SlicedTables& T, int S, const double* X,
                             long long ld, double* G, const Epilogue<double>& ep, void* work,
                             int* err, cudaStream_t st, int stage, int* launches, size_t bytes) {
  SlPlan p(H, T, S, G, work, err, st, bytes);
  SlArgs& a = p.a;
  cudaError_t e;
  if (stage == 0) {
    e = p.radial_synth(X, ld);
  } else if (stage == 2) {
    e = p.radial_anal(ep);
  } else {
    SL_TRY(p.scales());
    e = p.chunks([&]() -> cudaError_t {
      SL_TRY(p.synth());
      const int rows = p.rows();
      ++p.n;
      SL_TRY(launch_chain(a.early, k_sl_pointwise, (unsigned)(((long long)rows * a.SB + 31) / 32), 1, 256, 0,
                        st, a.W, a.eW, T.wv, T.ewv, rows, a.SB, a.Nt, p.Np, a.Q, a.k0, p.shP, p.uP,
                        p.U));
      return p.anal();
    });
  }
  *launches = p.n;
  return e;
}

cudaError_t launch_sliced_grid(const HostTables& H, const SlicedTables& T, int S, const double* X,
                               long long ld, double* G, double* f, void* work, int* err,
                               cudaStream_t st, int* launches) {
  SlPlan p(H, T, S, G, work, err, st);
  SlArgs& a = p.a;
  if (X) SL_TRY(p.radial_synth(X, ld));
  SL_TRY(p.scales());
  SL_TRY(p.chunks([&]() -> cudaError_t {
    SL_TRY(p.synth());
    const int rows = p.rows();
    ++p.n;
    return launch_chain(a.early, k_sl_grid, warp_grid((long long)rows * a.SB), 1, 256, 0, st, a.W, a.eW, rows,
                      a.SB, a.s0, a.k0, a.Nt, p.Np, a.Q, H.n_r, f);
  }));
  *launches = p.n;
  return cudaSuccess;
}

cudaError_t launch_sliced_density(const HostTables& H, const SlicedTables& T, int S,
                                  const double* X, long long ld, const double* occ, bool add,
                                  double* G, double* rho, void* work, int* err, cudaStream_t st,
                                  int* launches) {
  SlPlan p(H, T, S, G, work, err, st);
  SlArgs& a = p.a;
  SL_TRY(p.radial_synth(X, ld));
  SL_TRY(p.scales());
  const int smem = (4 * a.Q * 33 + 32) * (int)sizeof(double);
  SL_TRY(cudaFuncSetAttribute(k_sl_density, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  SL_TRY(p.chunks([&]() -> cudaError_t {
    SL_TRY(p.synth());
    ++p.n;
    return launch_chain(a.early, k_sl_density, (unsigned)p.rows(), 1, 256, smem, st, a.W, a.eW, a.SB, a.Nt,
                      p.Np, a.Q, a.k0, occ + a.s0, rho, add || a.s0 > 0 ? 1 : 0);
  }));
  *launches = p.n;
  return cudaSuccess;
}

cudaError_t launch_sliced_forward(const HostTables& H, const SlicedTables& T, int S,
                                  const double* g, const double* wkj, double* G,
                                  const Epilogue<double>& ep, void* work, int* err,
                                  cudaStream_t st, int* launches) {
  SlPlan p(H, T, S, G, work, err, st);
  SlArgs& a = p.a;
  SL_TRY(p.chunks([&]() -> cudaError_t {
    SL_TRY(p.clear_units());
    const int rows = p.rows();
    ++p.n;
    SL_TRY(launch_chain(a.early, k_sl_fold, warp_grid((long long)rows * a.SB), 1, 256, 0, st, g, wkj, rows,
                      a.SB, a.s0, a.k0, a.Nt, p.Np, a.Q, H.n_r, a.W, p.shP, p.uP, p.U));
    return p.anal();
  }));
  SL_TRY(p.radial_anal(ep));
  *launches = p.n;
  return cudaSuccess;
}

}  // namespace cs
