// FP64 squares and products on the tcgen05 tensor cores, as exact sums of digit products.
//
// The FP64 pipe of this GPU runs 2 fused multiply-adds per clock and SM; the tensor cores run about
// 4096 with fp16 inputs.  A row x_i of X is scaled by 2^-e_i (|x_ik| <= 2^(e_i - 1), ||x_i|| < 2^e_i) and
// written as ND = 7 signed digits of 8 bits,
//     x_ik 2^-e_i = sum_a d_a 2^(-8 (a + 1)),   |d_a| <= 128   (56 bits, rounded to nearest),
// each an integer that fp16 holds exactly.  Then
//     sum_k x_ik x_jk = 2^(e_i + e_j) sum_s 2^(-8 (s + 2)) V_s,   V_s = sum over k and a + b = s of d_a d'_b,
// and the 34 digit products with s <= 7 are formed on the tensor cores.  The FP32 accumulators hold every
// V_s exactly up to 2^24, and each is drained before it can pass that (period); the V_s are added in 64-bit
// integer registers in units of 2^-62 (|sum| < 1 by Cauchy's inequality, so it fits) and the total is rounded
// to FP64 once.  V_0 .. V_5 are whole numbers of units; V_6 2^-2 and V_7 2^-10 are rounded to the unit at each of
// their drains, at most ld / 128 + ks times each in the ks CTAs that share a tile, so the last bits depend on the
// split, and with it on the device's SMs and clusters.  (Digit splittings of this kind: K. Ozaki, T. Ogita, S. Oishi,
// S. M. Rump, "Error-free transformations of matrix multiplication by using fast routines of matrix multiplication
// and its applications", Numer. Algorithms 59, 2012.)
//
// Error against the exact product, in units of 2^(e_i + e_j) <= 16 ||x_i|| ||x_j||: the digits' own rounding, at most
// 2^-57 per value; the products with s >= 8 that are left out, at most 5.02 K 2^-66 and for random digits about
// sqrt(5 K) 2^-67.6; at most ld / 128 + ks units of 2^-62 from the drains.  In all at most (2^-54 sqrt(K) + 2^-59 K)
// ||x_i|| ||x_j|| and half a unit in the last place, against K 2^-53 |x_i| |x_j| for an FMA chain.  The bound holds for
// norms only: an element far below its row's norm has fewer digits (56 - k bits at 2^-k of the scale), and where
// |x_i| |x_j| is far below ||x_i|| ||x_j||, as far from the diagonal of a local matrix, the result loses the relative
// accuracy that an FMA chain keeps (entries that decay by ten per eight off the diagonal, one square: 2e-11 of an
// element of 6e-8, 2e-6 at 7e-13; below about 1e-17 noise or zero).
// ||D - D_exact||_F / ||D||_F against the exact projector at N = 400 / 1001 / 1500 (McW-ACC) / 2048: 8.5e-15 / 2.0e-14 /
// 2.3e-14 / 4.2e-14, with FMA chains 1.3e-14 / 2.9e-14 / 4.2e-14 / 6.1e-14.  The lower floor of ||X - X^2|| can move the
// stop by a few steps where it falls on that floor (12 of 60 drawn problems), with the smaller error each time.
//
// Time of one purification against the FP64 units (64 x 64 tiles, 0.98 of their peak at large N): N = 400
// 1.34 ms against 18.4, N = 1500 (McW-ACC) 5.18 against 77.5, N = 2048 16.7 against 418.
//
// Tiles are 128 x bn (bn = 32 or 64), over the upper triangle; where they are fewer than the SMs, or fill the
// last round badly, a cluster of ks CTAs shares a tile's k range (choose_tiles): each sums its part, then gives
// each of the others its columns through distributed shared memory, and every CTA finishes 64 / ks columns.  A stage holds
// the 7 digits of 32 k-columns of both operands, so 14 digit planes feed 34 products.  What bounds the
// products is the reading of A from shared memory: a 128 x 64 x 16 product takes 48 clocks for 32 of
// arithmetic.  Warp roles as in the other tensor-core kernels: warp 0 copies, warp 1 issues the products,
// warps 4..11 drain and run the epilogue.  Every wait is bounded (2 s).
#include <cuda_fp16.h>

#include <cstring>

#include "../../include/sp2_testing.h"
#include "sp2_common.cuh"
#include "sp2_f64_tc.cuh"
#include "sp2_kernels.h"
#include "tc_ptx.cuh"

namespace sp2 {
namespace f64tc {

using namespace sp2::ptx;

constexpr int DBITS = 8;                 // bits per digit
constexpr int BM = 128;                  // tile rows
constexpr int NS = 8;                    // digit sums kept: a + b <= 7, 34 products
constexpr int KB = 32;                   // k-columns per stage: 64-byte rows, 64-byte swizzle
// Digits in memory, and in a stage: for each block of 32 k-columns, groups of 8 rows; a group holds its ND
// digits one after the other, each 8 rows x 64 bytes with the 16-byte chunks of row r exchanged by
// chunk ^ (r / 2 % 4), the 64-byte swizzle that the tensor cores read.  A tile's rows are then one contiguous
// piece of memory: two plain bulk copies fill a stage and no tensor map is needed (boxes of a tensor map over
// planes of digits were as fast).
constexpr int ROWB = KB * 2;             // bytes of one digit row
constexpr int DIGB = 8 * ROWB;           // one digit of a row group
constexpr int GRPB = ND * DIGB;          // a row group: 3584 bytes
constexpr int MAXSTG = 3;
constexpr int THREADS = 384;             // warps 0 TMA, 1 MMA, 2 idle; 8 epilogue warps
constexpr int kBadExp = INT32_MIN;       // exponent of a row that holds a NaN or an infinity
constexpr uint64_t kWaitNs = 2000000000ull;

constexpr int A_BYTES = BM / 8 * GRPB;   // 56 KB
__host__ __device__ constexpr int b_bytes(int bn) { return bn / 8 * GRPB; }
__host__ __device__ constexpr int stage_bytes(int bn) { return A_BYTES + b_bytes(bn); }
__host__ __device__ constexpr int stages_of(int bn) {
  return 226 * 1024 / stage_bytes(bn) < MAXSTG ? 226 * 1024 / stage_bytes(bn) : MAXSTG;
}
// Exchange buffer of a split tile: from each of the other CTAs, the sums of this CTA's columns.
__host__ __device__ constexpr int exchange_bytes(int ks) { return (ks - 1) * (BM * 64 * 8 / ks); }
__host__ __device__ constexpr int smem_bytes(int bn, int ks) {
  return stages_of(bn) * stage_bytes(bn) + exchange_bytes(ks) + 1024;
}
static_assert(smem_bytes(64, 8) <= 227 * 1024 - 512, "shared memory");
static_assert(stages_of(64) == 2 && stages_of(32) == 3, "stages");

// Each digit sum has a tensor-memory accumulator of its own (NS x bn columns), closed and drained once in
// period(s) blocks of 32 k-columns, at phase(s), and at the end of the tile: a drain costs a warp about 1.2 k clocks,
// and with two buffers in turn, drained every block, the drains took three times the products.  The phases spread
// the drains over the blocks, two at most in one, so that a block's products (3 k clocks) hide them: a sum's next
// product comes a block after it was closed.  A product adds at most 2^14 per term, so the sums stay exact:
// (pairs of s) x 32 period <= 2^10.
__host__ __device__ constexpr int period(int s) { return s < 2 ? 16 : (s < 4 ? 8 : 4); }
__host__ __device__ constexpr int phase(int s) { return (int)((0x210315b7u >> (4 * s)) & 15u); }   // 7 11 5 1 3 0 1 2
__host__ __device__ constexpr bool closes(int kb, int s) { return (kb & (period(s) - 1)) == phase(s); }
// The sums that close at blocks kb = 8 h .. 8 h + 7 (mod 16), a byte of bits each.
__host__ __device__ constexpr uint64_t closing(int h) {
  uint64_t m = 0;
  for (int kb = 0; kb < 8; ++kb)
    for (int s = 0; s < NS; ++s) m |= (uint64_t)(closes(8 * h + kb, s) ? 1 : 0) << (8 * kb + s);
  return m;
}
__host__ __device__ constexpr int first_pair(int s) { return s < ND ? 0 : s - ND + 1; }   // smallest a of a + b = s
__host__ __device__ constexpr int pairs(int s) { return (s < ND ? s : ND - 1) - first_pair(s) + 1; }
__host__ __device__ constexpr bool sums_exact() {
  for (int s = 0; s < NS; ++s)
    if (pairs(s) * KB * period(s) > (1 << 10)) return false;
  return true;
}
static_assert(sums_exact(), "digit sums exact in FP32");

// Upper tiles: row I of tiles holds the columns J >= I * BM / bn of ceil(ld / bn).
__host__ __device__ inline int tiles_of(int ld, int bn) {
  const int rows = (ld + BM - 1) / BM, cols = (ld + bn - 1) / bn;
  int n = 0;
  for (int I = 0; I < rows; ++I) n += cols - I * (BM / bn);
  return n;
}

__device__ __forceinline__ void locate(int t, int cols, int step, int& I, int& J) {
  int i = 0, w = cols;
  while (t >= w) { t -= w; ++i; w -= step; }
  I = i;
  J = i * step + t;
}

// ---- digits --------------------------------------------------------------------------------
constexpr int DT = 256;                  // one warp per row of a group

__device__ __forceinline__ void load4(const double* p, double (&x)[4]) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(x[0]), "=d"(x[1]), "=d"(x[2]), "=d"(x[3]) : "l"(p));
}
__device__ __forceinline__ void store4(double* p, const double (&x)[4]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(x[0]), "d"(x[1]), "d"(x[2]), "d"(x[3])
               : "memory");
}

// |x| 2^(1023 - m) as FP32 (rounded toward zero), m the largest exponent field of the row.
__device__ __forceinline__ float scaled_abs(double x, int m) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
  const int e = (int)(hi >> 20) - m + 127;
  if (e <= 0) return 0.f;
  return __uint_as_float(((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

// x 2^(56 - e), rounded to the nearest integer (|x| <= 2^(e - 1)).
__device__ __forceinline__ long long fixed56(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return 0;                               // zero (subnormals are below every unit used)
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = ex - 1075 + ND * DBITS - e;
  unsigned long long y;
  if (sh >= 0) y = m << sh;                            // sh <= 3 by the choice of e
  else if (sh < -54) y = 0;
  else y = (m + (1ull << (-sh - 1))) >> -sh;
  return b < 0 ? -(long long)y : (long long)y;
}

// One warp per row, 8 rows (a row group) per CTA: the row's exponent, then its digits.  Bound by memory
// (8 B read, 14 B written per value).
__global__ void __launch_bounds__(DT)
digits_kernel(const DevState* st, const double* buf0, const double* buf1, const double* S, int ld, int N, __half* dig,
              int32_t* exps) {
  // the stop test beside it may set st->done: one reading per warp, whose lanes stay together (the digits of a run
  // that is over are not used)
  int over = 0;
  if ((threadIdx.x & 31) == 0) over = *static_cast<const volatile int32_t*>(&st->done);
  if (__shfl_sync(0xffffffffu, over, 0)) return;
  const double* X = S ? S : (st->wrote ? buf1 : buf0);
  const int rr = threadIdx.x >> 5, r = blockIdx.x * 8 + rr, lane = threadIdx.x & 31;
  if (r >= N) return;
  const double* row = X + (int64_t)r * ld;
  int m = 0;
  for (int c = 4 * lane; c < ld; c += 128) {
    double x[4];
    load4(row + c, x);
    #pragma unroll
    for (int j = 0; j < 4; ++j) m = max(m, (__double2hiint(x[j]) >> 20) & 0x7ff);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  const bool bad = m == 0x7ff;
  float n2 = 0.f;
  for (int c = 4 * lane; c < ld; c += 128) {
    double x[4];
    load4(row + c, x);
    #pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float f = scaled_abs(x[j], m);
      n2 = fmaf(f, f, n2);
    }
  }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  n2 *= 1.001f;                                        // above the rounding of the sum and of its terms
  // |x| < 2^(m - 1022) <= 2^(e - 1) and ||x||^2 <= n2 2^(2 (m - 1023)) < 2^(2 e)
  const int lg = (__float_as_int(n2) >> 23) - 127;     // floor(log2 n2), n2 >= 1
  const int e = bad || m == 0 ? 0 : max(m - 1021, m - 1023 + lg / 2 + 1);
  if (lane == 0) exps[r] = bad ? kBadExp : e;
  const int64_t kstride = (int64_t)padded_rows(ld) / 8 * GRPB;
  uint8_t* out = reinterpret_cast<uint8_t*>(dig) + (int64_t)blockIdx.x * GRPB + rr * ROWB;
  for (int c = 4 * lane; c < ld; c += 128) {
    double x[4];
    load4(row + c, x);
    long long y[4];
    #pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = bad ? 0 : fixed56(x[j], e);
    uint8_t* dst = out + (c / KB) * kstride + (((c % KB) / 8) ^ (rr / 2)) * 16 + (c % 8) * 2;
    #pragma unroll
    for (int a = ND - 1; a >= 0; --a) {
      // digit of 8 bits in [-128, 127] (the top one takes what is left, at most 128): 1536 + d as fp16
      // bits is 0x6600 + d, and subtracting 1536 is exact
      int d[4];
      #pragma unroll
      for (int j = 0; j < 4; ++j) {
        d[j] = a ? (int)(int8_t)y[j] : (int)y[j];
        y[j] = (y[j] - d[j]) >> DBITS;
      }
      const unsigned w0 = (unsigned)(0x6600 + d[0]) | ((unsigned)(0x6600 + d[1]) << 16);
      const unsigned w1 = (unsigned)(0x6600 + d[2]) | ((unsigned)(0x6600 + d[3]) << 16);
      const __half2 off = __float2half2_rn(1536.f);
      uint2 o;
      const __half2 h0 = __hsub2(*reinterpret_cast<const __half2*>(&w0), off);
      const __half2 h1 = __hsub2(*reinterpret_cast<const __half2*>(&w1), off);
      o.x = *reinterpret_cast<const unsigned*>(&h0);
      o.y = *reinterpret_cast<const unsigned*>(&h1);
      *reinterpret_cast<uint2*>(dst + a * DIGB) = o;
    }
  }
}

// ---- product ---------------------------------------------------------------------------------
struct Args {
  DevState* st;
  double *buf0, *buf1, *S;
  double* part;
  const uint8_t *digA, *digB;            // digits of the A and the B operand
  const int32_t *ea, *eb;                // row exponents of the A and the B operand
  uint64_t wait_ns;                      // limit of every wait
  int32_t ld, tiles, op;
  int32_t hook;                          // 0, or a Hook of the testing entry
};

enum Hook : int32_t {
  HOOK_SKIP_COPY = 1,   // CTA 0 leaves its first stage uncopied: waits run out
  HOOK_OTHERS_OVER = 2, // the CTAs of a cluster but its first find the run over
  HOOK_FIRST_OVER = 3   // only the first does
};

// What the epilogue writes: out = pk ? s : 2 x - s, or ca s + cb x + cc I with gen set.
struct Poly {
  const double* in;
  double* out;
  double ca, cb, cc;
  int gen, pk;
};

__device__ __forceinline__ Poly poly_of(const Args& a) {
  const DevState* st = a.st;
  Poly p;
  p.ca = p.cb = p.cc = 0.0;
  p.gen = 0;
  p.pk = 1;
  const int k = st->k;
  if (a.op == OP_MCW_SQ) {               // S_s = alpha^2 X^2 + 2 alpha c X + c^2 I, c = (1 - alpha) / 2
    const double al = st->alpha[k + 1], c = 0.5 * (1.0 - al);
    p.in = (k & 1) ? a.buf1 : a.buf0;
    p.out = a.S;
    p.gen = 1; p.ca = al * al; p.cb = 2.0 * al * c; p.cc = c * c;
  } else if (a.op == OP_MCW_PROD) {      // X_k = (3 - 2 c) S_s - 2 alpha S_s X_{k-1}, k already recorded
    const double al = st->alpha[k], c = 0.5 * (1.0 - al);
    p.in = a.S;
    p.out = (k & 1) ? a.buf1 : a.buf0;
    p.gen = 1; p.ca = -2.0 * al; p.cb = 3.0 - 2.0 * c;
  } else {
    p.in = (k & 1) ? a.buf1 : a.buf0;
    p.out = (k & 1) ? a.buf0 : a.buf1;
    if (st->acc) {
      p.pk = acc_step(st, k + 1, p.ca, p.cb, p.cc);
      p.gen = 1;
    } else {
      p.pk = st->tr[k] > (double)st->nocc ? 1 : 0;     // Alg. 3 trace test
    }
  }
  return p;
}

__device__ __forceinline__ void give_up(DevState* st, volatile int* abort_s) {
  *abort_s = 1;
  atomicExch(&st->status, (int)SP2_ERR_TIMEOUT);
  st->out_mode = OUT_NAN;
  st->done = 1;
}

// 16 or 32 consecutive 32-bit tensor-memory columns.
__device__ __forceinline__ void tmem_ld(uint32_t addr, uint32_t (&r)[32]) { tmem_ld32(addr, r); }
__device__ __forceinline__ void tmem_ld(uint32_t addr, uint32_t (&r)[16]) { tmem_ld16(addr, r); }

// Four 64-bit sums whose low and high words lie in two tensor-memory areas.
__device__ __forceinline__ void load_sums(uint32_t lo, uint32_t hi, long long (&t)[4]) {
  uint32_t a[4], b[4];
  tmem_ld4(lo, a);
  tmem_ld4(hi, b);
  tmem_wait_ld();
  #pragma unroll
  for (int j = 0; j < 4; ++j) t[j] = (long long)(((unsigned long long)b[j] << 32) | a[j]);
}

// T += V_s of one period, in units of 2^-62: the weight of s is 2^(46 - 8 s), for s <= 1
// in the high word alone (modulo 2^32: the total fits); s = 6 and 7 are rounded to the unit.  One piece of code for every s: as
// straight-line code for each of them the drains were bound by the instruction fetch (2 k clocks a drain; the integer
// conversions, 8.5 clocks a warp each, take 550).
template <int G>
__device__ __forceinline__ void add_digit_sums(int s, const uint32_t (&raw)[G], long long (&T)[G]) {
  if (s <= 1) {                          // only the high word changes
    const int m = 1 << (14 - 8 * s);
    #pragma unroll
    for (int j = 0; j < G; ++j)
      T[j] += (long long)((unsigned long long)((unsigned)__float2int_rn(__uint_as_float(raw[j])) * (unsigned)m) << 32);
    return;
  }
  const float scale = s <= 5 ? 1.f : (s == 6 ? 0x1p-2f : 0x1p-10f);
  const int m = s <= 5 ? 1 << (46 - 8 * s) : 1;
  #pragma unroll
  for (int j = 0; j < G; ++j) T[j] += (long long)__float2int_rn(__uint_as_float(raw[j]) * scale) * m;
}

// T 2^(ei + ej - 62) where the result is no normal number.
__device__ __noinline__ double scaled_sum_rare(long long t, int ei, int ej) {
  if (ei == kBadExp || ej == kBadExp) return __longlong_as_double(0x7ff8000000000000ll);
  return ldexp((double)t, ei + ej - 62);
}

// T 2^(ei + ej - 62): the scale goes into the exponent field where the result is a normal number (an FP64
// multiplication takes 70 clocks a warp here, the conversion from the integer 6).
__device__ __forceinline__ double scaled_sum(long long t, int ei, int ej) {
  const int es = ei + ej - 62;
  if (ei == kBadExp || ej == kBadExp || es <= -1000 || es >= 900) return scaled_sum_rare(t, ei, ej);
  const double s = (double)t;
  return t ? __hiloint2double(__double2hiint(s) + (es << 20), __double2loint(s)) : 0.0;
}

template <int BN, int KS>
__global__ void __cluster_dims__(KS, 1, 1) __launch_bounds__(THREADS, 1)
f64_product_kernel(const Args a) {
  static_assert(KS == 1 || BN == 64, "split tiles are 64 wide");
  constexpr int STG = stages_of(BN), SBYTES = stage_bytes(BN);
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STG];
  __shared__ __align__(8) uint64_t empty_bar[STG];
  __shared__ __align__(8) uint64_t accf_bar[NS];
  __shared__ __align__(8) uint64_t acce_bar[NS];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ __align__(8) uint64_t xfull_bar[8];     // split tiles, per epilogue warp: the others' sums are here,
  __shared__ __align__(8) uint64_t xempty_bar[8];    // and the others have taken this CTA's
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;
  __shared__ volatile int over_s;        // st->done as thread 0 read it

  DevState* st = a.st;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int ld = a.ld, cols = (ld + BN - 1) / BN;
  const int rank = KS > 1 ? (int)cluster_ctarank() : 0;
  const int unit = blockIdx.x / KS, units = gridDim.x / KS;       // clusters
  const int kb0 = (ld / KB) * rank / KS, nkb = (ld / KB) * (rank + 1) / KS - kb0;   // this CTA's k-blocks
  const uint64_t wait_ns = a.wait_ns;
  if (threadIdx.x == 0) {
    int over = st->done;
    if (KS > 1 && a.hook >= HOOK_OTHERS_OVER) over |= (a.hook == HOOK_FIRST_OVER) == (rank == 0) ? 1 : 0;
    over_s = over;
    if (blockIdx.x == 0 && !over && a.op != OP_MCW_SQ) st->wrote = (st->k + (a.op == OP_SP2 ? 1 : 0)) & 1;
    for (int w = 0; w < 8; ++w) { mbar_init(&xfull_bar[w], KS > 1 ? KS - 1 : 1); mbar_init(&xempty_bar[w], KS > 1 ? KS - 1 : 1); }
    for (int s = 0; s < STG; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int b = 0; b < NS; ++b) { mbar_init(&accf_bar[b], 1); mbar_init(&acce_bar[b], 8); }
    mbar_init(&drain_bar, 1);
    abort_s = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, NS * BN);
  tc_fence_before();
  if (KS > 1) cluster_sync();            // the barriers of every CTA are initialised
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;

  // A CTA that finds the run over stays until the cluster's last barrier all the same: a wait that gives up elsewhere
  // sets st->done during the launch, and the others of its cluster may have found it clear and write here.  (They then
  // wait for sums that do not come, and give up in turn.)  Reading the first CTA's flag through distributed shared
  // memory instead would spare them that, but made the split products a third slower (N = 1500, McW-ACC: 5.31 -> 7.21 ms).
  if (over_s) {
  } else if (warp < 4) {
    if (warp == 0) {
      if (elect_one()) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        const int64_t kstride = (int64_t)padded_rows(ld) / 8 * GRPB;
        int armed[STG];
        uint32_t armed_par[STG];
        for (int s = 0; s < STG; ++s) { armed[s] = 0; armed_par[s] = 0; }
        for (int t = unit; t < a.tiles && ok; t += units) {
          int I, J;
          locate(t, cols, BM / BN, I, J);
          for (int kb = 0; kb < nkb; ++kb) {
            if (abort_s || !mbar_wait(&empty_bar[stage], phase ^ 1, globaltimer_ns() + wait_ns)) { ok = false; break; }
            if (a.hook == HOOK_SKIP_COPY && blockIdx.x == 0 && t == unit && kb == 0) {
              if (++stage == STG) { stage = 0; phase ^= 1; }
              continue;
            }
            uint8_t* sA = smem + stage * SBYTES;
            mbar_arrive_expect_tx(&full_bar[stage], SBYTES);
            bulk_load(sA, a.digA + (kb0 + kb) * kstride + (int64_t)I * A_BYTES, A_BYTES, &full_bar[stage]);
            bulk_load(sA + A_BYTES, a.digB + (kb0 + kb) * kstride + (int64_t)J * b_bytes(BN), b_bytes(BN), &full_bar[stage]);
            armed[stage] = 1;
            armed_par[stage] = phase;
            if (++stage == STG) { stage = 0; phase ^= 1; }
          }
        }
        if (!ok) give_up(st, &abort_s);
        for (int s = 0; s < STG; ++s)    // wait (bounded) until every copy issued here has landed
          if (armed[s]) mbar_wait(&full_bar[s], armed_par[s], globaltimer_ns() + wait_ns);
      }
    } else if (warp == 1) {
      if (elect_one()) {
        constexpr uint32_t idesc = idesc_f16_f32(BM, BN);
        int stage = 0;
        uint32_t phase = 0, phases = 0;  // phases: bit s, the parity of accumulator s
        bool ok = true;
        for (int t = unit; t < a.tiles && ok; t += units) {
          for (int kb = 0; kb < nkb && ok; ++kb) {
            if (abort_s || !mbar_wait(&full_bar[stage], phase, globaltimer_ns() + wait_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sA = smem_u32(smem + stage * SBYTES);
            const uint32_t sB = sA + A_BYTES;
            #pragma unroll
            for (int s = 0; s < NS; ++s) {
              const uint32_t dt = tmem_base + (uint32_t)(s * BN);
              uint32_t accumulate = 1;
              if (kb == 0 || closes(kb - 1, s)) {
                if (abort_s || !mbar_wait(&acce_bar[s], ((phases >> s) & 1u) ^ 1u, globaltimer_ns() + wait_ns)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                accumulate = 0;
              }
              #pragma unroll
              for (int i = first_pair(s); i < first_pair(s) + pairs(s); ++i) {
                #pragma unroll
                for (int kk = 0; kk < KB / 16; ++kk) {
                  mma_bf16(dt, smem_desc_sw64_stride(sA + i * DIGB + kk * 32, GRPB),
                           smem_desc_sw64_stride(sB + (s - i) * DIGB + kk * 32, GRPB), idesc, accumulate);
                  accumulate = 1;
                }
              }
              if (closes(kb, s) || kb + 1 == nkb) {
                mma_commit(&accf_bar[s]);
                phases ^= 1u << s;
              }
            }
            if (!ok) break;
            mma_commit(&empty_bar[stage]);
            if (++stage == STG) { stage = 0; phase ^= 1; }
          }
        }
        if (!ok) give_up(st, &abort_s);
        mma_commit(&drain_bar);
        mbar_wait(&drain_bar, 0, globaltimer_ns() + wait_ns);
      }
    }
  } else {
    const int ew = warp - 4;
    const int q = warp & 3;              // tensor-memory lanes 32 q .. 32 q + 31
    const int hc = ew >> 2;              // columns hc BN / 2 .. of the tile
    constexpr int G = BN / 2, C = G / KS;       // columns a warp sums, and finishes
    uint32_t xphase = 0;
    const Poly P = poly_of(a);
    const int N = st->N, T64 = ld / 64;
    uint32_t phases = 0;
    bool ok = true;
    const uint32_t trow = tmem_base + (uint32_t)(hc * G) + ((uint32_t)(32 * q) << 16);
    for (int t = unit; t < a.tiles && ok; t += units) {
      int I, J;
      locate(t, cols, BM / BN, I, J);
      long long T[G];
      #pragma unroll
      for (int j = 0; j < G; ++j) T[j] = 0;
      uint32_t held = 0;                 // accumulators 6 and 7 stay with this warp until its tile is finished
      for (int kb = 0; ok && kb < nkb; ++kb) {
        const bool last = kb == nkb - 1;
        constexpr uint64_t c0 = closing(0), c1 = closing(1);
        uint32_t todo = last ? 255u : (uint32_t)(((kb & 8) ? c1 : c0) >> (8 * (kb & 7))) & 255u;
        while (todo) {
          const int s = __ffs(todo) - 1;
          todo &= todo - 1u;
          int got = 0;
          if (lane == 0) got = !abort_s && mbar_wait(&accf_bar[s], (phases >> s) & 1u, globaltimer_ns() + wait_ns);
          got = __shfl_sync(0xffffffffu, got, 0);
          if (!got) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint32_t raw[G];
          tmem_ld(trow + (uint32_t)(s * BN), raw);
          tmem_wait_ld();
          phases ^= 1u << s;
          if (last && s >= 6) {
            held |= 1u << s;
          } else {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce_bar[s]);
          }
          add_digit_sums(s, raw, T);
        }
      }
      // the sums go to the columns of accumulators 6 (low words) and 7 (high words), from which the rest takes
      // them four at a time in loops
      const uint32_t lo = trow + 6 * BN, hi = trow + 7 * BN;
      if (nkb > 0 && ok) {
        uint32_t wlo[G], whi[G];
        #pragma unroll
        for (int j = 0; j < G; ++j) {
          wlo[j] = (uint32_t)(unsigned long long)T[j];
          whi[j] = (uint32_t)((unsigned long long)T[j] >> 32);
        }
        #pragma unroll
        for (int j = 0; j < G; j += 16) {
          tmem_st16(lo + j, wlo + j);
          tmem_st16(hi + j, whi + j);
        }
        tmem_wait_st();
      }
      if constexpr (KS > 1) {
        // to every other CTA its columns, from every other CTA this one's; the slot of sender p is p, less
        // one past the receiver
        const uint32_t slots = smem_u32(smem + STG * SBYTES);
        const uint64_t until = globaltimer_ns() + wait_ns;
        // every lane waits, since the wait orders the accesses of its own lane only (as lane 0's wait, a shuffle and a
        // __syncwarp, the runs at N = 400 and 1500 took 3 % longer)
        int go = __all_sync(0xffffffffu, ok && !abort_s && mbar_wait_cluster(&xempty_bar[ew], xphase ^ 1, until));
        if (go) {
          #pragma unroll 1
          for (int j = 0; j < G; j += 4) {
            const int o = j / C;
            if (o == rank) continue;
            long long t[4] = {0, 0, 0, 0};
            if (nkb > 0) load_sums(lo + j, hi + j, t);
            const uint32_t dst = mapa_shared(slots, o) +
                                 (uint32_t)((((rank < o ? rank : rank - 1) * 8 + ew) * C + j % C) * 256 + lane * 8);
            #pragma unroll
            for (int d = 0; d < 4; ++d) st_cluster_u64(dst + d * 256, (unsigned long long)t[d]);
          }
          __syncwarp();
          if (lane == 0) {
            #pragma unroll 1
            for (int o = 0; o < KS; ++o)
              if (o != rank) mbar_arrive_cluster(mapa_shared(smem_u32(&xfull_bar[ew]), o));
          }
          go = __all_sync(0xffffffffu, mbar_wait_cluster(&xfull_bar[ew], xphase, until));
        }
        if (!go) ok = false;
      }
      // after the tile: the others may overwrite the exchanged sums, the products the held accumulators
      auto release = [&]() {
        if (KS > 1) {
          __syncwarp();
          if (lane == 0) {
            #pragma unroll 1
            for (int o = 0; o < KS; ++o)
              if (o != rank) mbar_arrive_cluster(mapa_shared(smem_u32(&xempty_bar[ew]), o));
          }
          xphase ^= 1;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (held & 64u) mbar_arrive(&acce_bar[6]);
          if (held & 128u) mbar_arrive(&acce_bar[7]);
        }
      };
      if (!ok) {
        if (lane == 0) give_up(st, &abort_s);
        break;
      }
      // epilogue: this warp's 32 rows, C columns; only blocks on or above the diagonal
      const int r0 = I * BM + 32 * q, r = r0 + lane;
      const int c0 = J * BN + hc * G + rank * C;
      if (r0 >= ld || c0 >= ld || c0 + C <= r0) {
        release();
        continue;
      }
      const int ei = a.ea[r];
      const bool off = c0 >= r0 + 32;    // wholly above the diagonal
      double v2 = 0.0, trc = 0.0;
      double xl[4];                      // the old values, loaded a step ahead
      load4(P.in + (int64_t)r * ld + c0, xl);
      #pragma unroll 1
      for (int j0 = 0; j0 < C; j0 += 4) {
        double x[4] = {xl[0], xl[1], xl[2], xl[3]}, xn[4];
        if (j0 + 4 < C) load4(P.in + (int64_t)r * ld + c0 + j0 + 4, xl);
        long long F[4] = {0, 0, 0, 0};
        if (nkb > 0) load_sums(lo + rank * C + j0, hi + rank * C + j0, F);
        if constexpr (KS > 1) {
          const unsigned long long* src = reinterpret_cast<const unsigned long long*>(smem + STG * SBYTES);
          #pragma unroll
          for (int p = 0; p < KS - 1; ++p)
            #pragma unroll
            for (int j = 0; j < 4; ++j) F[j] += (long long)src[((p * 8 + ew) * C + j0 + j) * 32 + lane];
        }
        #pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = c0 + j0 + j;
          const double s = scaled_sum(F[j], ei, a.eb[c]);
          const double d = x[j] - s;
          if (off || c > r) v2 = fma(d, d, v2);
          else if (c == r) v2 = fma(0.5 * d, d, v2);
          xn[j] = P.gen ? fma(P.ca, s, fma(P.cb, x[j], (c == r && r < N) ? P.cc : 0.0)) : (P.pk ? s : (2.0 * x[j] - s));
          if (c == r) trc = xn[j];
          if (off || c > r) P.out[(int64_t)c * ld + r] = xn[j];
        }
        if (off) {
          store4(P.out + (int64_t)r * ld + c0 + j0, xn);
        } else {
          #pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c0 + j0 + j >= r) P.out[(int64_t)r * ld + c0 + j0 + j] = xn[j];
        }
      }
      release();
      v2 *= 2.0;                         // each element above the diagonal stands for two
      #pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v2 += __shfl_xor_sync(0xffffffffu, v2, o);
        trc += __shfl_xor_sync(0xffffffffu, trc, o);
      }
      if (lane == 0) {
        // record of these 32 rows and C columns within their 64 x 64 tile
        constexpr int half = 64 / C;     // records of 32 rows
        double* dst = a.part + 2 * (2 * half * upper_index(r0 / 64, c0 / 64, T64) + half * ((r0 >> 5) & 1) + (c0 & 63) / C);
        dst[0] = v2;
        dst[1] = trc;
      }
    }
  }

  if (KS > 1) {                          // the others' accesses to this CTA's shared memory are over
    __syncwarp();
    cluster_sync();
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, NS * BN);
  }
}

// ---- host side ---------------------------------------------------------------------------------
static const void* kernel_of(int bn, int ks) {
  if (bn == 32) return (const void*)f64_product_kernel<32, 1>;
  return ks == 8   ? (const void*)f64_product_kernel<64, 8>
         : ks == 4 ? (const void*)f64_product_kernel<64, 4>
         : ks == 2 ? (const void*)f64_product_kernel<64, 2>
                   : (const void*)f64_product_kernel<64, 1>;
}

// Tiles that run at once: SMs, or the clusters of ks that the GPU holds.  Sets the kernels' attributes first; 0 if
// that fails.
static int find_slots(int dev, int bn, int ks) {
  int sms = 0;
  if (cudaFuncSetAttribute(kernel_of(bn, ks), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(bn, ks)) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (ks == 1) return sms;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ks * (sms / ks));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem_bytes(bn, ks);
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel_of(bn, ks), &cfg) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

static int slots_of(int bn, int ks) {
  static PerDevice slots[2][4];
  return slots[bn == 64][ks == 8 ? 3 : ks / 2].get([&](int dev) { return find_slots(dev, bn, ks); });
}

static void set_tiles(Plan& P, int ld, int bn, int ks) {
  P.ld = ld;
  P.bn = bn;
  P.ks = ks;
  P.recs = 2 * 64 / (bn / 2 / ks);
}

// The shape with the least time in this model: rounds of tiles, each its k-blocks (68 products of 48 clocks, 44 at
// width 32: reading A bounds them) and about 12 k clocks for filling the pipe, the last drains and the epilogue,
// less with fewer columns to finish.  One iteration of a run, unsplit and split: N = 400 54 -> 35 us (16 tiles, 152 SMs),
// N = 700 76 -> 42, N = 1500 (156 tiles) 260 -> 205; N = 2048 stays unsplit.
void choose_tiles(Plan& P, int ld) {
  P.ld = ld;
  double best = 1e300;
  for (int i = 0; i < 5; ++i) {
    const int bn = i == 4 ? 32 : 64, ks = i == 4 ? 1 : 1 << i;
    const int slots = slots_of(bn, ks);
    if (slots < 1) continue;
    const int n = tiles_of(ld, bn), kb = (ld / KB + ks - 1) / ks;
    const double tile = kb * 2.0 * 34.0 * (bn == 64 ? 48.0 : 44.0) + 6000.0 + (bn == 64 ? 8000.0 / ks : 4000.0) +
                        (ks > 1 ? 2000.0 : 0.0);
    const double t = (double)((n + slots - 1) / slots) * tile;
    if (t < best) {
      best = t;
      set_tiles(P, ld, bn, ks);
    }
  }
}

cudaError_t Sink::put(const void* func, dim3 grid, dim3 block, size_t smem, void** args) {
  if (!g) return cudaLaunchKernel(func, grid, block, args, smem, s);
  cudaKernelNodeParams kp = {};
  kp.func = const_cast<void*>(func);
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.sharedMemBytes = (unsigned)smem;
  kp.kernelParams = args;
  cudaGraphNode_t node;
  const cudaError_t e = cudaGraphAddKernelNode(&node, g, last ? &last : nullptr, last ? 1 : 0, &kp);
  if (e == cudaSuccess) last = node;
  return e;
}

cudaError_t emit_digits(Sink& sink, const DevState* st, const double* buf0, const double* buf1, const double* S,
                        const Plan& P, int N) {
  const Digits& d = S ? P.S : P.X;
  int ld = P.ld;
  __half* dig = d.dig;
  int32_t* exps = d.exp;
  void* args[] = {&st, &buf0, &buf1, &S, &ld, &N, &dig, &exps};
  return sink.put((const void*)digits_kernel, dim3((N + 7) / 8), dim3(DT), 0, args);
}

cudaError_t emit_product(Sink& sink, DevState* st, double* buf0, double* buf1, double* S, double* part,
                         const Plan& P, Op op, int hook, int wait_ms) {
  const Digits& A = op == OP_MCW_PROD ? P.S : P.X;
  Args a;
  std::memset(&a, 0, sizeof(a));
  a.st = st;
  a.buf0 = buf0;
  a.buf1 = buf1;
  a.S = S;
  a.part = part;
  a.digA = reinterpret_cast<const uint8_t*>(A.dig);
  a.digB = reinterpret_cast<const uint8_t*>(P.X.dig);
  a.ea = A.exp;
  a.eb = P.X.exp;
  a.ld = P.ld;
  a.tiles = tiles_of(P.ld, P.bn);
  a.op = op;
  a.hook = hook;
  a.wait_ns = wait_ms > 0 ? (uint64_t)wait_ms * 1000000ull : kWaitNs;
  const int slots = slots_of(P.bn, P.ks);
  if (slots < 1) return cudaErrorNotSupported;
  void* args[] = {&a};
  const int units = a.tiles < slots ? a.tiles : slots;
  return sink.put(kernel_of(P.bn, P.ks), dim3(units * P.ks), dim3(THREADS), smem_bytes(P.bn, P.ks), args);
}

}  // namespace f64tc
}  // namespace sp2

extern "C" int32_t sp2_test_f64_product(const double* X_dev, int64_t N, int32_t bn, int32_t ks, int32_t hook,
                                        int32_t wait_ms, double* out_dev, int32_t* exp_dev, void* stream) {
  using namespace sp2::f64tc;
  const bool shape = (bn == 32 && ks == 1) || (bn == 64 && (ks == 1 || ks == 2 || ks == 4 || ks == 8));
  if (!X_dev || !out_dev || N < 1 || N > 8192 || !shape || hook < 0 || hook > 3 || wait_ms < 0 || wait_ms > 2000)
    return SP2_ERR_INVALID_ARG;
  const cudaStream_t s = (cudaStream_t)stream;
  const int ld = (int)(N + 63) / 64 * 64, T = ld / 64;
  const size_t bytes = sizeof(double) * (size_t)ld * ld, row = sizeof(double) * (size_t)N;
  const size_t pbytes = part_bytes(kMinN, T, MAX_RECS);
  Plan P;
  set_tiles(P, ld, bn, ks);
  sp2::DevState h;
  std::memset(&h, 0, sizeof(h));
  h.N = (int)N;
  h.ld = ld;
  h.tr[0] = 1.0;                         // above nocc = 0: X_1 = X_0^2
  sp2::DevState* st = nullptr;
  double *buf = nullptr, *part = nullptr;
  Sink sink;
  sink.s = s;
  bool ok = cudaMalloc(&st, sizeof(h)) == cudaSuccess && cudaMalloc(&buf, 2 * bytes) == cudaSuccess &&
            cudaMalloc(&part, pbytes) == cudaSuccess && cudaMalloc(&P.X.dig, digit_bytes(ld)) == cudaSuccess &&
            cudaMalloc(&P.X.exp, exp_bytes(ld)) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(st, &h, sizeof(h), cudaMemcpyHostToDevice, s) == cudaSuccess &&
       cudaMemsetAsync(buf, 0, 2 * bytes, s) == cudaSuccess &&
       cudaMemsetAsync(P.X.dig, 0, digit_bytes(ld), s) == cudaSuccess &&
       cudaMemsetAsync(P.X.exp, 0, exp_bytes(ld), s) == cudaSuccess &&
       cudaMemcpy2DAsync(buf, sizeof(double) * ld, X_dev, row, row, N, cudaMemcpyDeviceToDevice, s) == cudaSuccess;
  double* buf1 = buf + (size_t)ld * ld;
  ok = ok && emit_digits(sink, st, buf, buf1, nullptr, P, (int)N) == cudaSuccess &&
       emit_product(sink, st, buf, buf1, nullptr, part, P, OP_SP2, hook, wait_ms) == cudaSuccess &&
       cudaMemcpy2DAsync(out_dev, row, buf1, sizeof(double) * ld, row, N, cudaMemcpyDeviceToDevice, s) == cudaSuccess &&
       (!exp_dev || cudaMemcpyAsync(exp_dev, P.X.exp, sizeof(int32_t) * N, cudaMemcpyDeviceToDevice, s) == cudaSuccess) &&
       cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, s) == cudaSuccess;
  ok = cudaStreamSynchronize(s) == cudaSuccess && ok;
  cudaFree(st);
  cudaFree(buf);
  cudaFree(part);
  cudaFree(P.X.dig);
  cudaFree(P.X.exp);
  if (!ok) {
    (void)cudaGetLastError();
    return SP2_ERR_CUDA;
  }
  return h.status;
}
