// Spectral-norm stop of the FP64 path (§2: the stop is defined on e_i = ||X_i - X_i^2||_2;
// the Frobenius v_i and the mixed norm m_i are its upper bounds).
//
// After square k the buffers hold X_{k-1} and the stored product Y = a X_{k-1}^2 + b X_{k-1} + c I
// of this step: X_k itself (SP2: (a, b, c) = (1, 0, 0) or (-1, 2, 0); SP2-ACC: the scheduled
// coefficients) or the McWeeny step's shifted square S_s (alpha^2, 2 alpha c, c^2).  So
//     A = X_{k-1} - X_{k-1}^2 = ((a + b) X_{k-1} - Y + c I) / a
// is available without forming X^2, and e_{k-1} = ||A||_2 = max |lambda(A)| is estimated by
// kLzSteps steps of the symmetric Lanczos recurrence (three-term, no reorthogonalisation: lost
// orthogonality only repeats converged extreme Ritz values) from a fixed start vector.  The
// extreme eigenvalues of the tridiagonal matrix come from multisection with Sturm counts (512
// points a side, three rounds, in FP32: the tridiagonal of the scaled A is O(1) and the estimate
// only needs a few digits).  The Ritz values are inside the spectrum, so the estimate is a lower
// bound of e that approaches it from below; the stop test only needs its logarithm.
//
// Per estimate: start (1 CTA: coefficients, start vector, a power-of-two scale 2^-s with 2^s near
// v_{k-1} from the square's Frobenius partials), form (A 2^-s rounded to FP32 once: the ld x ld
// FP32 matrix, half the bytes of one FP64 iterate, is then read kLzSteps times, from L2 where it
// fits), kLzSteps x step, eig (1 CTA).  Step j first finishes step j - 1: every CTA sums the partials of
// alpha_{j-1}, forms r = w - alpha q_{j-1} - beta q_{j-2}, ||r|| and q_j = r / ||r|| for all N entries by itself
// (FP64; 2 N clocks of the SM's FP64 units), then multiplies its rows: w = A q_j, one warp per row, FP32 products
// summed in FP32 per lane and FP64 across lanes.  The steps thus have one launch between them and no CTA that
// the others wait for; up to N = kLzClusterN one cluster does them all in one launch (lz_cluster_kernel).  With the
// last CTA to finish doing the update alone, a step took 15 us at N = 1001, most of it in that CTA's serial FP64
// sums.  The FP32 rounding of A and of the products perturbs A by about 1e-7 of its norm, far below the Lanczos
// truncation error.
#include <math.h>

#include "sp2_common.cuh"
#include "sp2_f64_tc.cuh"
#include "sp2_kernels.h"
#include "sp2_tc.cuh"
#include "tc_ptx.cuh"

namespace sp2 {
namespace {

constexpr int kLzSteps = 32;          // Lanczos steps per estimate
constexpr int kLzThreads = 1024;      // start: one CTA
constexpr int kLzMvBlocks = 152;      // step grid cap (one CTA per SM) = number of partial sums
constexpr int kLzMvThreads = 1024;    // threads of a step: 512 while the grid cap is not reached, else 1024
constexpr int kLzSmemN = 16384;       // q_j in shared memory up to this size
constexpr int kLzCtas = 16;           // CTAs of the cluster that does all steps
constexpr int kLzClThreads = 512;
// Largest N it takes.  Time of one FP64 purification with 32 step launches and with the cluster (both with the
// spectral stop): N = 130 13.5 -> 7.7 ms, 400 16.3 -> 10.0, 700 18.8 -> 13.0, 1001 21.7 -> 17.9, 1300 26.0 -> 25.5,
// 1600 33.1 -> 33.4, 2000 39.1 -> 44.0: past the line 16 SMs read the matrix more slowly than 152.
constexpr int kLzClusterN = 1280;
constexpr int kLzClSmem = 222 * 1024; // dynamic shared memory it may have
constexpr int kSturmThreads = 1024;   // 512 points per side
constexpr int kSturmRounds = 3;       // 513^3 > 2^27: below FP32 resolution of the interval

struct LzScratch {
  double scale;               // 2^-s applied before rounding A to FP32
  int32_t m;                  // finished steps (alpha[0 .. m-1])
  int32_t live;               // 0 once the Krylov space is invariant (beta = 0) or not finite
  double alpha[kLzSteps];     // diagonal of the tridiagonal matrix
  double beta[kLzSteps + 1];  // beta[j] couples q_{j-1} and q_j; beta[0] = 0
  double part[2][kLzMvBlocks];  // per-CTA partials of q_j . A q_j, by the parity of j
};
// followed by three vectors q (q_j in j % 3) and two w (w_j in j % 2), FP64, ld each, q_j in FP32 (ld; used for
// N > kLzSmemN) and A 2^-s in FP32 (ld x ld)

constexpr size_t kVecOff = (sizeof(LzScratch) + 255) / 256 * 256;

__device__ __forceinline__ double* lz_vec(LzScratch* lz, int ld, int which) {
  return reinterpret_cast<double*>(reinterpret_cast<char*>(lz) + kVecOff) + (size_t)which * ld;
}
__device__ __forceinline__ float* lz_q32(LzScratch* lz, int ld) {
  return reinterpret_cast<float*>(lz_vec(lz, ld, 5));
}
__device__ __forceinline__ float* lz_a32(LzScratch* lz, int ld) { return lz_q32(lz, ld) + ld; }

// Start vector entry i: SplitMix64 (Steele, Lea, Flood 2014) of the index, mapped to [-1, 1).
__device__ __forceinline__ double start_entry(int i) {
  unsigned long long z = (unsigned long long)(i + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * 0x1p-52 - 1.0;
}

// X_{k-1}, the stored product Y and its coefficients (a, b, c) for the square just written.
__device__ __forceinline__ void lz_operands(const DevState* st, const double* buf0, const double* buf1,
                                            const double* S, const double*& Xa, const double*& Y, double& a,
                                            double& b, double& c) {
  const int k = st->k;
  Xa = (k & 1) ? buf1 : buf0;
  if (st->mcw) {                                 // S_s = (alpha X + c0 I)^2, c0 = (1 - alpha) / 2
    const double al = st->alpha[k + 1], c0 = 0.5 * (1.0 - al);
    a = al * al; b = 2.0 * al * c0; c = c0 * c0;
    Y = S;
    return;
  }
  if (st->acc) {
    acc_step(st, k + 1, a, b, c);
  } else {
    const int pk = st->tr[k] > (double)st->nocc ? 1 : 0;
    a = pk ? 1.0 : -1.0; b = pk ? 0.0 : 2.0; c = 0.0;
  }
  Y = (k & 1) ? buf0 : buf1;
}

// n x n operator stored with leading dimension ld; the square's partial records (v^2 first, `rec`
// doubles each), ntiles of them, set the scale.
__global__ void __launch_bounds__(kLzThreads)
lz_start_kernel(const DevState* st, const double* __restrict__ part, int ntiles, int rec, LzScratch* lz, int N, int ld) {
  __shared__ double sm[96];
  if (st->done) return;
  double v2 = 0.0, ss = 0.0, none = 0.0;         // v_{k-1}^2 from the square's partials
  for (int t = threadIdx.x; t < ntiles; t += kLzThreads) v2 += part[rec * (int64_t)t];
  for (int i = threadIdx.x; i < N; i += kLzThreads) {
    const double u = start_entry(i);
    ss = fma(u, u, ss);
  }
  block_sum3<kLzThreads>(v2, ss, none, kLzThreads, sm);
  if (threadIdx.x == 0) {
    const double v = sqrt(v2);
    int e = (v > 0.0 && isfinite(v)) ? ilogb(v) : 0;
    e = e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
    lz->scale = ldexp(1.0, -e);
    lz->m = 0;
    lz->live = 1;
    lz->beta[0] = 0.0;
  }
  double* q = lz_vec(lz, ld, 0);
  if (threadIdx.x == 0) sm[0] = 1.0 / sqrt(ss);
  __syncthreads();
  const double inv = sm[0];
  for (int i = threadIdx.x; i < N; i += kLzThreads) q[i] = start_entry(i) * inv;
}

// A 2^-s = ((a + b) X_{k-1} - Y + c I) (2^-s / a), rounded to FP32, over the whole ld x ld
// buffer (the zero border stays zero; the identity term on the N true diagonal entries).
__global__ void lz_form_kernel(const DevState* st, const double* buf0, const double* buf1, const double* S,
                               LzScratch* lz) {
  if (st->done) return;
  const int N = st->N, ld = st->ld;
  const double* Xa;
  const double* Y;
  double a, b, c;
  lz_operands(st, buf0, buf1, S, Xa, Y, a, b, c);
  const double ab = a + b, f = lz->scale / a;
  const double2* __restrict__ X2 = reinterpret_cast<const double2*>(Xa);
  const double2* __restrict__ Y2 = reinterpret_cast<const double2*>(Y);
  float2* __restrict__ A2 = reinterpret_cast<float2*>(lz_a32(lz, ld));
  const int h = ld / 2;
  const int64_t total = (int64_t)ld * h;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / h), c2 = 2 * (int)(e % h);
    const double2 x = X2[e], y = Y2[e];
    double d0 = fma(ab, x.x, -y.x), d1 = fma(ab, x.y, -y.y);
    if (r < N && r == c2) d0 += c;
    if (r < N && r == c2 + 1) d1 += c;
    A2[e] = make_float2((float)(d0 * f), (float)(d1 * f));
  }
}

// The same operator on the tensor-core path (one problem): X_{k-1} and X_k are slots of the
// instance's piece arena, each element the exact FP32 value of its pieces, so
//     A 2^-s = ((a + b) X_{k-1} - X_k + c I) (2^-s / a), rounded to FP32,
// with the step's coefficients (SP2: (1, 0, 0) after X^2, (-1, 2, 0) after 2X - X^2).
__global__ void lz_form_tc_kernel(const DevState* st, const tc::Instance* inst, LzScratch* lz) {
  if (st->done) return;
  const tc::Instance& In = inst[0];
  const int N = st->N, ld = In.ld, k = st->k;
  double a, b, c;
  if (st->acc) {
    acc_step(st, k + 1, a, b, c);
  } else {
    const int pk = st->tr[k] > (double)st->nocc ? 1 : 0;
    a = pk ? 1.0 : -1.0; b = pk ? 0.0 : 2.0; c = 0.0;
  }
  const double ab = a + b, f = lz->scale / a;
  const int64_t plane = (int64_t)ld * ld;
  const __nv_bfloat16* xs = In.arena + (int64_t)tc::xslot(In.lowmem, In.hist0, k) * In.slot_elems;
  const __nv_bfloat16* ys = In.arena + (int64_t)tc::xslot(In.lowmem, In.hist0, k + 1) * In.slot_elems;
  float* A = lz_a32(lz, ld);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < plane; e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / ld), col = (int)(e % ld);
    const double x = (double)tc::piece_load(In.fmt, xs, plane, e);
    const double y = (double)tc::piece_load(In.fmt, ys, plane, e);
    double d = fma(ab, x, -y);
    if (r < N && r == col) d += c;
    A[e] = (float)(d * f);
  }
}

// Sum over the CTA (fixed order), the result in every thread; sm: 33 doubles.
__device__ __forceinline__ double cta_sum(double x, double* sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if (lane == 0) sm[warp] = x;
  __syncthreads();
  if (warp == 0) {
    double t = lane < nw ? sm[lane] : 0.0;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) sm[32] = t;
  }
  __syncthreads();
  return sm[32];
}

// Step j of the recurrence (see the header): q_j for all entries, then w_j and the CTA's share of alpha_j for its
// rows.  Vectors alternate, so no CTA writes what another may still read.
__global__ void __launch_bounds__(kLzMvThreads)
lz_step_kernel(const DevState* st, LzScratch* lz, int j, int N, int ld) {
  extern __shared__ __align__(16) float lz_smem[];
  __shared__ double sm[2][33];
  __shared__ double s_alpha, s_b, s_ib;
  if (st->done || !lz->live) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  // the warp's first row of A (up to 1024 columns of it), which does not wait for q_j
  constexpr int PRE = 8;
  const float4* __restrict__ A = reinterpret_cast<const float4*>(lz_a32(lz, ld));
  const int h = ld / 4, row0 = blockIdx.x * nw + warp;
  float4 pre[PRE];
  if (row0 < N) {
    #pragma unroll
    for (int n = 0; n < PRE; ++n)
      if (lane + 32 * n < h) pre[n] = A[(int64_t)row0 * h + lane + 32 * n];
  }
  float* q32 = N <= kLzSmemN ? lz_smem : lz_q32(lz, ld);   // past it every CTA writes the same values
  double* q = lz_vec(lz, ld, j % 3);
  const int per = nw;                                       // rows of a CTA per sweep: one per warp
  auto mine = [&](int i) { return (i / per) % (int)gridDim.x == (int)blockIdx.x; };
  if (j == 0) {
    for (int i = threadIdx.x; i < ld; i += blockDim.x) q32[i] = i < N ? (float)q[i] : 0.f;
  } else {
    const double* q1 = lz_vec(lz, ld, (j + 2) % 3);         // q_{j-1}
    const double* q2 = lz_vec(lz, ld, (j + 1) % 3);         // q_{j-2}
    const double* w1 = lz_vec(lz, ld, 3 + ((j - 1) & 1));
    if (warp == 0) {
      double a = 0.0;
      for (int t = lane; t < (int)gridDim.x; t += 32) a += lz->part[(j - 1) & 1][t];
      #pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) s_alpha = a;
    }
    __syncthreads();
    const double a = s_alpha, bj = lz->beta[j - 1];
    double ss = 0.0;
    auto residual = [&](int i) { return w1[i] - a * q1[i] - (j > 1 ? bj * q2[i] : 0.0); };
    double keep[4];                                         // this thread's first entries, kept for the second pass
    #pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int i = threadIdx.x + n * blockDim.x;
      keep[n] = i < N ? residual(i) : 0.0;
      ss = fma(keep[n], keep[n], ss);
    }
    for (int i = threadIdx.x + 4 * blockDim.x; i < N; i += blockDim.x) {
      const double r = residual(i);
      ss = fma(r, r, ss);
    }
    ss = cta_sum(ss, sm[0]);
    if (threadIdx.x == 0) {                                 // one thread: FP64 operations run at 2 a clock and SM
      s_b = sqrt(ss);
      s_ib = 1.0 / s_b;
    }
    __syncthreads();
    const double b = s_b;
    const bool finite = isfinite(a) && isfinite(b);
    const bool more = finite && b > 1e-300;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      lz->alpha[j - 1] = finite ? a : __longlong_as_double(0x7ff8000000000000ll);
      lz->m = j;
      lz->beta[j] = b;
      if (!more) lz->live = 0;
    }
    if (!more) return;
    const double ib = s_ib;
    auto put = [&](int i, double u) {
      q32[i] = (float)u;
      if (i < N && mine(i)) q[i] = u;
    };
    #pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int i = threadIdx.x + n * blockDim.x;
      if (i < ld) put(i, keep[n] * ib);
    }
    for (int i = threadIdx.x + 4 * blockDim.x; i < ld; i += blockDim.x) put(i, i < N ? residual(i) * ib : 0.0);
  }
  __syncthreads();
  const float4* q4 = reinterpret_cast<const float4*>(q32);
  double* w = lz_vec(lz, ld, 3 + (j & 1));
  double pa = 0.0;
  auto dot4 = [](const float4& x, const float4& v, float s) {
    s = fmaf(x.x, v.x, s); s = fmaf(x.y, v.y, s); s = fmaf(x.z, v.z, s);
    return fmaf(x.w, v.w, s);
  };
  for (int r = row0; r < N; r += gridDim.x * per) {
    const float4* ar = A + (int64_t)r * h;
    float s0 = 0.f, s1 = 0.f;
    int i = lane;
    if (r == row0) {
      #pragma unroll
      for (int n = 0; n < PRE; ++n) {
        const int c = lane + 32 * n;
        if (c < h) (n & 1 ? s1 : s0) = dot4(pre[n], q4[c], n & 1 ? s1 : s0);
      }
      i += 32 * PRE;
    }
    for (; i + 32 < h; i += 64) {
      const float4 x0 = ar[i], v0 = q4[i], x1 = ar[i + 32], v1 = q4[i + 32];
      s0 = dot4(x0, v0, s0);
      s1 = dot4(x1, v1, s1);
    }
    if (i < h) s0 = dot4(ar[i], q4[i], s0);
    double s = (double)s0 + (double)s1;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      w[r] = s;
      pa = fma(q[r], s, pa);
    }
  }
  pa = cta_sum(pa, sm[1]);
  if (threadIdx.x == 0) lz->part[j & 1][blockIdx.x] = pa;
}

// All steps in one launch, for N <= kLzClusterN: one cluster of kLzCtas CTAs, each with the entries and rows
// c S .. c S + S - 1 (S = ceil(N / kLzCtas)), one entry of q_j and q_{j-1} in a register of its first S threads.
// A step has two exchanges through distributed shared memory, each closed by a cluster barrier: the warps'
// partials of alpha_j go to every CTA; then those of ||r||^2 and the entries of r, from which every CTA rounds
// its own FP32 copy of q_{j+1}.  Every CTA adds the same partials in the same order, so all take the same
// decisions.  A CTA keeps the first R of its rows of A in shared memory and reads the others from L2 in each step;
// a warp multiplies four rows at a time, so that the loads of q and the FP64 sums across the lanes (16 clocks an
// instruction and SM) are shared.  A step takes 5.5 us at N = 130, the chain of FP64 sums, root and barriers, and
// 10.6 at N = 1001, where the rows from shared memory and L2 add to it; a step launch took 10 and 13.1.
__device__ __forceinline__ double warp_sum(double x) {
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__global__ void __cluster_dims__(kLzCtas, 1, 1) __launch_bounds__(kLzClThreads, 1)
lz_cluster_kernel(const DevState* st, LzScratch* lz, int N, int ld, int R) {
  extern __shared__ __align__(16) float lz_smem[];
  constexpr int kParts = kLzCtas * ((kLzClusterN / kLzCtas + 31) / 32);
  __shared__ double p_alpha[kParts], p_ss[kParts], s_w[kLzClusterN / kLzCtas];
  __shared__ double s_b, s_ib;
  if (st->done || !lz->live) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = kLzClThreads / 32;
  const int c = blockIdx.x, S = (N + kLzCtas - 1) / kLzCtas, ew = (S + 31) / 32;   // ew: warps with entries
  const int i0 = c * S, rows = N - i0 < S ? (N - i0 > 0 ? N - i0 : 0) : S;
  double* r64 = reinterpret_cast<double*>(lz_smem);                                 // r of all entries
  float* q32 = reinterpret_cast<float*>(r64 + kLzCtas * S);
  float4* own = reinterpret_cast<float4*>(q32 + ld);                                // rows 0 .. R - 1
  const double* q0 = lz_vec(lz, ld, 0);
  const int h = ld / 4, G = (rows + 3) / 4;
  const float4* A = reinterpret_cast<const float4*>(lz_a32(lz, ld)) + (int64_t)i0 * h;
  for (int i = tid; i < (rows < R ? rows : R) * h; i += kLzClThreads) own[i] = A[i];
  double q = tid < rows ? q0[i0 + tid] : 0.0, qp = 0.0, bj = 0.0;
  for (int i = tid; i < ld; i += kLzClThreads) q32[i] = i < N ? (float)q0[i] : 0.f;
  const uint32_t a_pa = ptx::smem_u32(p_alpha), a_ps = ptx::smem_u32(p_ss), a_r = ptx::smem_u32(r64);
  // lane l < kLzCtas of a warp stores the warp's sum into the array of CTA l
  auto share = [&](uint32_t arr, double x) {
    if (lane < kLzCtas) ptx::st_cluster_f64(ptx::mapa_shared(arr + 8 * (c * ew + warp), lane), x);
  };
  auto total = [&](const double* p) {
    double t = 0.0;
    for (int n = lane; n < kLzCtas * ew; n += 32) t += p[n];
    return warp_sum(t);
  };
  ptx::cluster_sync();                                     // every CTA runs before the first remote store
  for (int j = 0; j < kLzSteps; ++j) {
    const float4* q4 = reinterpret_cast<const float4*>(q32);
    auto dot4 = [](const float4& x, const float4& v, float s) {
      s = fmaf(x.x, v.x, s); s = fmaf(x.y, v.y, s); s = fmaf(x.z, v.z, s);
      return fmaf(x.w, v.w, s);
    };
    for (int g = warp; g < G; g += nw) {                   // rows g, g + G, g + 2 G, g + 3 G
      const float4* x[4];
      #pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = g + k * G < rows ? g + k * G : g;
        x[k] = r < R ? own + r * h : A + (int64_t)r * h;
      }
      float s0[4] = {}, s1[4] = {};
      for (int i = lane; i < h; i += 64) {
        const bool more = i + 32 < h;
        const int i1 = more ? i + 32 : i;
        float4 a0[4], a1[4];
        #pragma unroll
        for (int k = 3; k >= 0; --k) { a0[k] = x[k][i]; a1[k] = x[k][i1]; }
        const float4 v0 = q4[i], v1 = q4[i1];
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
          s0[k] = dot4(a0[k], v0, s0[k]);
          if (more) s1[k] = dot4(a1[k], v1, s1[k]);
        }
      }
      // the sums of four rows across the lanes: halves, then quarters, of the warp take a row each
      double t[4];
      #pragma unroll
      for (int k = 0; k < 4; ++k) t[k] = (double)s0[k] + (double)s1[k];
      const bool up = lane & 16, odd = lane & 8;
      double u0 = up ? t[2] : t[0], u1 = up ? t[3] : t[1];
      u0 += __shfl_xor_sync(0xffffffffu, up ? t[0] : t[2], 16);
      u1 += __shfl_xor_sync(0xffffffffu, up ? t[1] : t[3], 16);
      double v = odd ? u1 : u0;
      v += __shfl_xor_sync(0xffffffffu, odd ? u0 : u1, 8);
      #pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int r = g + (lane >> 3) * G;
      if ((lane & 7) == 0 && r < rows) s_w[r] = v;
    }
    __syncthreads();
    const double w = tid < rows ? s_w[tid] : 0.0;
    if (warp < ew) share(a_pa, warp_sum(q * w));
    ptx::cluster_sync();
    double a = 0.0, r = 0.0;
    if (warp < ew) {
      a = total(p_alpha);
      if (j + 1 < kLzSteps) {
        r = w - a * q - (j > 0 ? bj * qp : 0.0);
        if (tid < S)
          for (int o = 0; o < kLzCtas; ++o) ptx::st_cluster_f64(ptx::mapa_shared(a_r + 8 * (c * S + tid), o), r);
        share(a_ps, warp_sum(r * r));
      }
    }
    if (j + 1 == kLzSteps) {                               // the last alpha closes the tridiagonal matrix
      if (c == 0 && tid == 0) {
        lz->alpha[j] = a;
        lz->m = kLzSteps;
        lz->live = 0;
      }
      break;
    }
    ptx::cluster_sync();
    if (warp == 0) {
      const double ss = total(p_ss);
      if (lane == 0) {                                     // one thread: FP64 operations run at 2 a clock and SM
        const double b = sqrt(ss);
        const bool finite = isfinite(a) && isfinite(b), more = finite && b > 1e-300;
        s_b = more ? b : -1.0;
        s_ib = 1.0 / b;
        if (c == 0) {
          lz->alpha[j] = finite ? a : __longlong_as_double(0x7ff8000000000000ll);
          lz->m = j + 1;
          lz->beta[j + 1] = b;
          if (!more) lz->live = 0;
        }
      }
    }
    __syncthreads();
    if (s_b < 0.0) break;                                  // the same in every CTA
    bj = s_b;
    const double ib = s_ib;
    qp = q;
    q = r * ib;
    for (int i = tid; i < N; i += kLzClThreads) q32[i] = (float)(r64[i] * ib);
    __syncthreads();
  }
  ptx::cluster_sync();                                     // no CTA leaves while another still writes to it
}

// Number of eigenvalues of the m x m tridiagonal (alpha, beta) below x: the count of negative
// pivots of the LDL^T factorisation of T - x I (Sturm sequence), tiny pivots pushed to -pivmin.
__device__ __forceinline__ int sturm_count(const float* al, const float* be2, int m, float x) {
  constexpr float kPivMin = 1e-30f;
  float d = al[0] - x;
  if (fabsf(d) < kPivMin) d = -kPivMin;
  int cnt = d < 0.0f;
  for (int i = 1; i < m; ++i) {
    d = (al[i] - x) - be2[i] / d;
    if (fabsf(d) < kPivMin) d = -kPivMin;
    cnt += d < 0.0f;
  }
  return cnt;
}

// Closes the last step (alpha from its partials, `blocks` of them) and takes the extreme eigenvalues of the
// tridiagonal matrix: 512 threads per side, each a point of the bracket.
__global__ void __launch_bounds__(kSturmThreads)
lz_eig_kernel(DevState* st, const LzScratch* lz, int blocks) {
  __shared__ float al[kLzSteps], be2[kLzSteps];
  __shared__ int s_bad, s_cnt[2];
  __shared__ float s_lo[2], s_hi[2];
  if (st->done) return;
  const int tid = threadIdx.x, lane = tid & 31, side = tid >> 9, pt = tid & 511;
  const int done = lz->m;                        // finished in the steps; a live run has one more to close
  const int m = done + (lz->live ? 1 : 0);
  if (tid < 32) {
    double last = 0.0;
    for (int t = lane; t < blocks; t += 32) last += lz->part[(m - 1) & 1][t];
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) last += __shfl_xor_sync(0xffffffffu, last, o);
    bool bad = m < 1;
    if (lane < m) {
      const double a = lane < done ? lz->alpha[lane] : last, b = lane ? lz->beta[lane] : 0.0;
      bad = bad || !isfinite(a) || !isfinite(b) || fabs(a) > 1e30 || fabs(b) > 1e15;
      al[lane] = (float)a;
      be2[lane] = (float)(b * b);
    }
    bad = __any_sync(0xffffffffu, bad);
    __syncwarp();
    if (lane == 0) s_bad = bad;
    // Gershgorin interval of T
    float lo = INFINITY, hi = -INFINITY;
    if (!bad && lane < m) {
      const float rad = sqrtf(be2[lane]) + (lane + 1 < m ? sqrtf(be2[lane + 1]) : 0.0f);
      lo = al[lane] - rad;
      hi = al[lane] + rad;
    }
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      const float pad = 1e-30f + 0x1p-20f * fmaxf(fabsf(lo), fabsf(hi));
      s_lo[0] = s_lo[1] = lo - pad;              // brackets of the largest (side 0) and the smallest (side 1)
      s_hi[0] = s_hi[1] = hi + pad;
    }
  }
  __syncthreads();
  if (s_bad) {
    if (tid == 0) st->spec_e = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  for (int round = 0; round < kSturmRounds; ++round) {
    if (tid < 2) s_cnt[tid] = 0;
    __syncthreads();
    const float lo = s_lo[side], hi = s_hi[side];
    auto point = [&](int i) { return lo + (hi - lo) * ((float)(i + 1) / 513.0f); };
    const int c = sturm_count(al, be2, m, point(pt));
    // largest: the points with fewer than m eigenvalues below them form a prefix; smallest: those with none
    const unsigned v = __ballot_sync(0xffffffffu, side == 0 ? c <= m - 1 : c == 0);
    if (lane == 0) atomicAdd(&s_cnt[side], __popc(v));
    __syncthreads();
    const int n = s_cnt[side];
    __syncthreads();
    if (pt == 0) {
      if (n > 0) s_lo[side] = point(n - 1);
      if (n < 512) s_hi[side] = point(n);
    }
    __syncthreads();
  }
  if (tid == 0) {
    const double top = 0.5 * ((double)s_lo[0] + (double)s_hi[0]), bot = 0.5 * ((double)s_lo[1] + (double)s_hi[1]);
    st->spec_e = fmax(fabs(top), fabs(bot)) / lz->scale;
  }
}

// Block-sparse path: the mixed norm's matrix of block norms M_IJ = ||(X - X^2)_IJ||_F (nb x nb,
// both triangles) from the square's upper-pair records (v^2 part counted twice off the
// diagonal), scaled and rounded to FP32 after a zero fill.
__global__ void lz_zero_kernel(const DevState* st, LzScratch* lz, int ld) {
  if (st->done) return;
  float4* A = reinterpret_cast<float4*>(lz_a32(lz, ld));
  const int64_t total = (int64_t)ld * ld / 4;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    A[e] = make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void lz_form_pairs_kernel(const DevState* st, const int* __restrict__ row, const int* __restrict__ col,
                                     const int* nnz_p, const double* __restrict__ part, LzScratch* lz, int ld) {
  if (st->done) return;
  const int nnz = *nnz_p;
  const double sc = lz->scale;
  float* A = lz_a32(lz, ld);
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += gridDim.x * blockDim.x) {
    const int I = row[q], J = col[q];
    const double v2 = part[2 * (int64_t)q] * (I == J ? 1.0 : 0.5);
    const float w = (float)(sqrt(v2) * sc);
    A[(int64_t)I * ld + J] = w;
    A[(int64_t)J * ld + I] = w;
  }
}

// Step launch: a row per warp, 16 warps a CTA up to the grid cap, then 32.
int step_threads(int N) { return N <= 16 * kLzMvBlocks ? 512 : kLzMvThreads; }
int step_blocks(int N) {
  const int per = step_threads(N) / 32, b = (N + per - 1) / per;
  return b < kLzMvBlocks ? (b < 1 ? 1 : b) : kLzMvBlocks;
}
int step_smem(int N, int ld) { return N <= kLzSmemN ? 4 * ld : 0; }

// Shared memory of the cluster's CTAs without rows of A, and how many rows fit beside it.
int cluster_base(int N, int ld) { return 8 * kLzCtas * ((N + kLzCtas - 1) / kLzCtas) + 4 * ld; }
int cluster_rows(int N, int ld) {
  const int S = (N + kLzCtas - 1) / kLzCtas, fit = (kLzClSmem - cluster_base(N, ld)) / (4 * ld);
  return fit < S ? fit : S;
}

// Whether the device can hold the cluster (its size is above the portable eight).
bool cluster_fits() {
  static PerDevice fits;
  return fits.get([](int) {
    const void* k = (const void*)lz_cluster_kernel;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kLzCtas);
    cfg.blockDim = dim3(kLzClThreads);
    cfg.dynamicSmemBytes = kLzClSmem;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kLzCtas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kLzClSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      return 1;
    }
    return 2;
  }) == 2;
}

int form_blocks(int ld) {
  const int64_t b = ((int64_t)ld * (ld / 2) + 255) / 256;
  return (int)(b < 152 * 16 ? b : 152 * 16);
}

}  // namespace

cudaError_t lanczos_prepare() {
  (void)cluster_fits();                          // asks the device once, before any capture
  static PerDevice done;
  cudaError_t e = cudaSuccess;
  done.get([&](int) {
    e = cudaFuncSetAttribute(lz_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kLzSmemN + 4096);
    return e == cudaSuccess ? 1 : 0;
  });
  return e;
}

size_t lanczos_scratch_bytes(int ld) {
  return kVecOff + 5 * sizeof(double) * (size_t)ld + sizeof(float) * ((size_t)ld + (size_t)ld * ld);
}

// start, form (the caller's kernel and arguments), the steps and eig, on a stream or as a chain of graph nodes.
static cudaError_t emit(f64tc::Sink& sink, DevState* st, const double* part, int ntiles, int rec, LzScratch* lz,
                        int N, int ld, const void* form, void** form_args, const void* fill = nullptr,
                        void** fill_args = nullptr) {
  cudaError_t e = lanczos_prepare();
  if (e != cudaSuccess) return e;
  const DevState* cst = st;
  const LzScratch* clz = lz;
  void* a0[] = {&cst, &part, &ntiles, &rec, &lz, &N, &ld};
  if ((e = sink.put((const void*)lz_start_kernel, dim3(1), dim3(kLzThreads), 0, a0)) != cudaSuccess) return e;
  if (fill && (e = sink.put(fill, dim3(form_blocks(ld)), dim3(256), 0, fill_args)) != cudaSuccess) return e;
  if ((e = sink.put(form, dim3(form_blocks(ld)), dim3(256), 0, form_args)) != cudaSuccess) return e;
  if (N <= kLzClusterN && cluster_fits()) {
    int R = cluster_rows(N, ld);
    void* a[] = {&cst, &lz, &N, &ld, &R};
    e = sink.put((const void*)lz_cluster_kernel, dim3(kLzCtas), dim3(kLzClThreads), cluster_base(N, ld) + 4 * ld * R, a);
    if (e != cudaSuccess) return e;
  } else {
    for (int j = 0; j < kLzSteps; ++j) {
      void* a[] = {&cst, &lz, &j, &N, &ld};
      e = sink.put((const void*)lz_step_kernel, dim3(step_blocks(N)), dim3(step_threads(N)), step_smem(N, ld), a);
      if (e != cudaSuccess) return e;
    }
  }
  int blocks = step_blocks(N);
  void* a1[] = {&st, &clz, &blocks};
  return sink.put((const void*)lz_eig_kernel, dim3(1), dim3(kSturmThreads), 0, a1);
}

static cudaError_t emit_f64(f64tc::Sink& sink, DevState* st, const double* buf0, const double* buf1, const double* S,
                            const double* part, int ntiles, void* scratch, int N, int ld) {
  LzScratch* lz = static_cast<LzScratch*>(scratch);
  const DevState* cst = st;
  void* form[] = {&cst, &buf0, &buf1, &S, &lz};
  return emit(sink, st, part, ntiles, 2, lz, N, ld, (const void*)lz_form_kernel, form);
}

static cudaError_t emit_tc(f64tc::Sink& sink, DevState* st, const tc::Instance* inst, const double* part, int nparts,
                           void* scratch, int N, int ld) {
  LzScratch* lz = static_cast<LzScratch*>(scratch);
  const DevState* cst = st;
  void* form[] = {&cst, &inst, &lz};
  return emit(sink, st, part, nparts, 4, lz, N, ld, (const void*)lz_form_tc_kernel, form);
}

cudaError_t add_lanczos_nodes(cudaGraph_t g, cudaGraphNode_t dep, DevState* st, const double* buf0,
                              const double* buf1, const double* S, const double* part, int ntiles, void* scratch,
                              int N, int ld, cudaGraphNode_t* last) {
  f64tc::Sink sink;
  sink.g = g;
  sink.last = dep;
  const cudaError_t e = emit_f64(sink, st, buf0, buf1, S, part, ntiles, scratch, N, ld);
  *last = sink.last;
  return e;
}

cudaError_t launch_lanczos(DevState* st, const double* buf0, const double* buf1, const double* S,
                           const double* part, int ntiles, void* scratch, int N, int ld, cudaStream_t s) {
  f64tc::Sink sink;
  sink.s = s;
  return emit_f64(sink, st, buf0, buf1, S, part, ntiles, scratch, N, ld);
}

// Tensor-core path, one problem: the estimate for the square just written into `inst`'s arena;
// `part` holds its nparts records of 4 doubles (v^2 first).
cudaError_t add_lanczos_tc_nodes(cudaGraph_t g, cudaGraphNode_t dep, DevState* st, const tc::Instance* inst,
                                 const double* part, int nparts, void* scratch, int N, int ld,
                                 cudaGraphNode_t* last) {
  f64tc::Sink sink;
  sink.g = g;
  sink.last = dep;
  const cudaError_t e = emit_tc(sink, st, inst, part, nparts, scratch, N, ld);
  *last = sink.last;
  return e;
}

cudaError_t launch_lanczos_tc(DevState* st, const tc::Instance* inst, const double* part, int nparts, void* scratch,
                              int N, int ld, cudaStream_t s) {
  f64tc::Sink sink;
  sink.s = s;
  return emit_tc(sink, st, inst, part, nparts, scratch, N, ld);
}

cudaError_t launch_lanczos_pairs(DevState* st, const int* row, const int* col, const int* nnz_p, const double* part,
                                 const double* sums, int nsums, void* scratch, int nb, int ld, cudaStream_t s) {
  LzScratch* lz = static_cast<LzScratch*>(scratch);
  const DevState* cst = st;
  f64tc::Sink sink;
  sink.s = s;
  void* fill[] = {&cst, &lz, &ld};
  void* form[] = {&cst, &row, &col, &nnz_p, &part, &lz, &ld};
  return emit(sink, st, sums, nsums, 2, lz, nb, ld, (const void*)lz_form_pairs_kernel, form,
              (const void*)lz_zero_kernel, fill);
}

}  // namespace sp2
