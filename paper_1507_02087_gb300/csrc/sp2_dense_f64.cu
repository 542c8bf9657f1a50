// FP64 dense SP2 path: Gershgorin bounds, the initial scaling, the symmetric
// squaring with its fused polynomial epilogue, the device-side stop test and the
// output copy (Alg. 3 of Kruchinina, Rudberg, Rubensson, arXiv:1507.02087).
//
// Data layout: the two ping-pong buffers hold X_{i-1} and X_i as ld x ld FP64
// row-major matrices, ld = N rounded up to a multiple of 64, with a zero border.
// The border stays zero through the iteration (0^2 = 0 and 2*0 - 0 = 0), so the
// squaring works on whole 64 x 64 tiles with no bounds checks.
#include "sp2_common.cuh"
#include "sp2_f64_tc.cuh"
#include "sp2_kernels.h"

namespace sp2 {

// ---- Gershgorin bounds (a1) ------------------------------------------------------------
// One warp per row: lo_i = F_ii - sum_{j != i} |F_ij|, hi_i = F_ii + sum_{j != i} |F_ij|.
// Each block keeps the min / max over its rows; the init kernel combines blocks.
constexpr int kGershThreads = 256;

__global__ void __launch_bounds__(kGershThreads)
gershgorin_kernel(const double* __restrict__ F, int64_t ldf, int N, double* __restrict__ part_lo,
                  double* __restrict__ part_hi, int* __restrict__ part_bad) {
  __shared__ double s_lo[kGershThreads / 32], s_hi[kGershThreads / 32];
  __shared__ int s_bad[kGershThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int warps_total = gridDim.x * (kGershThreads / 32);
  double lo = INFINITY, hi = -INFINITY;
  int bad = 0;
  for (int i = blockIdx.x * (kGershThreads / 32) + warp; i < N; i += warps_total) {
    const double* row = F + (int64_t)i * ldf;
    double r = 0.0;
    for (int j = lane; j < N; j += 32) {
      double a = row[j];
      if (j != i) r += fabs(a);
      if (!isfinite(a)) bad = 1;
    }
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    const double d = row[i];
    lo = fmin(lo, d - r);
    hi = fmax(hi, d + r);
  }
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; s_bad[warp] = bad; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kGershThreads / 32; ++w) {
      s_lo[0] = fmin(s_lo[0], s_lo[w]);
      s_hi[0] = fmax(s_hi[0], s_hi[w]);
      s_bad[0] |= s_bad[w];
    }
    part_lo[blockIdx.x] = s_lo[0];
    part_hi[blockIdx.x] = s_hi[0];
    part_bad[blockIdx.x] = s_bad[0];
  }
}

// ---- run initialisation: bounds, special cases, Tr[X_0] -------------------------------
constexpr int kInitThreads = 1024;

__global__ void __launch_bounds__(kInitThreads)
init_kernel(DevState* st, const double* __restrict__ F, int64_t ldf, const double* __restrict__ part_lo,
            const double* __restrict__ part_hi, const int* __restrict__ part_bad, int nparts) {
  __shared__ double sm[32];
  __shared__ double s_lmin, s_lmax;
  __shared__ int s_bad;
  if (threadIdx.x == 0) {
    double lo = INFINITY, hi = -INFINITY;
    int bad = 0;
    for (int b = 0; b < nparts; ++b) {
      lo = fmin(lo, part_lo[b]);
      hi = fmax(hi, part_hi[b]);
      bad |= part_bad[b];
    }
    if (!isfinite(lo) || !isfinite(hi)) bad = 1;
    if (st->ubounds) {                           // any outer bounds of the spectrum serve (§3)
      lo = st->ub_lo;
      hi = st->ub_hi;
    }
    s_lmin = lo; s_lmax = hi; s_bad = bad;
  }
  __syncthreads();
  const double lmin = s_lmin, lmax = s_lmax;
  const int N = st->N, nocc = st->nocc;
  // X_0 = (sa I - F) / sw: (lmax, lmax - lmin) for SP2 (Alg. 3), (mu + gamma/2, gamma) with
  // gamma = 2 max(lmax - mu, mu - lmin) for McWeeny (§3)
  double sa = lmax, sw = lmax - lmin;
  if (st->mcw) {
    sw = 2.0 * fmax(lmax - st->mu, st->mu - lmin);
    sa = st->mu + 0.5 * sw;
  }
  // Tr[X_0] over the stored diagonal, each entry rounded exactly as the scaling kernel
  // rounds it.
  double t = 0.0;
  const double w = sw;
  const int r32 = st->round_fp32;
  for (int i = threadIdx.x; i < N; i += kInitThreads) {
    const double x = (sa - F[(int64_t)i * ldf + i]) / w;
    t += r32 ? (double)(float)x : x;
  }
  t = block_sum<kInitThreads>(t, sm);
  if (threadIdx.x == 0) {
    st->lmin = lmin; st->lmax = lmax;
    st->scale_a = sa; st->scale_w = sw;
    st->dk = 0;
    st->tr_shift = 0.0;
    st->wrote = 0;
    st->k = 0; st->done = 0; st->n_out = 0; st->reason = SP2_STOP_EXACT;
    st->status = SP2_OK; st->out_buf = 0; st->out_mode = OUT_COPY; st->hist_len = 0;
    st->tr[0] = 0.0; st->p[0] = 0;
    if (s_bad) {
      st->status = SP2_ERR_NONFINITE; st->done = 1; st->out_mode = OUT_NAN;
    } else if (nocc == 0) {
      st->done = 1; st->out_mode = OUT_ZERO;
    } else if (nocc == N) {
      st->done = 1; st->out_mode = OUT_IDENTITY;
    } else if (!(lmax > lmin)) {
      st->status = SP2_ERR_NO_GAP; st->done = 1; st->out_mode = OUT_NAN;
    } else {
      st->tr[0] = t;
      if (st->mcw) {
        if (!(sw > 0.0)) { st->status = SP2_ERR_NO_GAP; st->done = 1; st->out_mode = OUT_NAN; }
        else mcw_schedule(st, sw);
      } else if (st->acc && !acc_schedule(st)) {   // SP2-ACC: Alg. 4 from the bounds just found
        st->status = SP2_ERR_INVALID_ARG; st->done = 1; st->out_mode = OUT_NAN;
      }
    }
  }
}

// ---- initial scaling X_0 = (lmax I - F) / (lmax - lmin) (a2) -------------------------
__global__ void scale_kernel(const DevState* st, const double* __restrict__ F, int64_t ldf,
                             double* __restrict__ X0, int ld) {
  if (st->done) return;
  const int N = st->N;
  const double lmax = st->scale_a, w = st->scale_w;   // (lmax, lmax - lmin) for SP2
  __shared__ double s_iw;
  if (threadIdx.x == 0) s_iw = 1.0 / w;
  __syncthreads();
  const double iw = s_iw;
  const int64_t total = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / N), j = (int)(e % N);
    const double f = F[(int64_t)i * ldf + j];
    X0[(int64_t)i * ld + j] = divide_shared((i == j ? lmax : 0.0) - f, w, iw);
  }
}

// ---- symmetric squaring with the fused SP2 epilogue (a3, a4, a5) -----------------------
// CTA tile 64 x 64 of S = X X^T (= X^2, X symmetric) for an upper tile (I <= J), K in
// steps of 16 staged through shared memory, 256 threads each owning a 4 x 4 block.
// Epilogue: X_k = S (p_k = 1) or 2 X - S (p_k = 0) written to the tile and its mirror;
// the tile's share of ||X_{k-1} - S||_F^2 (off-diagonal tiles count twice) and of
// Tr[X_k] go to a per-tile slot, summed in a fixed order by the finalize kernel.
constexpr int kTile = 64, kTK = 16, kSyrkThreads = 256;

// gen = 1 (accelerated path): X_k = ca S + cb X + cc I, the identity term on the N true
// diagonal entries only (the zero border stays zero).
// Bin (if given): the product is Xin Bin^T instead of Xin Xin^T (the McWeeny step's S X);
// the epilogue's x is still the element of Xin.
__device__ __forceinline__ void syrk_f64_tile(const double* __restrict__ Xin, double* __restrict__ Xout, int ld,
                                              int pk, double* __restrict__ part, int gen = 0, double ca = 0.0,
                                              double cb = 0.0, double cc = 0.0, int N = 0,
                                              const double* __restrict__ Bin = nullptr) {
  __shared__ double As[2][kTK][kTile + 1];
  __shared__ double Bs[2][kTK][kTile + 1];
  __shared__ double sred[32];
  const int T = ld / kTile;
  int I, J;
  upper_tile(blockIdx.x, T, I, J);
  const int tid = threadIdx.x;
  const int ty = tid >> 4, tx = tid & 15;
  const int lm = tid >> 4, lk = tid & 15;        // loader: rows lm + 16 j, column lk
  const double* Arow = Xin + (int64_t)(I * kTile) * ld;
  const double* Brow = (Bin ? Bin : Xin) + (int64_t)(J * kTile) * ld;

  double acc[4][4];
  #pragma unroll
  for (int r = 0; r < 4; ++r)
    #pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

  double ra[4], rb[4];
  #pragma unroll
  for (int j = 0; j < 4; ++j) {
    ra[j] = Arow[(int64_t)(lm + 16 * j) * ld + lk];
    rb[j] = Brow[(int64_t)(lm + 16 * j) * ld + lk];
  }
  int buf = 0;
  for (int k0 = 0; k0 < ld; k0 += kTK) {
    #pragma unroll
    for (int j = 0; j < 4; ++j) {
      As[buf][lk][lm + 16 * j] = ra[j];
      Bs[buf][lk][lm + 16 * j] = rb[j];
    }
    __syncthreads();
    if (k0 + kTK < ld) {
      #pragma unroll
      for (int j = 0; j < 4; ++j) {
        ra[j] = Arow[(int64_t)(lm + 16 * j) * ld + k0 + kTK + lk];
        rb[j] = Brow[(int64_t)(lm + 16 * j) * ld + k0 + kTK + lk];
      }
    }
    #pragma unroll
    for (int kk = 0; kk < kTK; ++kk) {
      double a[4], b[4];
      #pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[buf][kk][ty * 4 + r];
      #pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = Bs[buf][kk][tx * 4 + c];
      #pragma unroll
      for (int r = 0; r < 4; ++r)
        #pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    buf ^= 1;
  }

  double v2 = 0.0, trace = 0.0;
  #pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int gi = I * kTile + ty * 4 + r;
    #pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int gj = J * kTile + tx * 4 + c;
      const double x = Xin[(int64_t)gi * ld + gj];
      const double s = acc[r][c];
      const double d = x - s;
      v2 = fma(d, d, v2);
      const double xn = gen ? fma(ca, s, fma(cb, x, (gi == gj && gi < N) ? cc : 0.0)) : (pk ? s : (2.0 * x - s));
      Xout[(int64_t)gi * ld + gj] = xn;
      if (I != J) Xout[(int64_t)gj * ld + gi] = xn;
      if (gi == gj) trace += xn;
    }
  }
  if (I != J) v2 *= 2.0;
  v2 = block_sum<kSyrkThreads>(v2, sred);
  trace = block_sum<kSyrkThreads>(trace, sred);
  if (tid == 0) {
    part[2 * blockIdx.x] = v2;
    part[2 * blockIdx.x + 1] = trace;
  }
}


// ---- the same for the smallest problems, in 8 x 8 tiles ------------------------------------------
// Up to N = kSmallN a 64 x 64 tile per CTA leaves almost the whole chip idle while one SM works through the
// tile at 2 multiply-adds a clock (65 us at N = 64).  Here a CTA of 128 threads has an 8 x 8 tile of the upper
// triangle, one element per pair of threads, each with half of the k range; the rows of both operands are
// staged whole.  A tile's record goes to its place among the 64 of its 64 x 64 tile.  One purification at
// N = 64: 2.78 -> 0.54 ms.
constexpr int kSmallN = f64tc::kMinN - 1;        // 128
constexpr int kST = 8, kSmallThreads = 128, kSmallRecs = 64;
constexpr int kSmallLd = kSmallN + 2;            // row stride in shared memory: rows on different banks

__device__ __forceinline__ void syrk_small_tile(const double* __restrict__ Xin, const double* __restrict__ Bin,
                                                double* __restrict__ Xout, int ld, int N, int pk,
                                                double* __restrict__ part, int gen, double ca, double cb, double cc) {
  __shared__ __align__(16) double As[kST][kSmallLd], Bs[kST][kSmallLd];
  __shared__ double half[kST * kST];
  __shared__ double sred[2][2];
  int I, J;
  upper_tile(blockIdx.x, (N + kST - 1) / kST, I, J);
  const int tid = threadIdx.x;
  const int K = (N + 7) & ~7;                    // the border beyond N is zero
  for (int e = tid; e < kST * (K / 2); e += kSmallThreads) {
    const int r = e / (K / 2), c = 2 * (e % (K / 2));
    *reinterpret_cast<double2*>(&As[r][c]) = *reinterpret_cast<const double2*>(Xin + (int64_t)(I * kST + r) * ld + c);
    *reinterpret_cast<double2*>(&Bs[r][c]) = *reinterpret_cast<const double2*>(Bin + (int64_t)(J * kST + r) * ld + c);
  }
  __syncthreads();
  const int el = tid & 63, r = el >> 3, c = el & 7, kh = tid >> 6;
  double acc = 0.0;
  const int k0 = kh * (K / 2), k1 = k0 + K / 2;
  #pragma unroll 8
  for (int k = k0; k < k1; ++k) acc = fma(As[r][k], Bs[c][k], acc);
  if (kh) half[el] = acc;
  __syncthreads();
  double v2 = 0.0, trace = 0.0;
  if (kh == 0) {
    const double s = acc + half[el];
    const int gi = I * kST + r, gj = J * kST + c;
    const double x = Xin[(int64_t)gi * ld + gj];
    const double d = x - s;
    v2 = I == J ? d * d : 2.0 * (d * d);
    const double xn = gen ? fma(ca, s, fma(cb, x, (gi == gj && gi < N) ? cc : 0.0)) : (pk ? s : (2.0 * x - s));
    if (gj >= gi) {
      Xout[(int64_t)gi * ld + gj] = xn;
      if (gj > gi) Xout[(int64_t)gj * ld + gi] = xn;
    }
    if (gi == gj) trace = xn;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v2 += __shfl_xor_sync(0xffffffffu, v2, o);
      trace += __shfl_xor_sync(0xffffffffu, trace, o);
    }
    if ((tid & 31) == 0) { sred[tid >> 5][0] = v2; sred[tid >> 5][1] = trace; }
  }
  __syncthreads();
  if (tid == 0) {
    double* dst = part + 2 * (kSmallRecs * upper_index(I / 8, J / 8, ld / kTile) + 8 * (I & 7) + (J & 7));
    dst[0] = sred[0][0] + sred[1][0];
    dst[1] = sred[0][1] + sred[1][1];
  }
}

// One product of the loop, small problems: op 0 the SP2 square, 1 the McWeeny step's shifted square into S, 2 its
// product S X_{k-1} (after the stop test).  The polynomials are those of the kernels below.
__global__ void __launch_bounds__(kSmallThreads)
small_product_kernel(const DevState* st, double* buf0, double* buf1, double* S, double* part, int op) {
  if (st->done) return;
  const int k = st->k, ld = st->ld, N = st->N;
  if (op == 1) {
    const double* Xin = (k & 1) ? buf1 : buf0;
    const double a = st->alpha[k + 1], c = 0.5 * (1.0 - a);
    syrk_small_tile(Xin, Xin, S, ld, N, 1, part, 1, a * a, 2.0 * a * c, c * c);
  } else if (op == 2) {
    const double a = st->alpha[k], c = 0.5 * (1.0 - a);
    syrk_small_tile(S, ((k - 1) & 1) ? buf1 : buf0, (k & 1) ? buf1 : buf0, ld, N, 1, part, 1, -2.0 * a, 3.0 - 2.0 * c, 0.0);
  } else {
    const double* Xin = (k & 1) ? buf1 : buf0;
    double* Xout = (k & 1) ? buf0 : buf1;
    double ca = 0.0, cb = 0.0, cc = 0.0;
    const int pk = st->acc ? acc_step(st, k + 1, ca, cb, cc) : (st->tr[k] > (double)st->nocc ? 1 : 0);
    syrk_small_tile(Xin, Xin, Xout, ld, N, pk, part, st->acc, ca, cb, cc);
  }
}

__global__ void __launch_bounds__(kSyrkThreads)
syrk_f64_kernel(const DevState* st, double* buf0, double* buf1, double* __restrict__ part) {
  if (st->done) return;
  const int kprev = st->k;                      // X_{k-1} with k = kprev + 1
  const double* Xin = (kprev & 1) ? buf1 : buf0;
  double* Xout = (kprev & 1) ? buf0 : buf1;
  if (st->acc) {                                // Alg. 5: the scheduled polynomial
    double ca, cb, cc;
    const int pk = acc_step(st, kprev + 1, ca, cb, cc);
    syrk_f64_tile(Xin, Xout, st->ld, pk, part, 1, ca, cb, cc, st->N);
    return;
  }
  const int pk = st->tr[kprev] > (double)st->nocc ? 1 : 0;   // Alg. 3 trace test
  syrk_f64_tile(Xin, Xout, st->ld, pk, part);
}

// ---- McWeeny expansion (§3), two products per step ------------------------------------------
// Step k (from X_{k-1} in buf[(k-1) & 1]), with X_s = alpha (X - I/2) + I/2 = alpha X + c I,
// c = (1 - alpha)/2:  mcw_square writes S_s = X_s^2 = alpha^2 X^2 + 2 alpha c X + c^2 I to S and
// the partials of ||X_{k-1} - X_{k-1}^2||_F for the stop test; mcw_prod (after the test, unless
// it stopped) writes X_k = 3 S_s - 2 S_s X_s = (3 - 2c) S_s - 2 alpha S_s X_{k-1} to buf[k & 1].
__global__ void __launch_bounds__(kSyrkThreads)
mcw_square_kernel(const DevState* st, const double* buf0, const double* buf1, double* S, double* __restrict__ part) {
  if (st->done) return;
  const int j = st->k + 1;
  const double* Xin = (st->k & 1) ? buf1 : buf0;
  const double a = st->alpha[j], c = 0.5 * (1.0 - a);
  syrk_f64_tile(Xin, S, st->ld, 1, part, 1, a * a, 2.0 * a * c, c * c, st->N);
}

__global__ void __launch_bounds__(kSyrkThreads)
mcw_prod_kernel(const DevState* st, double* buf0, double* buf1, const double* S, double* __restrict__ part) {
  if (st->done) return;
  const int k = st->k;                             // the square just recorded
  const double* Xprev = ((k - 1) & 1) ? buf1 : buf0;
  double* Xout = (k & 1) ? buf1 : buf0;
  const double a = st->alpha[k], c = 0.5 * (1.0 - a);
  syrk_f64_tile(S, Xout, st->ld, 1, part, 1, -2.0 * a, 3.0 - 2.0 * c, 0.0, st->N, Xprev);
}

// FP64 purification step on the mixed path's result: the polynomial alternates with
// the last one of the low-precision expansion (step 0 takes the other one, step 1 the
// same one), so each pair squares the remaining eigenvalue error (the composition of
// x^2 and 2x - x^2, §4).
__global__ void __launch_bounds__(kSyrkThreads)
refine_f64_kernel(const DevState* st, const double* Xin, double* Xout, int ld, int step,
                  double* __restrict__ part) {
  if (!corrects_run(st)) return;      // failed or capped runs: D stays the assembled X_n
  const int plast = st->p[st->n_out];
  const int pk = step == 2 ? 1 : (step == 0 ? 1 - plast : plast);   // step 2: the plain square X^2
  syrk_f64_tile(Xin, Xout, ld, pk, part);
}

// ---- per-iteration reduction and stop test (a5 reductions, a7) ----------------------------
constexpr int kFinThreads = 1024;

// Partials come in records of `stride` doubles.  FP64 path (stride 2): (v^2 part,
// Tr[X_k] part) with Tr[X_k] summed over the stored diagonal.  Mixed path (stride 4):
// (v^2 part, ||X_{k-1}||_F^2 part, Tr[X_{k-1}] part, 0): there Tr[X_k] is taken from
// the identity Tr[X^2] = ||X||_F^2 for symmetric X (Tr[X_k] = ||X_{k-1}||_F^2 after
// X^2, 2 Tr[X_{k-1}] - ||X_{k-1}||_F^2 after 2X - X^2), so the polynomial choice does
// not inherit the bias of the tensor cores' accumulation.  A 64 x 64 tile has `recs` records (see
// recs_of).
__global__ void __launch_bounds__(kFinThreads)
finalize_kernel(DevState* st, const double* __restrict__ part, int nparts, int stride, int recs,
                cudaGraphConditionalHandle cond, double* mscr) {
  __shared__ double sm[96];
  if (st->done) {
    if (threadIdx.x == 0) cudaGraphSetConditional(cond, 0);
    return;
  }
  touch_state(st, st->k);
  double a = 0.0, b = 0.0, c = 0.0;
  for (int t = threadIdx.x; t < nparts; t += kFinThreads) {
    a += part[(int64_t)stride * t];
    b += part[(int64_t)stride * t + 1];
    if (stride > 2) c += part[(int64_t)stride * t + 2];
  }
  block_sum3<kFinThreads>(a, b, c, nparts, sm);
  double vk = 0.0;                               // v_{k-1} = ||X_{k-1} - X_{k-1}^2||_F; one thread takes the root: FP64
  if (threadIdx.x == 0) vk = st->norm == 2 ? st->spec_e : sqrt(a);   // operations run at 2 a clock and SM, so in all
                                                 // 1024 threads it took 5 us (or e_{k-1}, the Lanczos estimate)
  if (st->norm == 1 && mscr) {                   // or m_{k-1}, the mixed norm over 64 x 64 tiles
    const int T = st->ld / kTile;
    vk = mixed_norm_cta<kFinThreads>(T, mscr, sm, [&](int I, int J) {
      double v2 = 0.0;
      for (int q = 0; q < recs; ++q) v2 += part[(int64_t)stride * (recs * upper_index(I, J, T) + q)];
      return I == J ? v2 : 0.5 * v2;             // off-diagonal tiles hold both mirror halves
    });
  }
  if (threadIdx.x != 0) return;

  const int k = st->k + 1;                       // the square just completed
  double ca = 0.0, cb = 0.0, cc = 0.0;
  const int pk = st->mcw ? 1 : st->acc ? acc_step(st, k, ca, cb, cc) : (st->tr[k - 1] > (double)st->nocc ? 1 : 0);
  double tr_new, tr_ref;
  if (stride > 2) {
    tr_new = st->acc ? ca * b + cb * c + cc * (double)st->N : (pk ? b : 2.0 * c - b);
    tr_ref = c;
  } else {
    tr_new = st->mcw ? 0.0 : b + st->tr_shift;   // McWeeny: no trace rule, none recorded
    tr_ref = st->tr[k - 1];
  }
  if (record_and_test(st, pk, vk, tr_new, tr_ref)) cudaGraphSetConditional(cond, 0);
}

// ---- output -----------------------------------------------------------------------------
__global__ void copy_out_kernel(const DevState* st, const double* __restrict__ buf0,
                                const double* __restrict__ buf1, int ld, double* __restrict__ D,
                                int64_t ldd) {
  const int N = st->N;
  const int mode = st->out_mode;
  const double* __restrict__ X = st->out_buf ? buf1 : buf0;
  const int64_t total = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / N), j = (int)(e % N);
    double val;
    if (mode == OUT_COPY) val = X[(int64_t)i * ld + j];
    else if (mode == OUT_ZERO) val = 0.0;
    else if (mode == OUT_IDENTITY) val = (i == j) ? 1.0 : 0.0;
    else val = __longlong_as_double(0x7ff8000000000000ll);
    D[(int64_t)i * ldd + j] = val;
  }
}

// Reduction + stop test of one FP64 square for loops driven without a CUDA graph:
// the same rules as finalize_kernel (stride 2), ending the loop through st->done only.
__global__ void __launch_bounds__(kFinThreads)
finalize_plain_kernel(DevState* st, const double* __restrict__ part, int nparts, int recs, double* mscr) {
  __shared__ double sm[96];
  if (st->done) return;
  touch_state(st, st->k);
  double a = 0.0, b = 0.0, c = 0.0;
  for (int t = threadIdx.x; t < nparts; t += kFinThreads) {
    a += part[2 * (int64_t)t];
    b += part[2 * (int64_t)t + 1];
  }
  block_sum3<kFinThreads>(a, b, c, nparts, sm);
  double vk = 0.0;
  if (threadIdx.x == 0) vk = st->norm == 2 ? st->spec_e : sqrt(a);
  if (st->norm == 1 && mscr) {
    const int T = st->ld / kTile;
    vk = mixed_norm_cta<kFinThreads>(T, mscr, sm, [&](int I, int J) {
      double v2 = 0.0;
      for (int q = 0; q < recs; ++q) v2 += part[2 * (recs * upper_index(I, J, T) + q)];
      return I == J ? v2 : 0.5 * v2;
    });
  }
  if (threadIdx.x != 0) return;
  const int k = st->k + 1;
  double ca, cb, cc;
  const int pk = st->acc ? acc_step(st, k, ca, cb, cc) : (st->tr[k - 1] > (double)st->nocc ? 1 : 0);
  record_and_test(st, st->mcw ? 1 : pk, vk, st->mcw ? 0.0 : b + st->tr_shift, st->tr[k - 1]);
}

// ---- prescribed perturbation (Alg. 1: X~_i = X_i + E_i) ----------------------------------------
// E holds `count` consecutive N x N row-major matrices; E_i (i < count) is added to X_i as soon
// as it is formed: X_0 after the scaling (initial = 1, Tr[E_0] added to Tr[X_0] at once), X_k
// after square k (Tr[E_k] to st->tr_shift, which the finalize adds to the square's trace).  The
// trace is summed by block 0 in a fixed order.
__global__ void perturb_kernel(DevState* st, double* buf0, double* buf1, const double* __restrict__ E,
                               int64_t count, int initial) {
  __shared__ double sm[32];
  if (st->done) return;
  const int i = initial ? 0 : st->k + 1;
  if (i >= count) {
    if (!initial && blockIdx.x == 0 && threadIdx.x == 0) st->tr_shift = 0.0;
    return;
  }
  const int N = st->N, ld = st->ld;
  double* X = initial ? buf0 : (((st->k + 1) & 1) ? buf1 : buf0);
  const double* Ei = E + (int64_t)i * N * N;
  const int64_t total = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / N), c = (int)(e % N);
    X[(int64_t)r * ld + c] += Ei[e];
  }
  if (blockIdx.x != 0) return;
  double t = 0.0;
  for (int j = threadIdx.x; j < N; j += blockDim.x) t += Ei[(int64_t)j * N + j];
  t = block_sum<256>(t, sm);
  if (threadIdx.x == 0) {
    if (initial) st->tr[0] += t;
    else st->tr_shift = t;
  }
}

// ---- host-side launchers ------------------------------------------------------------------
static int elementwise_blocks(int64_t total) {
  int64_t b = (total + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

cudaError_t launch_bounds_and_init(DevState* st, const double* F, int64_t ldf, int N,
                                   double* part_lo, double* part_hi, int* part_bad, int nparts,
                                   cudaStream_t s) {
  gershgorin_kernel<<<nparts, kGershThreads, 0, s>>>(F, ldf, N, part_lo, part_hi, part_bad);
  init_kernel<<<1, kInitThreads, 0, s>>>(st, F, ldf, part_lo, part_hi, part_bad, nparts);
  return cudaGetLastError();
}

cudaError_t launch_scale_f64(const DevState* st, const double* F, int64_t ldf, int N, double* X0,
                             int ld, cudaStream_t s) {
  scale_kernel<<<elementwise_blocks((int64_t)N * N), 256, 0, s>>>(st, F, ldf, X0, ld);
  return cudaGetLastError();
}

cudaError_t launch_perturb(DevState* st, double* buf0, double* buf1, const double* E, int64_t count, int N,
                           int initial, cudaStream_t s) {
  perturb_kernel<<<elementwise_blocks((int64_t)N * N), 256, 0, s>>>(st, buf0, buf1, E, count, initial);
  return cudaGetLastError();
}

// ---- one product of the loop, by size ------------------------------------------------------------
// The digits a tensor-core product needs are made before the loop (X_0, launch_f64_digits) and after each product:
// of the new iterate, beside the stop test (which only that needs), and of the McWeeny step's square.
// N <= 128: 8 x 8 tiles on the FP64 units, which stage their rows whole in shared memory of that width; else the tensor
// cores, or 64 x 64 tiles on the FP64 units where the digit buffers were not to be had.  A round takes 16 us at N = 128
// and 28 us on the tensor cores at N = 129 (230 us in 64 x 64 tiles), so the line is the staging's limit; how far
// past it the 8 x 8 tiles would still win was not measured.
enum ProductOp { kSquare = 0, kMcwSquare = 1, kMcwProd = 2 };

static int recs_of(const f64tc::Plan* tc, int N) { return tc ? tc->recs : (N <= kSmallN ? kSmallRecs : 1); }

static cudaError_t emit_product(f64tc::Sink& sink, ProductOp op, DevState* st, double* buf0, double* buf1, double* S,
                                double* part, int T, const f64tc::Plan* tc, int N) {
  if (tc) {
    static constexpr f64tc::Op ops[3] = {f64tc::OP_SP2, f64tc::OP_MCW_SQ, f64tc::OP_MCW_PROD};
    return f64tc::emit_product(sink, st, buf0, buf1, S, part, *tc, ops[op]);
  }
  if (N <= kSmallN) {
    const int t = (N + kST - 1) / kST;
    int o = op;
    void* args[] = {&st, &buf0, &buf1, &S, &part, &o};
    return sink.put((const void*)small_product_kernel, dim3(t * (t + 1) / 2), dim3(kSmallThreads), 0, args);
  }
  const dim3 grid(T * (T + 1) / 2), block(kSyrkThreads);
  if (op == kSquare) {
    void* args[] = {&st, &buf0, &buf1, &part};
    return sink.put((const void*)syrk_f64_kernel, grid, block, 0, args);
  }
  void* args[] = {&st, &buf0, &buf1, &S, &part};
  return sink.put(op == kMcwSquare ? (const void*)mcw_square_kernel : (const void*)mcw_prod_kernel, grid, block, 0, args);
}

cudaError_t launch_f64_step_plain(DevState* st, double* buf0, double* buf1, double* part, int T,
                                  cudaStream_t s, const f64tc::Plan* tc, double* mscr, void* lz, int N, const double* E,
                                  int64_t ecount) {
  const int recs = recs_of(tc, N), nrec = T * (T + 1) / 2 * recs;
  f64tc::Sink sink;
  sink.s = s;
  cudaError_t e = emit_product(sink, kSquare, st, buf0, buf1, nullptr, part, T, tc, N);
  if (e != cudaSuccess) return e;
  if (lz && (e = launch_lanczos(st, buf0, buf1, nullptr, part, nrec, lz, N, T * kTile, s)) != cudaSuccess) return e;
  if (E && (e = launch_perturb(st, buf0, buf1, E, ecount, N, 0, s)) != cudaSuccess) return e;
  finalize_plain_kernel<<<1, kFinThreads, 0, s>>>(st, part, nrec, recs, mscr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return tc ? f64tc::emit_digits(sink, st, buf0, buf1, nullptr, *tc, N) : cudaSuccess;
}

cudaError_t launch_f64_digits(const DevState* st, const double* buf0, const double* buf1, const f64tc::Plan& P, int N,
                              cudaStream_t s) {
  f64tc::Sink sink;
  sink.s = s;
  return f64tc::emit_digits(sink, st, buf0, buf1, nullptr, P, N);
}

cudaError_t add_mcw_loop_body(cudaGraph_t body, DevState* st, double* buf0, double* buf1, double* S, double* part,
                              int T, cudaGraphConditionalHandle cond, const f64tc::Plan* tc, double* mscr, void* lz,
                              int N) {
  const int recs = recs_of(tc, N), nrec = T * (T + 1) / 2 * recs;
  f64tc::Sink sink;
  sink.g = body;
  cudaError_t e = emit_product(sink, kMcwSquare, st, buf0, buf1, S, part, T, tc, N);
  if (e != cudaSuccess) return e;
  cudaGraphNode_t before[2] = {sink.last, sink.last};          // what the product waits for
  if (tc) {                                                    // digits of S beside the estimate and the test
    f64tc::Sink side;
    side.g = body;
    side.last = sink.last;
    if ((e = f64tc::emit_digits(side, st, buf0, buf1, S, *tc, N)) != cudaSuccess) return e;
    before[1] = side.last;
  }
  if (lz && (e = add_lanczos_nodes(body, sink.last, st, buf0, buf1, S, part, nrec, lz, N, T * kTile, &sink.last)) !=
                cudaSuccess)
    return e;
  if ((e = add_finalize_node(body, &sink.last, 1, st, part, nrec, 2, recs, cond, &before[0], mscr)) != cudaSuccess)
    return e;
  if (tc) {
    if ((e = cudaGraphAddEmptyNode(&sink.last, body, before, 2)) != cudaSuccess) return e;
  } else {
    sink.last = before[0];
  }
  if ((e = emit_product(sink, kMcwProd, st, buf0, buf1, S, part, T, tc, N)) != cudaSuccess) return e;
  return tc ? f64tc::emit_digits(sink, st, buf0, buf1, nullptr, *tc, N) : cudaSuccess;
}

cudaError_t launch_mcw_step_plain(DevState* st, double* buf0, double* buf1, double* S, double* part, int T,
                                  cudaStream_t s, const f64tc::Plan* tc, double* mscr, void* lz, int N) {
  const int recs = recs_of(tc, N), nrec = T * (T + 1) / 2 * recs;
  f64tc::Sink sink;
  sink.s = s;
  cudaError_t e = emit_product(sink, kMcwSquare, st, buf0, buf1, S, part, T, tc, N);
  if (e != cudaSuccess) return e;
  if (tc && (e = f64tc::emit_digits(sink, st, buf0, buf1, S, *tc, N)) != cudaSuccess) return e;
  if (lz && (e = launch_lanczos(st, buf0, buf1, S, part, nrec, lz, N, T * kTile, s)) != cudaSuccess) return e;
  finalize_plain_kernel<<<1, kFinThreads, 0, s>>>(st, part, nrec, recs, mscr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = emit_product(sink, kMcwProd, st, buf0, buf1, S, part, T, tc, N)) != cudaSuccess) return e;
  return tc ? f64tc::emit_digits(sink, st, buf0, buf1, nullptr, *tc, N) : cudaSuccess;
}

cudaError_t add_finalize_node(cudaGraph_t g, const cudaGraphNode_t* deps, int ndeps, DevState* st,
                              double* part, int nparts, int stride, int recs, cudaGraphConditionalHandle cond,
                              cudaGraphNode_t* node, double* mscr) {
  void* args[] = {&st, &part, &nparts, &stride, &recs, &cond, &mscr};
  cudaKernelNodeParams kp = {};
  kp.func = (void*)finalize_kernel;
  kp.gridDim = dim3(1);
  kp.blockDim = dim3(kFinThreads);
  kp.kernelParams = args;
  return cudaGraphAddKernelNode(node, g, deps, ndeps, &kp);
}

cudaError_t add_f64_loop_body(cudaGraph_t body, DevState* st, double* buf0, double* buf1, double* part,
                              int T, cudaGraphConditionalHandle cond, const f64tc::Plan* tc, double* mscr, void* lz,
                              int N, const double* E, int64_t ecount) {
  const int recs = recs_of(tc, N), nrec = T * (T + 1) / 2 * recs;
  cudaGraphNode_t n_sq, n_fin;
  cudaKernelNodeParams kp = {};
  f64tc::Sink sink;
  sink.g = body;
  cudaError_t e = emit_product(sink, kSquare, st, buf0, buf1, nullptr, part, T, tc, N);
  if (e != cudaSuccess) return e;
  n_sq = sink.last;
  if (lz && (e = add_lanczos_nodes(body, n_sq, st, buf0, buf1, nullptr, part, nrec, lz, N, T * kTile, &n_sq)) != cudaSuccess) return e;
  if (E) {
    int initial = 0;
    void* pa[] = {&st, &buf0, &buf1, &E, &ecount, &initial};
    kp.func = (void*)perturb_kernel;
    kp.gridDim = dim3(elementwise_blocks((int64_t)N * N));
    kp.blockDim = dim3(256);
    kp.kernelParams = pa;
    cudaGraphNode_t n_pt;
    if ((e = cudaGraphAddKernelNode(&n_pt, body, &n_sq, 1, &kp)) != cudaSuccess) return e;
    n_sq = n_pt;
    sink.last = n_pt;
  }
  // digits of the new iterate, beside the estimate and the stop test
  if (tc && (e = f64tc::emit_digits(sink, st, buf0, buf1, nullptr, *tc, N)) != cudaSuccess) return e;
  return add_finalize_node(body, &n_sq, 1, st, part, nrec, 2, recs, cond, &n_fin, mscr);
}

cudaError_t launch_refine_f64(const DevState* st, const double* Xin, double* Xout, int ld, int step, double* part,
                              cudaStream_t s) {
  const int T = ld / kTile;
  refine_f64_kernel<<<T * (T + 1) / 2, kSyrkThreads, 0, s>>>(st, Xin, Xout, ld, step, part);
  return cudaGetLastError();
}

__global__ void copy_f64_kernel(const DevState* st, const double* __restrict__ X, int ld, double* __restrict__ D,
                                int64_t ldd) {
  const int N = st->N;
  const int64_t total = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / N), j = (int)(e % N);
    D[(int64_t)i * ldd + j] = X[(int64_t)i * ld + j];
  }
}

cudaError_t launch_copy_f64(const DevState* st, const double* X, int ld, int N, double* D, int64_t ldd,
                            cudaStream_t s) {
  copy_f64_kernel<<<elementwise_blocks((int64_t)N * N), 256, 0, s>>>(st, X, ld, D, ldd);
  return cudaGetLastError();
}

cudaError_t launch_copy_out(const DevState* st, const double* buf0, const double* buf1, int ld, int N,
                            double* D, int64_t ldd, cudaStream_t s) {
  copy_out_kernel<<<elementwise_blocks((int64_t)N * N), 256, 0, s>>>(st, buf0, buf1, ld, D, ldd);
  return cudaGetLastError();
}

}  // namespace sp2
