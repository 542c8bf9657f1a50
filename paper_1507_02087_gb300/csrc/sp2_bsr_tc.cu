// Tensor-core block products of the block-truncated expansion: the numeric square of one round
// (S = X~_{k-1}^2 on the upper pairs of its pattern, the SP2 epilogue, the per-pair partials of
// ||X~_{k-1} - S||_F^2 and Tr[X_k], the fixed-order block norms and the keep flags of the
// per-block truncation rule), on tcgen05 tensor cores.
//
// The square is cut into tiles of 4 block rows x 8 block columns (M = 128, N = 256); a tile is
// computed when it holds at least one upper pair of the square's pattern.  For tile (I0, J0),
// S[I0.., J0..] = sum over K of X[I0.., K] X[J0.., K]^T (X symmetric), the sum over the K blocks
// that one of the tile's 4 rows and one of its 8 columns both hold; a block a row lacks is the
// all-zero block.  Each iterate keeps, beside its FP32 blocks, every block as two fp16 pieces of
// 2^14 x (the FMT_FP16X2 format of the dense path) in the order of a ring stage, so a K block is 12 contiguous
// copies of 4 KB (as 24 tensor-map boxes of 32 rows x 64 bytes they bounded the kernel: 6.2 ms a square on the
// 32 x 24 x 24 lattice, 2.9 now, with the epilogue's loop and its halved FP64 work), and a tile's product is the three piece products p0 q0 + p0 q1 +
// p1 q0 per 16-wide k-step, accumulated in tensor memory in chunks of 4 K blocks (24 truncating
// FP32 additions, as on the dense path) and added into registers with round-to-nearest additions.
//
// Warp roles (one CTA per SM, persistent over the tile list): warp 0 finds the K blocks (OR of the
// tile rows' bitmap words, AND of the two ORs) and the 12 block positions of each from the words'
// popcounts, and issues the TMA copies; warp 1 issues the MMAs; warps 4..11 drain the chunks (two
// warps per tensor-memory lane quadrant = block row, 128 columns = 4 blocks each) and run the
// epilogue of the tile's pairs.  Every wait is bounded (2 s); a wait that gives up records
// SP2_ERR_TIMEOUT in the run's state, ends the run and winds the kernel down.
#include <cstring>

#include "../../include/sp2.h"
#include "sp2_bsr.cuh"
#include "sp2_kernels.h"
#include "sp2_tc.cuh"
#include "tc_ptx.cuh"

namespace sp2 {
namespace bsr {

using namespace sp2::ptx;

constexpr int TSTG = 4;                            // ring stages, one K block each
constexpr int BLK = 4 * BE;                        // a block's two pieces
constexpr int GRP = BLK / 4;                       // its 8-row groups, both pieces
constexpr int A_BYTES = TTR * BLK;                 // the 128 rows of A
constexpr int TSTAGE = (TTR + TTC) * BLK;          // 48 KB
constexpr int TSMEM = TSTG * TSTAGE + 1024;        // + alignment slack
constexpr int TCHK = 4;                            // K blocks per tensor-memory chunk
constexpr int TN = TTC * B;                        // 256 accumulator columns per chunk buffer
constexpr int TTHREADS = 384;                      // warpgroup 0: TMA, MMA, 2 idle; 8 epilogue warps
constexpr int T_REG_CTRL = 40, T_REG_EPI = 232;    // 40 + 2 x 232 <= 3 x 168 launch registers
constexpr uint64_t kTcWaitNs = 2000000000ull;
static_assert(T_REG_CTRL + 2 * T_REG_EPI <= 3 * 168, "register split exceeds the launch budget");
static_assert(2 * TN <= 512, "tensor memory columns");

__device__ __forceinline__ void tc_give_up(DevState* st, volatile int* abort_s) {
  *abort_s = 1;
  atomicExch(&st->status, (int)SP2_ERR_TIMEOUT);
  st->out_mode = OUT_NAN;
  st->done = 1;
}

constexpr int TMAXW = 64;                          // bitmap words per row (nb <= 2048)

struct TcArgs {
  DevState* st;
  Mat X;
  int nb, W, ncg;                                  // ncg: column groups of 8 blocks
  int zero_blk;                                    // index of the all-zero block
  int64_t pair_cap;                                // capacity of the square's pair arrays
  TcRound r;
};

__global__ void __launch_bounds__(TTHREADS, 1) bsr_tc_kernel(const TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[TSTG];
  __shared__ __align__(8) uint64_t empty_bar[TSTG];
  __shared__ __align__(8) uint64_t accf_bar[2];
  __shared__ __align__(8) uint64_t acce_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;
  __shared__ uint32_t rbits_s[TTR + TTC][TMAXW];     // producer: the tile rows' bitmap words
  __shared__ int rrank_s[TTR + TTC][TMAXW];          // and their rank-table entries

  DevState* st = a.st;
  if (!st->iter_active) return;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int ntiles = *a.r.tnnz;
  const Mat& X = a.X;
  const int nb = a.nb, W = a.W;
  if (threadIdx.x == 0) {
    for (int s = 0; s < TSTG; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&accf_bar[b], 1); mbar_init(&acce_bar[b], 8); }
    mbar_init(&drain_bar, 1);
    abort_s = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 2 * TN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;

  if (warp < 4) {
    setmaxnreg_dec<T_REG_CTRL>();
    if (warp == 0) {
      // ---------------- K-block discovery + TMA producer ----------------
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int armed[TSTG];
      uint32_t armed_par[TSTG];
      for (int s = 0; s < TSTG; ++s) { armed[s] = 0; armed_par[s] = 0; }
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int code = a.r.tiles[t];
        const int I0 = (code / a.ncg) * TTR, J0 = (code % a.ncg) * TTC;
        const int rowj = lane < TTR ? I0 + lane : J0 + (lane - TTR);
        const bool vj = lane < TTR + TTC && rowj < nb;
        const int rpj = vj ? X.rp[rowj] : 0;
        // the 12 rows' bitmap words and ranks, all loads in flight at once
        __syncwarp();
        for (int e = lane; e < (TTR + TTC) * W; e += 32) {
          const int j = e / W, w = e % W;
          const int row = j < TTR ? I0 + j : J0 + (j - TTR);
          const bool v = row < nb;
          rbits_s[j][w] = v ? X.bits[(int64_t)row * W + w] : 0u;
          rrank_s[j][w] = v ? X.rank[(int64_t)row * W + w] : 0;
        }
        __syncwarp();
        for (int w = 0; w < W && ok; ++w) {
          const uint32_t bj = lane < TTR + TTC ? rbits_s[lane][w] : 0u;
          const int rkj = lane < TTR + TTC ? rrank_s[lane][w] : 0;
          const uint32_t am = __reduce_or_sync(0xffffffffu, lane < TTR ? bj : 0u);
          const uint32_t bm = __reduce_or_sync(0xffffffffu, lane >= TTR && lane < TTR + TTC ? bj : 0u);
          uint32_t m = am & bm;
          while (m && ok) {
            const int bit = __ffs(m) - 1;
            m &= m - 1u;
            const bool has = vj && ((bj >> bit) & 1u);
            int posj = has ? rpj + rkj + __popc(bj & ((1u << bit) - 1u)) : a.zero_blk;
            if (!dcheck(posj >= 0 && posj <= a.zero_blk, &st->status)) posj = a.zero_blk;
            int go = 1;
            if (lane == 0) go = !abort_s && mbar_wait(&empty_bar[stage], phase ^ 1, globaltimer_ns() + kTcWaitNs);
            go = __shfl_sync(0xffffffffu, go, 0);
            if (!go) {
              ok = false;
              break;
            }
            // lane j < 12 copies its own block: row j of A (j < 4) or row j - 4 of B; the expected bytes are
            // armed first, so no copy can complete the phase early
            if (lane == 0) {
              mbar_arrive_expect_tx(&full_bar[stage], TSTAGE);
              armed[stage] = 1;
              armed_par[stage] = phase;
            }
            __syncwarp();
            if (lane < TTR + TTC)
              bulk_load(smem + stage * TSTAGE + lane * BLK, reinterpret_cast<const char*>(X.pvals) + (int64_t)posj * BLK, BLK,
                        &full_bar[stage]);
            if (++stage == TSTG) { stage = 0; phase ^= 1; }
          }
        }
      }
      if (lane == 0) {
        if (!ok) tc_give_up(st, &abort_s);
        for (int s = 0; s < TSTG; ++s)   // wait (bounded) until every copy issued here has landed
          if (armed[s]) mbar_wait(&full_bar[s], armed_par[s], globaltimer_ns() + kTcWaitNs);
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer ----------------
      constexpr uint32_t idesc = idesc_f16_f32(TTR * B, TN);
      if (elect_one()) {
        int stage = 0, buf = 0;
        uint32_t phase = 0, bphase = 0;
        bool ok = true;
        unsigned long long kblocks = 0ull, needed = 0ull;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
          const int nk = a.r.meta[(int64_t)t * TMETA];
          kblocks += (unsigned long long)nk;
          needed += (unsigned long long)a.r.meta[(int64_t)t * TMETA + 65];
          for (int k0 = 0; k0 < nk && ok; k0 += TCHK) {
            if (abort_s || !mbar_wait(&acce_bar[buf], bphase ^ 1, globaltimer_ns() + kTcWaitNs)) { ok = false; break; }
            tc_fence_after();
            const uint32_t dt = tmem_base + (uint32_t)(buf * TN);
            uint32_t accumulate = 0;
            const int kend = min(nk, k0 + TCHK);
            for (int k = k0; k < kend; ++k) {
              if (abort_s || !mbar_wait(&full_bar[stage], phase, globaltimer_ns() + kTcWaitNs)) { ok = false; break; }
              tc_fence_after();
              const uint32_t sA = smem_u32(smem + stage * TSTAGE);
              const uint32_t sB = sA + A_BYTES;
              auto piece = [](uint32_t base, int p, int kk) { return smem_desc_sw64_stride(base + p * (GRP / 2) + kk * 32, GRP); };
              #pragma unroll
              for (int kk = 0; kk < B / 16; ++kk) {
                // p1 q0 and p0 q1 of the whole K block first, then p0 q0: the small products are
                // added while the accumulator is still small
                mma_bf16(dt, piece(sA, 1, kk), piece(sB, 0, kk), idesc, accumulate);
                accumulate = 1;
                mma_bf16(dt, piece(sA, 0, kk), piece(sB, 1, kk), idesc, 1);
              }
              #pragma unroll
              for (int kk = 0; kk < B / 16; ++kk) mma_bf16(dt, piece(sA, 0, kk), piece(sB, 0, kk), idesc, 1);
              mma_commit(&empty_bar[stage]);
              if (++stage == TSTG) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            mma_commit(&accf_bar[buf]);
            if (++buf == 2) { buf = 0; bphase ^= 1; }
          }
        }
        // executed 32 x 32 x 32 block products: the tile's 32 block pairs times its K blocks
        atomicAdd(&st->bprod, kblocks * (unsigned long long)(TTR * TTC));
        atomicAdd(&st->uprod, needed);   // the tiles' needed products (tile metadata)
        if (!ok) tc_give_up(st, &abort_s);
        mma_commit(&drain_bar);
        mbar_wait(&drain_bar, 0, globaltimer_ns() + kTcWaitNs);
      }
    }
  } else {
    setmaxnreg_inc<T_REG_EPI>();
    // ---------------- chunk draining + epilogue (warps 4..11) ----------------
    const int ew = warp - 4;
    const int q = warp & 3;        // tensor-memory lanes 32 q .. 32 q + 31 = block row q of the tile
    const int hc = ew >> 2;        // columns 128 hc .. 128 hc + 127 = block columns 4 hc .. 4 hc + 3
    const int kprev = st->k;
    double ca = 0.0, cb = 0.0, cc = 0.0;
    const int gen = st->acc;
    const int pk = gen ? acc_step(st, kprev + 1, ca, cb, cc) : (st->tr[kprev] > (double)st->nocc ? 1 : 0);
    const float fa = (float)ca, fb = (float)cb, fc = (float)cc;
    int buf = 0;
    uint32_t bphase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int code = a.r.tiles[t];
      const int I0 = (code / a.ncg) * TTR, J0 = (code % a.ncg) * TTC;
      const int* meta = a.r.meta + (int64_t)t * TMETA;
      const int nk = meta[0];
      float acc[4][32];
      #pragma unroll
      for (int g = 0; g < 4; ++g)
        #pragma unroll
        for (int j = 0; j < 32; ++j) acc[g][j] = 0.f;
      uint32_t trow = 0;
      for (int k0 = 0; k0 < nk; k0 += TCHK) {
        int got = 0;
        if (lane == 0) got = !abort_s && mbar_wait(&accf_bar[buf], bphase, globaltimer_ns() + kTcWaitNs);
        got = __shfl_sync(0xffffffffu, got, 0);
        if (!got) {
          if (lane == 0) tc_give_up(st, &abort_s);
          ok = false;
          break;
        }
        tc_fence_after();
        trow = tmem_base + (uint32_t)(buf * TN + hc * 128) + ((uint32_t)(32 * q) << 16);
        #pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t raw[32];
          tmem_ld32(trow + g * 32, raw);
          tmem_wait_ld();
          #pragma unroll
          for (int j = 0; j < 32; ++j) acc[g][j] += __uint_as_float(raw[j]);
        }
        if (k0 + TCHK >= nk) break;          // this buffer takes the sums for the epilogue
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce_bar[buf]);
        if (++buf == 2) { buf = 0; bphase ^= 1; }
      }
      if (!ok) break;
      if (nk > 0) {
        #pragma unroll
        for (int g = 0; g < 4; ++g) tmem_st32(trow + 32 * g, acc[g]);
        tmem_wait_st();
      }
      // epilogue of the tile's upper pairs in this warp's four blocks; lane = row of the block.  A loop over the
      // blocks, their sums taken back from tensor memory: four copies of its code are bound by the instruction fetch
      const int I = I0 + q;
      #pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        const int J = J0 + 4 * hc + g;
        const int qi = meta[1 + TTC * q + 4 * hc + g];   // -1: not an upper pair of the square's pattern
        if (qi < 0 || !dcheck(qi < a.pair_cap, &st->status)) continue;
        int po = meta[33 + TTC * q + 4 * hc + g];
        if (po >= 0 && !dcheck(po < a.zero_blk, &st->status)) po = -1;
        float old[32];
        if (po >= 0) {
          const float4* src = reinterpret_cast<const float4*>(X.vals + (int64_t)po * BE + lane * B);
          #pragma unroll
          for (int v = 0; v < 8; ++v) {
            const float4 o4 = src[v];
            old[4 * v] = o4.x; old[4 * v + 1] = o4.y; old[4 * v + 2] = o4.z; old[4 * v + 3] = o4.w;
          }
        } else {
          #pragma unroll
          for (int j = 0; j < 32; ++j) old[j] = 0.f;
        }
        float sv32[32];
        {
          uint32_t raw[32];
          if (nk > 0) {
            tmem_ld32(trow + 32 * g, raw);
            tmem_wait_ld();
          } else {
            #pragma unroll
            for (int j = 0; j < 32; ++j) raw[j] = 0u;
          }
          #pragma unroll
          for (int j = 0; j < 32; ++j) sv32[j] = __uint_as_float(raw[j]) * tc::kF16InvScale2;
        }
        float4* dst = reinterpret_cast<float4*>(a.r.svals + (int64_t)qi * BE + lane * B);
        if (I == J) {
          // a diagonal block of the square: the tensor cores sum (r, c) and (c, r) in different
          // orders, so the upper triangle is mirrored (staged through the pair's output block)
          #pragma unroll
          for (int v = 0; v < 8; ++v)
            dst[v] = make_float4(sv32[4 * v], sv32[4 * v + 1], sv32[4 * v + 2], sv32[4 * v + 3]);
          __syncwarp();
          const float* blk = a.r.svals + (int64_t)qi * BE;
          #pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j < lane) sv32[j] = blk[j * B + lane];
          __syncwarp();
        }
        float vloc = 0.f, diag = 0.f;
        double trloc = 0.0, rs = 0.0;
        float nwv[32];
        #pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float sv = sv32[j];
          nwv[j] = gen ? fmaf(fa, sv, fmaf(fb, old[j], (I == J && lane == j) ? fc : 0.f))
                       : (pk ? sv : fmaf(2.0f, old[j], -sv));
          const float d = old[j] - sv;
          vloc = fmaf(d, d, vloc);
          if (lane == j) diag = nwv[j];
          const double x = (double)nwv[j];
          rs = __fma_rn(x, x, rs);                      // row `lane`, left to right (the square is exact)
        }
        #pragma unroll
        for (int v = 0; v < 8; ++v) dst[v] = make_float4(nwv[4 * v], nwv[4 * v + 1], nwv[4 * v + 2], nwv[4 * v + 3]);
        double n2 = 0.0;                                  // then the rows top to bottom
        for (int rr = 0; rr < 32; ++rr) n2 = __dadd_rn(n2, __shfl_sync(0xffffffffu, rs, rr));
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) vloc += __shfl_xor_sync(0xffffffffu, vloc, o);
        if (I == J) {
          trloc = (double)diag;
          #pragma unroll
          for (int o = 16; o > 0; o >>= 1) trloc += __shfl_xor_sync(0xffffffffu, trloc, o);
        }
        if (lane == 0) {
          a.r.spart[2 * (int64_t)qi] = (I == J ? 1.0 : 2.0) * (double)vloc;
          a.r.spart[2 * (int64_t)qi + 1] = trloc;
          a.r.skeep[qi] = (I == J || n2 >= a.r.tau2) ? 1 : 0;
          a.r.sn2[qi] = n2;
        }
      }
      if (nk > 0) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce_bar[buf]);
        if (++buf == 2) { buf = 0; bphase ^= 1; }
      }
    }
  }

  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 2 * TN);
  }
}

// One CTA per SM; sets the kernel's attribute on the current device first.
static int tc_grid() {
  static PerDevice grid;
  return grid.get([](int) {
    if (cudaFuncSetAttribute(bsr_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TSMEM) != cudaSuccess)
      (void)cudaGetLastError();
    return sm_count();
  });
}

void tc_prepare() { (void)tc_grid(); }

cudaError_t tc_numeric_launch(DevState* st, const Mat& X, int nb, int W, const TcRound& r, cudaStream_t s) {
  TcArgs a;
  std::memset(&a, 0, sizeof(a));
  a.st = st;
  a.X = X;
  a.nb = nb;
  a.W = W;
  a.ncg = (nb + TTC - 1) / TTC;
  a.zero_blk = nb * nb;
  a.pair_cap = (int64_t)nb * (nb + 1) / 2;
  a.r = r;
  bsr_tc_kernel<<<tc_grid(), TTHREADS, TSMEM, s>>>(a);
  return cudaGetLastError();
}

}  // namespace bsr
}  // namespace sp2
